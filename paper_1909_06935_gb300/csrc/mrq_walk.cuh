// The walk step, by distinct determinants (included by mrq.cu after mrq_cas.cuh).
//
// A walker's local evaluation (Eq. 5, Eq. 16, the reach-back overlaps of Eq. 6-7) depends on its
// determinant only, and the walkers of a system crowd on few of them: at 56 orbitals 4,096 walkers
// in the steady state sit on about 640 determinants of the CAS and 230 of the first-order space.
// So a step
//   k_group   finds the distinct determinants (a hash table over the walkers) and cuts each one's
//             walkers into task groups of at most MRQ_TGW;
//   k_prep    makes the determinant's constants: its diagonals and its single-excitation operator;
//   k_int     CAS determinants: the neighbours inside the CAS;
//   k_refs, k_insert, k_rows
//             CAS determinants: the overlaps outside the CAS.  O(m) depends on m alone, and the
//             determinants of a step share most of their active remnants, so the distinct rows
//             (remnant, core holes, virtual electrons) are found and computed once;
//   k_pairs   CAS determinants: every (X_a, Y_a) pair's neighbours, elements times rows;
//   k_fois_act; k_fgroups, k_frows, k_fois
//             first-order determinants: the neighbours that move active electrons only; the others, by
//             groups that share an active remnant (k_fgroups finds them, k_frows their overlaps);
//   k_move    adds the units' sums, takes each walker's winner, and looks up psi_s there;
//   k_accum   adds the step records into the accumulators.
// k_int, k_pairs and k_fois evaluate a determinant's neighbours once per task group, in work units
// spread over the whole chip, and run the move race of every walker of the group (its own Philox
// clocks against the shared rates).  They are kernels of their own because the walk is bound by
// instruction fetch when a warp scheduler's warps run different code (in one kernel 25 of 38 cycles
// per issue were waits for instructions).
// Every sum is formed in an order that depends on the determinant and its system alone, and the
// race's winner does not depend on any order, so a walker's step is the same whatever walkers
// share its determinant, alone or in a batch, and whatever the launch configuration.
//
// The units of a CAS determinant - chunks of the neighbours of an (X_a, Y_a) pair of active electrons
// removed / active holes filled - depend only on the system (all CAS determinants have the same active
// electron counts), so they are planned on the host at load.
//
// Per neighbour t = H_nm psi_s(m) is summed as |t| and t, and 1/psi_s(n) is applied once per
// determinant (S = |1/psi_n| sum |t|, E_L = H_nn + (1/psi_n) sum t).

#ifndef MRQ_MAXNW
#define MRQ_MAXNW 8           // warps per block (at most)
#endif
#define MRQ_VW 8              // virtual warps of the debug evaluation (MRQ_MAXNW <= MRQ_VW)
#define MRQ_CAS_CH 128        // neighbours per unit inside the CAS
#define MRQ_FOIS_CH 32        // neighbours per unit of a FOIS walker: one round (their reach-back is long)
#define MRQ_UNIT_NB 1024      // neighbours per unit of an (X_a, Y_a) pair (pairs are cut into chunks)
#define MRQ_TGW 32            // walkers per task group (at most): one per lane when they are read and moved
#define MRQ_NS_MAX 512        // slices of a determinant's units (at most): one warp task each

// constants of a CAS determinant
struct CasWalker {
    unsigned long long AOn, AEn, keyn;
    int cntO, cntE;
    double phin, c0;
};

__host__ __device__ __forceinline__ size_t cand_list_bytes(int cap) {
    return ((size_t)cap * sizeof(double) + (size_t)cap * sizeof(unsigned) + 15) / 16 * 16;
}

// the race's best candidate of a walker: FP32 clock, excitation, and t of its neighbour (16 bytes,
// replaced by one 128-bit compare-and-swap)
struct __align__(16) RaceBest {
    unsigned clk;             // FP32 image of the clock
    unsigned exc;             // excitation code, 0xFFFFFFFF: none yet
    double t;                 // H_nm psi_s(m)
};

// a run of walkers on one determinant
struct TaskGroup {
    int sys, first, count;    // members[first .. first + count): walkers of system sys
    int group;                // the determinant's index (its operator, constants and partial sums)
    int primary;              // the group of the determinant that stores its sums
    int pad;
};

struct GroupMeta {
    unsigned long long d[2][2];
    double psi, hnn, hdnn;
    double inv_psi, phi;      // 1/psi_s(n), psi_s(n)/c_0: divided once here (an FP64 division holds its SM's pipe for
                              // hundreds of cycles, and there are some 10^5 warp tasks per step)
    long long label;
    int h, p, sys, pad;
};

// counters of a step (WalkScratch::ctl)
enum {
    CTL_TGC, CTL_GC,              // CAS task groups, CAS determinants
    CTL_TGF, CTL_GF,              // first-order task groups, determinants
    CTL_INT, CTL_PAIRS, CTL_ACT, CTL_ROWTASK,   // next warp task of each kernel
    CTL_BIG, CTL_SMALL,           // tasks of k_rows in a wave: pieces of long rows, short rows
    CTL_FOIS, CTL_FG, CTL_FGTASK, // first-order waves: next task of k_fois, most groups of a determinant, next task
    CTL_FCUR = 14,                // (64 bits) doubles of the first-order row buffer in use
    CTL_N = CTL_FCUR + 2
};
enum { KNOWN_ROWS, KNOWN_EPOCH, KNOWN_CUR, KNOWN_N = KNOWN_CUR + 2 };   // rows, epoch, (64 bits) doubles of the buffer in use
#define MRQ_INT_SLICES 8          // warp tasks of a CAS determinant's neighbours inside the CAS
#define MRQ_ACT_SLICES 32         // warp tasks of a first-order determinant's active-only neighbours
#define MRQ_FOIS_SLICES 256       // warp tasks of its other neighbours
#define MRQ_BIG_ROW 1024          // entries of a task of k_rows; longer rows are cut (one warp took 1.3 ms on 65,000 entries)
#define MRQ_FG_NB 1024            // neighbours of a group of a first-order determinant (longer ones are cut)

// Neighbours of a first-order determinant that share an active remnant and an outer pattern: core
// electrons out (ac, sac of them alpha) and virtual orbitals entered (bv, sbv) run over all choices, the
// av virtual electrons that leave (the xs-th, or both) and the bc holes that are filled are fixed.
struct FGroup {
    unsigned long long ao;    // the neighbours' active remnant
    long long off;            // place of their psi_s in the row buffer
    int det, q0, nq;          // determinant; neighbours q0 ... q0 + nq - 1 of the choices
    unsigned char c, v, scn, sv;             // their core holes and virtual electrons (and alpha ones)
    unsigned char ac, sac, bv, sbv, av, bc, xs, ys;
};
#define MRQ_NOROW 255             // a reference without entries
#define MRQ_KNOWN 64              // flag of a reference whose row is known from an earlier step of the launch

// device workspace of a walk launch, sized for the slots [seg0, seg1) of the walk set
struct WalkScratch {
    int *rep, *cnt, *start;   // determinant tables, 4 entries per slot: first walker, walkers, first member
    int *tab_of, *pos_of;     // per slot: table entry and place in it
    int* members;             // walkers (local index) by determinant
    TaskGroup *tgc, *tgf;     // CAS and first-order task groups
    GroupMeta* meta;          // per determinant: CAS ones from the front, first-order ones from the back
    double* gops;             // single-excitation operators, gstride doubles per determinant
    double* part;             // [determinant][ns_max + MRQ_ACT_SLICES][3] partial sums (the last ones: k_int, k_fois_act)
    RaceBest* best;           // per slot
    unsigned* bound;          // per slot: FP32 bits of an upper bound of the best clock
    int* ctl;
    int* seen;                // most CAS determinants of a step so far
    // rows of a wave of at most wave_groups CAS determinants; a reference is (determinant of the wave,
    // row number in it), index determinant * nref_max + row number
    unsigned long long* ref_ao;   // the row's active remnant
    unsigned char* ref_cls;       // 3 (core holes) + (virtual electrons), MRQ_NOROW
    int* ref_rep;                 // the reference that owns the row
    long long* row_off;           // (owners and rows known from earlier) the row's place in rows
    int* table;                   // open addressing over references
    int2* ulist;                  // tasks of k_rows: owner, piece (cut rows from the front, whole ones from the back)
    int ulist_size;
    double* rows;
    int table_size, nref_max, wave_groups, wave0;
    // rows known in this launch: open addressing over row numbers (entry: epoch << 32 | row; another epoch's
    // entry is an empty one), the rows' remnants, systems and classes, and places
    unsigned long long* ktab;
    unsigned long long* k_ao;
    int* k_key;
    long long* k_off;
    int* kctl;                    // KNOWN_*
    int ktab_size;
    long long row_worst;
    // groups of a wave of at most fwave first-order determinants (fg_max each) and psi_s of their neighbours
    FGroup* fg;
    double* frows;
    int2* fg_of;              // per determinant of the wave: first group, groups
    int fg_max, fwave, fwave0;
    long long gstride, nseg;
    int ns_max, tgw;
    long long seg0, seg1;
};

__device__ __forceinline__ void write_rec(mrq_neighbour* rec, const unsigned long long* m, int W, double hnm,
                                          double hd, double om, double psim, double gamma, unsigned exc) {
#pragma unroll
    for (int w = 0; w < 4; w++) rec->det[w] = 0;
    for (int w = 0; w < W; w++) {
        rec->det[w] = m[w];
        rec->det[W + w] = m[2 + w];
    }
    rec->h = hnm;
    rec->hd = hd;
    rec->o = om;
    rec->psi = psim;
    rec->gamma = gamma;
    rec->exc = exc;
    rec->pad = 0;
}

template <int W>
__device__ __forceinline__ void det_words(const unsigned long long (&m)[2][W], unsigned long long* out4) {
    for (int w = 0; w < 2; w++) out4[w] = out4[2 + w] = 0;
#pragma unroll
    for (int w = 0; w < W; w++) {
        out4[w] = m[0][w];
        out4[2 + w] = m[1][w];
    }
}

__device__ __forceinline__ unsigned exc_code(int r1, int r2, int a1, int a2) {
    return (unsigned)r1 | ((unsigned)r2 << 8) | ((unsigned)a1 << 16) | ((unsigned)a2 << 24);
}

// spin-resolved candidate blocks: R' (ne electrons of m's active occupation) and A' (nf holes),
// alpha(R') - alpha(A') = dsp; block b takes alpha(R') = ib[b]; its index is decoded by multiplying
// with precomputed reciprocals (mixed radix nRb x nAa x nAb, fastest last)
struct CandPlan {
    unsigned long long oa, ob, ea, eb;   // m's active electrons / holes by spin (combined bit positions)
    int coa, cob, cea, ceb;
    int nblk;
    int ib[3];
    int start[4];
    unsigned rAb[3], rAa[3], rRb[3];     // the radices and their magic32 reciprocals
    unsigned mAb[3], mAa[3], mRb[3];
};

__device__ __forceinline__ void cand_plan(CandPlan& P, unsigned long long AOm, unsigned long long AEm, int ne, int nf,
                                          int dsp) {
    P.oa = AOm & 0xFFFFFFFFull;
    P.ob = AOm & 0xFFFFFFFF00000000ull;
    P.ea = AEm & 0xFFFFFFFFull;
    P.eb = AEm & 0xFFFFFFFF00000000ull;
    P.coa = __popcll(P.oa);
    P.cob = __popcll(P.ob);
    P.cea = __popcll(P.ea);
    P.ceb = __popcll(P.eb);
    P.nblk = 0;
    P.start[0] = 0;
    for (int i = 0; i <= ne; i++) {
        const int j = i - dsp;
        if (j < 0 || j > nf) continue;
        if (i > P.coa || ne - i > P.cob || j > P.cea || nf - j > P.ceb) continue;
        const int nRa = nsub(P.coa, i), nRb = nsub(P.cob, ne - i), nAa = nsub(P.cea, j), nAb = nsub(P.ceb, nf - j);
        const int sz = nRa * nRb * nAa * nAb;
        if (sz == 0) continue;
        const int b = P.nblk;
        P.ib[b] = i;
        P.rAb[b] = (unsigned)nAb;
        P.rAa[b] = (unsigned)nAa;
        P.rRb[b] = (unsigned)nRb;
        P.mAb[b] = magic32((unsigned)nAb);
        P.mAa[b] = magic32((unsigned)nAa);
        P.mRb[b] = magic32((unsigned)nRb);
        P.start[b + 1] = P.start[b] + sz;
        P.nblk++;
    }
}

__device__ __forceinline__ void cand_decode(const SysDev& S, const CandPlan& P, int ne, int nf, int dsp, int t,
                                            unsigned long long& Rb, unsigned long long& Ab) {
    int b = 0;
    while (b + 1 < P.nblk && t >= P.start[b + 1]) b++;
    unsigned x = (unsigned)(t - P.start[b]);
    const int i = P.ib[b], j = i - dsp;
    unsigned q = div_m(x, P.mAb[b]);
    const int tAb = (int)(x - q * P.rAb[b]);
    x = q;
    q = div_m(x, P.mAa[b]);
    const int tAa = (int)(x - q * P.rAa[b]);
    x = q;
    q = div_m(x, P.mRb[b]);
    const int tRb = (int)(x - q * P.rRb[b]);
    const int tRa = (int)q;
    Rb = subset_bits(S.colex, P.oa, P.coa, i, tRa) | subset_bits(S.colex, P.ob, P.cob, ne - i, tRb);
    Ab = subset_bits(S.colex, P.ea, P.cea, j, tAa) | subset_bits(S.colex, P.eb, P.ceb, nf - j, tAb);
}

// build the candidate list of group (c, v, sc, sv) of active remnant (AOm, AEm): singles [0, n1) as
// codes, doubles [n1, count) as (signed weight, table base); the candidate of key keyn (the walker) is left out.  Kept
// out of line: it runs once per group, and its registers and code then stay out of the neighbour
// loop that follows (1.8 % faster at 56 orbitals)
template <int W, bool ROWS, class C>
__device__ __noinline__ int build_group_list(const SysDev& S, unsigned long long keyn,
                                                const unsigned long long (&mref)[2][W], unsigned long long AOm,
                                                unsigned long long AEm, int c, int v, int sc, int sv, int rxc0,
                                                int rxc1, int ryv0, int ryv1, int par_ref, double* cphi,
                                                unsigned* ccode, int& n1, int lane, C& ctr) {
    const unsigned lt = (1u << lane) - 1u;
    int count = 0;
    n1 = 0;
    for (int rr = 1; rr <= 2; rr++) {
        if (rr == 2) n1 = count;
        if (rr == 1 && (c > 1 || v > 1)) continue;
        const int ne = rr - v, nf = rr - c;
        if (ne < 0 || nf < 0) continue;
        const int dsp = sc - sv;                  // alpha(R') - alpha(A') = alpha(X_c) - alpha(Y_v)
        CandPlan P;
        cand_plan(P, AOm, AEm, ne, nf, dsp);
        const int tot = P.start[P.nblk];
        for (int base = 0; base < tot; base += 32) {
            const int t = base + lane;
            bool valid = t < tot;
            unsigned long long Rb = 0, Ab = 0;
            double phi = 0.0;
            if (valid) {
                cand_decode(S, P, ne, nf, dsp, t, Rb, Ab);
                const unsigned long long kact = (AOm & ~Rb) | Ab;
                const unsigned long long key = hash_key(S, (unsigned)kact, (unsigned)(kact >> 32));
                ctr.cand();
                if (key == keyn) valid = false;
                else {
                    phi = hash_lookup(S, key, ctr);
                    valid = (__double_as_longlong(phi) << 1) != 0;      // phi != 0 without an FP64 compare
                }
            }
            const unsigned vm = __ballot_sync(0xffffffffu, valid);
            if (valid) {
                const int pos = count + __popc(vm & lt);
                if (pos < S.cand_cap) {
                    if (rr == 1) {
                        int sgn = 0;
                        if (ROWS) {     // <k|H|m> changes sign between the group's neighbours as their core parity does
                            const int x = v ? ryv0 : act_so(S, __ffsll(Rb) - 1), y = c ? rxc0 : act_so(S, __ffsll(Ab) - 1);
                            const int sx = x >= S.n, px = x - sx * S.n, py = y - sx * S.n;
                            sgn = popc_sel<W>(mref, sx, min(px, py), max(px, py)) + par_ref;
                        }
                        cphi[pos] = neg_if(phi, sgn);
                        ccode[pos] = pack_cand(Rb, Ab, rr);
                    } else {
                        double w;
                        unsigned bp;
                        dbl_entry<W>(S, mref, c, v, rxc0, rxc1, ryv0, ryv1, par_ref, Rb, Ab, phi, w, bp);
                        cphi[pos] = w;
                        ccode[pos] = bp;
                    }
                }
            }
            count += __popc(vm);
        }
    }
    if (count > S.cand_cap) {
        if (lane == 0) atomicOr(S.err, MRQ_ERR_CAP);
        count = S.cand_cap;
        n1 = min(n1, count);
    }
    __syncwarp();
    return count;
}

// lanes per neighbour in a round of nr neighbours
__device__ __forceinline__ int split_of(int nr) {
    return nr > 16 ? 1 : (nr > 8 ? 2 : (nr > 4 ? 4 : (nr > 2 ? 8 : (nr > 1 ? 16 : 32))));
}

// <m|H|n> of a double n -> m (removed r1 < r2 core/active, added a1 < a2 active/virtual) from the
// physicists' tables: <r1 r2||a1 a2> (same spin) or <r1 r2|a1 a2> (opposite), one gather
template <int W, class C>
__device__ __forceinline__ double double_elem_tab(const SysDev& S, const unsigned long long (&d)[2][W], int r1, int r2,
                                                  int a1, int a2, C& ctr) {
    const int n = S.n;
    const int s_r1 = r1 >= n, s_r2 = r2 >= n;
    const int pr1 = r1 - s_r1 * n, pr2 = r2 - s_r2 * n, pa1 = a1 - (a1 >= n) * n, pa2 = a2 - (a2 >= n) * n;
    int c1 = popc_sel<W>(d, s_r1, min(pr1, pa1), max(pr1, pa1));
    int c2;
    if (s_r2 == s_r1) {
        unsigned long long t[W];
#pragma unroll
        for (int w = 0; w < W; w++) t[w] = s_r1 ? d[1][w] : d[0][w];
        flip<W>(t, pr1);
        flip<W>(t, pa1);
        c2 = popc_between<W>(t, min(pr2, pa2), max(pr2, pa2));
    } else {
        c2 = popc_sel<W>(d, s_r2, min(pr2, pa2), max(pr2, pa2));
    }
    const unsigned sv = (unsigned)S.nav, sq = sv * sv, sp = sq * (unsigned)S.nca;
    const unsigned idx = (s_r1 == s_r2 ? S.tab_half : 0u) + (unsigned)pr1 * sp + (unsigned)pr2 * sq +
                         (unsigned)(pa1 - S.nc) * sv + (unsigned)(pa2 - S.nc);
    ctr.g();
    return neg_if(__ldg(S.tab + idx), c1 + c2);
}

// ------------------------------------------------------------------ CAS units

// neighbours of pair (X_a, Y_a) in the flat order of its groups; returns the total
__device__ __forceinline__ int pair_total(const SysDev& S, int ka, int kb, int d) {
    int tot = 0;
    for (int r = max(1, max(ka, kb)); r <= 2; r++) {
        const int c = r - ka, v = r - kb;
        if (c == 0 && v == 0) continue;
        for (int sc = 0; sc <= c; sc++) {
            const int sv = sc - d;
            if (sv < 0 || sv > v) continue;
            tot += shape_count(S.nc, c, sc) * shape_count(S.nv, v, sv);
        }
    }
    return tot;
}

// neighbours of one CAS unit (for the debug records' offsets)
__device__ __forceinline__ int cas_unit_count(const SysDev& S, const CasWalker& cw, int u) {
    if (u < S.cas_units) return min(MRQ_CAS_CH, S.cas_nb - u * MRQ_CAS_CH);
    int k = 0;
    while (k < 7 && u >= S.unit_off[k + 1]) k++;
    const int ka = k / 3, kb = k % 3, nch = S.nch[k];
    const int loc = u - S.unit_off[k];
    const int pair = loc / nch, ch = loc - pair * nch;
    const int nYa = nsub(cw.cntE, kb);
    const int xa = pair / nYa, ya = pair - xa * nYa;
    const unsigned long long Xb = subset_bits(S.colex, cw.AOn, cw.cntO, ka, xa);
    const unsigned long long Yb = subset_bits(S.colex, cw.AEn, cw.cntE, kb, ya);
    const int d = __popcll(Yb & 0xFFFFFFFFull) - __popcll(Xb & 0xFFFFFFFFull);
    const int tot = pair_total(S, ka, kb, d);
    const int lo = (int)((long long)ch * tot / nch), hi = (int)((long long)(ch + 1) * tot / nch);
    return hi - lo;
}

// excitations of active electrons into active holes (coa, cob: occupied alpha, beta; cea, ceb: empty)
__device__ __forceinline__ int active_neighbours(int coa, int cob, int cea, int ceb) {
    return coa * cea + cob * ceb + nsub(coa, 2) * nsub(cea, 2) + nsub(cob, 2) * nsub(ceb, 2) + coa * cea * cob * ceb;
}

// the idx-th of them, spin-resolved (alpha singles, beta singles, alpha-alpha, beta-beta, alpha-beta
// doubles): removed and added active bits; returns the rank
__device__ __forceinline__ int active_neighbour(const SysDev& S, unsigned long long oa, unsigned long long ob,
                                                unsigned long long ea, unsigned long long eb, int idx,
                                                unsigned long long& Xb, unsigned long long& Yb) {
    const int coa = __popcll(oa), cob = __popcll(ob), cea = __popcll(ea), ceb = __popcll(eb);
    const int b0 = coa * cea, b1 = b0 + cob * ceb, b2 = b1 + nsub(coa, 2) * nsub(cea, 2),
              b3 = b2 + nsub(cob, 2) * nsub(ceb, 2);
    if (idx < b1) {
        const bool al = idx < b0;
        const int x = al ? idx : idx - b0, ny = al ? cea : ceb;
        Xb = subset_bits(S.colex, al ? oa : ob, al ? coa : cob, 1, x / ny);
        Yb = subset_bits(S.colex, al ? ea : eb, ny, 1, x % ny);
        return 1;
    }
    if (idx < b3) {
        const bool al = idx < b2;
        const int x = al ? idx - b1 : idx - b2, ne = al ? cea : ceb, ny = nsub(ne, 2);
        Xb = subset_bits(S.colex, al ? oa : ob, al ? coa : cob, 2, x / ny);
        Yb = subset_bits(S.colex, al ? ea : eb, ne, 2, x % ny);
        return 2;
    }
    int x = idx - b3;                          // the beta excitation slowest
    const int ya = x % cea;
    x /= cea;
    const int xa = x % coa;
    x /= coa;
    Xb = subset_bits(S.colex, oa, coa, 1, xa) | subset_bits(S.colex, ob, cob, 1, x / ceb);
    Yb = subset_bits(S.colex, ea, cea, 1, ya) | subset_bits(S.colex, eb, ceb, 1, x % ceb);
    return 2;
}

// neighbours inside the CAS: spin-resolved blocks (alpha singles, beta singles, alpha-alpha,
// beta-beta, alpha-beta doubles) of the walker's active electrons / holes
template <int W, class Sink, class C>
__device__ __noinline__ void cas_internal_unit(const SysDev& S, const CasWalker& cw, const unsigned long long (&n)[2][W],
                                               int u, int lane, Sink& sink, C& ctr) {
    const unsigned long long oa = cw.AOn & 0xFFFFFFFFull, ob = cw.AOn & ~0xFFFFFFFFull;
    const unsigned long long ea = cw.AEn & 0xFFFFFFFFull, eb = cw.AEn & ~0xFFFFFFFFull;
    const int i0 = u * MRQ_CAS_CH;
    const int i1 = min(active_neighbours(__popcll(oa), __popcll(ob), __popcll(ea), __popcll(eb)), i0 + MRQ_CAS_CH);
    for (int base = i0; base < i1; base += 32) {
        const bool valid = base + lane < i1;
        const int idx = base + lane;
        unsigned long long m[2][W];
#pragma unroll
        for (int sg = 0; sg < 2; sg++)
#pragma unroll
            for (int w = 0; w < W; w++) m[sg][w] = n[sg][w];
        double hnm = 0.0, om = 0.0, psim = 0.0;
        unsigned exc = 0;
        if (valid) {
                unsigned long long Xb, Yb;
            const int r = active_neighbour(S, oa, ob, ea, eb, idx, Xb, Yb);
            int rem[2], add[2];
            act_list(S, Xb, rem);
            act_list(S, Yb, add);
            apply_exc<W>(m, S, rem, add, r);
            hnm = r == 1 ? single_elem<W>(S, n, rem[0], add[0], ctr)
                                      : double_elem_tab<W>(S, n, rem[0], rem[1], add[0], add[1], ctr);
            const unsigned long long km = (cw.AOn & ~Xb) | Yb;
            ctr.cand();
            om = hash_lookup(S, hash_key(S, (unsigned)km, (unsigned)(km >> 32)), ctr);
            exc = r == 1 ? exc_code(rem[0], rem[0], add[0], add[0]) : exc_code(rem[0], rem[1], add[0], add[1]);
            psim = cw.c0 * om;
        }
        sink.template post<W>(valid, idx - i0, m, hnm, 0.0, om, psim, exc);
    }
}

// one (X_a, Y_a) pair chunk [lo, hi) of a CAS walker with the lists of its own groups (the debug evaluation,
// which counts a determinant's own terms; the walk takes the shared rows, k_pairs)
template <int W, class Sink, class C>
__device__ void cas_pair_unit(const SysDev& S, const CasWalker& cw, const double* __restrict__ gops, double* cphi,
                              unsigned* ccode, const unsigned long long (&n)[2][W], int u, int lane, Sink& sink, C& ctr) {
    int k = 0;
    while (k < 7 && u >= S.unit_off[k + 1]) k++;
    const int ka = k / 3, kb = k % 3, nch = S.nch[k];
    const int loc = u - S.unit_off[k];
    const int pair = loc / nch, ch = loc - pair * nch;
    const int nYa = nsub(cw.cntE, kb);
    const int xa = pair / nYa, ya = pair - xa * nYa;
    const unsigned long long Xb = subset_bits(S.colex, cw.AOn, cw.cntO, ka, xa);
    const unsigned long long Yb = subset_bits(S.colex, cw.AEn, cw.cntE, kb, ya);
    const int d = __popcll(Yb & 0xFFFFFFFFull) - __popcll(Xb & 0xFFFFFFFFull);
    const int tot = pair_total(S, ka, kb, d);
    const int lo = (int)((long long)ch * tot / nch), hi = (int)((long long)(ch + 1) * tot / nch);
    if (lo >= hi) return;
    const unsigned long long AOm = (cw.AOn & ~Xb) | Yb, AEm = (cw.AEn & ~Yb) | Xb;
    const int xa0 = Xb ? act_so(S, __ffsll(Xb) - 1) : 0;
    const int xa1 = (ka == 2) ? act_so(S, 63 - __clzll(Xb)) : 0;
    const int ya0 = Yb ? act_so(S, __ffsll(Yb) - 1) : 0;
    const int ya1 = (kb == 2) ? act_so(S, 63 - __clzll(Yb)) : 0;
    const int nc = S.nc, nv = S.nv, voff = S.nc + S.na;
    int base = 0;
    for (int r = max(1, max(ka, kb)); r <= 2; r++) {
        const int c = r - ka, v = r - kb;
        if (c == 0 && v == 0) continue;
        for (int sc = 0; sc <= c; sc++) {
            const int sv = sc - d;
            if (sv < 0 || sv > v) continue;
            const int ncc = shape_count(nc, c, sc), nvc = shape_count(nv, v, sv);
            const int ni = ncc * nvc;
            const int q0 = max(lo, base) - base, q1 = min(hi, base + ni) - base;
            if (ni > 0 && q0 < q1) {
                // reference neighbour (the group's first) for the candidates' signs
                int rxc0, rxc1, ryv0, ryv1, rrm0, rrm1, rad0, rad1;
                unsigned long long mref[2][W];
                group_neighbour<W>(S, n, nc, nv, voff, c, sc, v, sv, 0, 0, ka, xa0, xa1, kb, ya0, ya1, r, rxc0, rxc1,
                                   ryv0, ryv1, rrm0, rrm1, rad0, rad1, mref);
                const int par_ref = (c >= 1 ? rxc0 - (rxc0 >= S.n ? S.n : 0) : 0) + (c == 2 ? rxc1 - (rxc1 >= S.n ? S.n : 0) : 0);
                int n1;
                // floor(q / nvc) = high word of q * ceil(2^64 / nvc), exact for q < 2^32 (nvc > 1)
                const unsigned long long mvc = ~0ull / (unsigned long long)nvc + 1ull;
                const int count = build_group_list<W, false>(S, cw.keyn, mref, AOm, AEm, c, v, sc, sv, rxc0, rxc1, ryv0, ryv1,
                                                      par_ref, cphi, ccode, n1, lane, ctr);
                for (int qb = q0; qb < q1; qb += 32) {
                    const int nr = min(32, q1 - qb);
                    const int f = split_of(nr), lf = __ffs(f) - 1;
                    const int qi = lane >> lf, part = lane & (f - 1);
                    const bool valid = qi < nr;
                    const int q = qb + (valid ? qi : 0);
                    int xc0, xc1, yv0, yv1, rm0, rm1, ad0, ad1;
                    unsigned long long m[2][W];
                    const int ic = nvc == 1 ? q : (int)__umul64hi((unsigned long long)q, mvc);     // q / nvc
                    group_neighbour<W>(S, n, nc, nv, voff, c, sc, v, sv, ic, q - ic * nvc, ka, xa0, xa1, kb, ya0,
                                       ya1, r, xc0, xc1, yv0, yv1, rm0, rm1, ad0, ad1, m);
                    unsigned offd, offx;
                    int par;
                    lane_offsets(S, c, v, xc0, xc1, yv0, yv1, offd, offx, par);
                    double hnm = 0.0, a0 = 0.0, a1 = 0.0;
                    if (valid) {
                        if (part == 0) {
                            if (r == 1) {
                                // single n -> m (x = rm0 -> y = ad0): the walker's operator G
                                const int sx = rm0 >= S.n, px = rm0 - sx * S.n, py = ad0 - sx * S.n;
                                hnm = neg_if(gops[(sx * S.nca + px) * S.nav + (py - S.nc)],
                                             sgn_sel<W>(n, sx, px, py) < 0 ? 1 : 0);
                                ctr.g();
                            } else {
                                hnm = double_elem_tab<W>(S, n, rm0, rm1, ad0, ad1, ctr);
                            }
                            a0 = neg_if(hnm * cw.phin, par);        // the k = n term
                        }
                        for (int e = part; e < n1; e += f)
                            a1 = fma(cphi[e], neg_if(sgl_elem_code<W>(S, gops, m, ccode[e], v, yv0, c, xc0, r, rm0,
                                                                       rm1, ad0, ad1, ctr), par), a1);
                        int e = n1 + ((part - n1) & (f - 1));
                        const int st = f;
                        for (; e + 3 * st < count; e += 4 * st) {
                            const unsigned p0 = ccode[e], p1 = ccode[e + st], p2 = ccode[e + 2 * st],
                                           p3 = ccode[e + 3 * st];
                            const double x0 = __ldg(S.tab + (p0 & 0x7FFFFFFFu) + ((p0 & 0x80000000u) ? offx : offd));
                            const double x1 = __ldg(S.tab + (p1 & 0x7FFFFFFFu) + ((p1 & 0x80000000u) ? offx : offd));
                            const double x2 = __ldg(S.tab + (p2 & 0x7FFFFFFFu) + ((p2 & 0x80000000u) ? offx : offd));
                            const double x3 = __ldg(S.tab + (p3 & 0x7FFFFFFFu) + ((p3 & 0x80000000u) ? offx : offd));
                            a0 = fma(cphi[e], x0, a0);
                            a1 = fma(cphi[e + st], x1, a1);
                            a0 = fma(cphi[e + 2 * st], x2, a0);
                            a1 = fma(cphi[e + 3 * st], x3, a1);
                            ctr.g(4);
                        }
                        for (; e < count; e += st) {
                            const unsigned p0 = ccode[e];
                            a0 = fma(cphi[e], __ldg(S.tab + (p0 & 0x7FFFFFFFu) + ((p0 & 0x80000000u) ? offx : offd)), a0);
                            ctr.g();
                        }
                    }
                    double s = a0 + a1;
                    for (int o = f >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                    double om = 0.0, psim = 0.0;
                    unsigned exc = 0;
                    const bool mine = valid && part == 0;
                    if (mine) {
                        ctr.term(count + 1);
                        om = neg_if(s, par);
                        const int h0 = xc0 >= S.n ? nc + (xc0 - S.n) : xc0;
                        const int h1 = xc1 >= S.n ? nc + (xc1 - S.n) : xc1;
                        const int p0 = yv0 >= S.n ? nv + (yv0 - S.n - voff) : yv0 - voff;
                        const int p1 = yv1 >= S.n ? nv + (yv1 - S.n - voff) : yv1 - voff;
                        const long long lm = set_rank(c, h0, h1, 2 * nc) * S.nPs + set_rank(v, p0, p1, 2 * nv);
                        ctr.g();
                        psim = __ldg(S.c + lm) * om;
                        exc = r == 1 ? exc_code(rm0, rm0, ad0, ad0) : exc_code(rm0, rm1, ad0, ad1);
                    }
                    sink.template post<W>(mine, base + q - lo, m, hnm, 0.0, om, psim, exc);
                }
                __syncwarp();
            }
            base += ni;
        }
    }
}

// ------------------------------------------------------------------ FOIS units

// neighbours [i0, i1) of the class-block enumeration, reach-back per lane (the debug evaluation)
template <int W, class Sink, class C>
__device__ __noinline__ void fois_unit(const SysDev& S, const WarpLists& sh, const double* __restrict__ gops,
                                       const unsigned long long (&n)[2][W], long long ln, double c0,
                                       unsigned long long self_key, double phi_self, int i0, int i1, int lane,
                                       Sink& sink, C& ctr) {
    for (int base = i0; base < i1; base += 32) {
        const int idx = base + lane;
        const bool valid = idx < i1;
        unsigned long long m[2][W];
#pragma unroll
        for (int sg = 0; sg < 2; sg++)
#pragma unroll
            for (int w = 0; w < W; w++) m[sg][w] = n[sg][w];
        double hnm = 0.0, hd = 0.0, om = 0.0, psim = 0.0;
        unsigned exc = 0;
        if (valid) {
            int lo = 0, hi = sh.nb - 1;          // block of idx: last b with bstart[b] <= idx
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (sh.bstart[mid] <= idx) lo = mid;
                else hi = mid - 1;
            }
            const unsigned desc = sh.bdesc[lo];
            int kind, r1, r2, a1, a2;
            decode_exc(sh, S.n, desc, idx - sh.bstart[lo], kind, r1, r2, a1, a2);
            {
                int s1 = r1 >= S.n, s2 = a1 >= S.n;
                flip_reg<W>(m, s1, r1 - s1 * S.n);
                flip_reg<W>(m, s2, a1 - s2 * S.n);
                if (kind != 0) {
                    int s3 = r2 >= S.n, s4 = a2 >= S.n;
                    flip_reg<W>(m, s3, r2 - s3 * S.n);
                    flip_reg<W>(m, s4, a2 - s4 * S.n);
                }
            }
            if (kind != 0) hnm = hb_screen(S, double_elem<W>(S, n, r1, r2, a1, a2, ctr));
            else if (gops != nullptr && in_walker_block(S, r1, a1))
                hnm = single_from_walker<W>(S, SglFromWalker{gops, 0, 0, 0, 0, 0}, n, r1, a1, ctr);
            else hnm = single_elem<W>(S, n, r1, a1, ctr);
            int hm, pm;
            const long long lm = det_label<W>(S, m, hm, pm);
            if (lm == 0) {
                ctr.cand();
                om = hash_lookup(S, hash_key(S, active_bits<W>(S, m[0]), active_bits<W>(S, m[1])), ctr);
                psim = c0 * om;
            } else {
                om = reach_back<W>(S, m, ctr, self_key, hnm * phi_self,
                                   SglFromWalker{gops, kind == 0 ? 1 : 2, r1, r2, a1, a2});
                ctr.g();
                psim = __ldg(S.c + lm) * om;
            }
            const bool same = ln > 0 && active_only(desc);
            hd = same ? ((kind == 0) ? hd_single_elem<W>(S, n, r1, a1, ctr) : hnm) : 0.0;
            exc = exc_code(r1, r2, a1, a2);
        }
        sink.template post<W>(valid, idx, m, hnm, hd, om, psim, exc);
    }
}

// ------------------------------------------------------------------ overlaps outside the CAS
//
// O(m) of a determinant m with active remnant A, c core holes and v virtual electrons (scn, sv of them
// alpha): the warp builds the candidate list of (A, c, v, scn, sv) once (row_list), and every m of that
// class sums it with its own orbitals' part of the table index (row_overlap).  The sum's sign is m's
// up to (-1)^(core-hole positions).

// the candidate list in shared memory; its signs are those of the class's first determinant (core holes
// and virtual electrons in the lowest orbitals).  Returns the entries, n1 of them singles.
template <int W, class C>
__device__ __noinline__ int row_list(const SysDev& S, unsigned long long AO, int c, int v, int scn, int sv, double* cphi,
                                     unsigned* ccode, int& n1, int lane, C& ctr) {
    const unsigned amask = (S.na >= 32) ? 0xFFFFFFFFu : ((1u << S.na) - 1u);
    const unsigned long long AE = ~AO & ((unsigned long long)amask | ((unsigned long long)amask << 32));
    int xc[2] = {0, 0}, yv[2] = {0, 0};
    shape_decode(S, S.nc, c, scn, 0, 0, xc, S.mag_c);
    shape_decode(S, S.nv, v, sv, S.nc + S.na, 0, yv, S.mag_v);
    unsigned long long m[2][W];
#pragma unroll
    for (int sg = 0; sg < 2; sg++) {
        const unsigned long long a = sg ? AO >> 32 : AO & 0xFFFFFFFFull;
#pragma unroll
        for (int w = 0; w < W; w++) {
            const int sh = S.nc - 64 * w;                      // the active block may straddle a word
            m[sg][w] = S.mcore[w] | ((sh >= 0 ? (sh < 64 ? a << sh : 0ull) : (sh > -64 ? a >> -sh : 0ull)) & S.mact[w]);
        }
    }
    int par = 0;
    for (int k = 0; k < c; k++) {
        const int x = xc[k] - (xc[k] >= S.n ? S.n : 0);
        flip_reg<W>(m, xc[k] >= S.n, x);
        par += x;
    }
    for (int k = 0; k < v; k++) flip_reg<W>(m, yv[k] >= S.n, yv[k] - (yv[k] >= S.n ? S.n : 0));
    return build_group_list<W, true>(S, MRQ_EMPTY_KEY, m, AO, AE, c, v, scn, sv, xc[0], xc[1], yv[0], yv[1], par, cphi,
                                     ccode, n1, lane, ctr);
}

// candidates e, e + st, ... < count: w T[base + lane part]
__device__ __forceinline__ double row_doubles(const double* __restrict__ tab, const double* cphi, const unsigned* ccode,
                                              int e, int count, int st, unsigned offd, unsigned offx) {
    double a0 = 0.0, a1 = 0.0;
    for (; e + 3 * st < count; e += 4 * st) {
        const unsigned p0 = ccode[e], p1 = ccode[e + st], p2 = ccode[e + 2 * st], p3 = ccode[e + 3 * st];
        const double x0 = __ldg(tab + (p0 & 0x7FFFFFFFu) + ((p0 & 0x80000000u) ? offx : offd));
        const double x1 = __ldg(tab + (p1 & 0x7FFFFFFFu) + ((p1 & 0x80000000u) ? offx : offd));
        const double x2 = __ldg(tab + (p2 & 0x7FFFFFFFu) + ((p2 & 0x80000000u) ? offx : offd));
        const double x3 = __ldg(tab + (p3 & 0x7FFFFFFFu) + ((p3 & 0x80000000u) ? offx : offd));
        a0 = fma(cphi[e], x0, a0);
        a1 = fma(cphi[e + st], x1, a1);
        a0 = fma(cphi[e + 2 * st], x2, a0);
        a1 = fma(cphi[e + 3 * st], x3, a1);
    }
    for (; e < count; e += st) {
        const unsigned p0 = ccode[e];
        a0 = fma(cphi[e], __ldg(tab + (p0 & 0x7FFFFFFFu) + ((p0 & 0x80000000u) ? offx : offd)), a0);
    }
    return a0 + a1;
}

// The list's sum for the determinant with core holes xc and virtual electrons yv (sorted), the entries
// part, part + f, ... of it added over f neighbouring lanes; par is its core parity.  A single candidate
// x -> y takes h_yx + sum over the remnant's electrons j of (yx|jj) - (yj|jx): m's own hole y and electron
// x drop out.  A double is one table read and one FMA.
__device__ __forceinline__ double row_overlap(const SysDev& S, unsigned long long AO, int c, int v, int xc0, int xc1, int yv0,
                                              int yv1, const double* cphi, const unsigned* ccode, int n1, int count, int part,
                                              int f, int& par) {
    unsigned offd, offx;
    lane_offsets(S, c, v, xc0, xc1, yv0, yv1, offd, offx, par);
    double s = 0.0;
    for (int e = part; e < n1; e += f) {
        const unsigned code = ccode[e];
        const int x = v ? yv0 : act_so(S, (int)(code & 127u)), y = c ? xc0 : act_so(S, (int)((code >> 14) & 127u));
        const int sx = x >= S.n, px = x - sx * S.n, py = y - sx * S.n;
        double g = __ldg(S.hc + py * S.n + px);
        const double* const col = S.sgl + py * S.nav + (px - S.nc);
        for (unsigned long long bits = AO; bits; bits &= bits - 1) {
            const int b = __ffsll(bits) - 1;
            g += __ldg(col + (long long)((b & 31) + (((b >= 32) == (sx == 1)) ? 0 : S.na)) * S.nca * S.nav);
        }
        s = fma(cphi[e], g, s);
    }
    s += row_doubles(S.tab, cphi, ccode, n1 + part, count, f, offd, offx);
    for (int o = f >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

// label of core holes xc and virtual electrons yv (sorted)
__device__ __forceinline__ long long row_label(const SysDev& S, int c, int v, int xc0, int xc1, int yv0, int yv1) {
    const int voff = S.nc + S.na;
    const int h0 = xc0 >= S.n ? S.nc + (xc0 - S.n) : xc0, h1 = xc1 >= S.n ? S.nc + (xc1 - S.n) : xc1;
    const int p0 = yv0 >= S.n ? S.nv + (yv0 - S.n - voff) : yv0 - voff;
    const int p1 = yv1 >= S.n ? S.nv + (yv1 - S.n - voff) : yv1 - voff;
    return set_rank(c, h0, h1, 2 * S.nc) * S.nPs + set_rank(v, p0, p1, 2 * S.nv);
}

// core holes and virtual electrons of a determinant (at most two each, spin orbitals, sorted)
template <int W>
__device__ __forceinline__ void outer_orbitals(const SysDev& S, const unsigned long long (&m)[2][W], int& c, int& v, int* xc,
                                               int* yv) {
    c = v = 0;
    xc[0] = xc[1] = yv[0] = yv[1] = 0;
#pragma unroll
    for (int sg = 0; sg < 2; sg++) {
        unsigned long long hm = ~m[sg][0] & S.mcore[0];
        while (hm) {
            const int i = __ffsll(hm) - 1;
            hm &= hm - 1;
            if (c == 0) xc[0] = sg * S.n + i;
            else xc[1] = sg * S.n + i;
            c++;
        }
#pragma unroll
        for (int w = 0; w < W; w++) {
            unsigned long long pm = m[sg][w] & S.mvirt[w];
            while (pm) {
                const int a = 64 * w + __ffsll(pm) - 1;
                pm &= pm - 1;
                if (v == 0) yv[0] = sg * S.n + a;
                else yv[1] = sg * S.n + a;
                v++;
            }
        }
    }
}

// O(m) of one first-order determinant by a whole warp
template <int W>
__device__ __noinline__ double reach_back_warp(const SysDev& S, const unsigned long long (&m)[2][W], double* cphi,
                                               unsigned* ccode, int lane) {
    int c, v, xc[2], yv[2];
    outer_orbitals<W>(S, m, c, v, xc, yv);
    const int scn = (c >= 1 && xc[0] < S.n) + (c == 2 && xc[1] < S.n), sv = (v >= 1 && yv[0] < S.n) + (v == 2 && yv[1] < S.n);
    const unsigned long long AO =
        (unsigned long long)active_bits<W>(S, m[0]) | ((unsigned long long)active_bits<W>(S, m[1]) << 32);
    NoCtr ctr;
    int n1, par;
    const int count = row_list<W>(S, AO, c, v, scn, sv, cphi, ccode, n1, lane, ctr);
    const double s = row_overlap(S, AO, c, v, xc[0], xc[1], yv[0], yv[1], cphi, ccode, n1, count, lane, 32, par);
    __syncwarp();
    return neg_if(s, par);
}

// ------------------------------------------------------------------ a determinant's constants

// the determinant's single-excitation operator G_yx(n) = h_yx + sum_{j in n} [(yx|jj) - delta (yj|jx)]
// for y in core + active, x in active + virtual (not both active), by a whole block: the full-core
// operator hc, n's active electrons, minus n's core holes, plus its virtual electrons
template <int W, class C>
__device__ void walker_operator(const SysDev& S, const unsigned long long (&n)[2][W], bool cas, double* gops, C& ctr) {
    const unsigned ao0 = active_bits<W>(S, n[0]), ao1 = active_bits<W>(S, n[1]);
    const unsigned long long AOn = (unsigned long long)ao0 | ((unsigned long long)ao1 << 32);
    int nh = 0, np = 0, hso[2] = {0, 0}, pso[2] = {0, 0};
    if (!cas) {
#pragma unroll
        for (int sg = 0; sg < 2; sg++) {
            unsigned long long hm = ~(sg ? n[1][0] : n[0][0]) & S.mcore[0];
            while (hm) {
                const int i = __ffsll(hm) - 1;
                hm &= hm - 1;
                if (nh == 0) hso[0] = sg * S.n + i;
                else hso[1] = sg * S.n + i;
                nh++;
            }
#pragma unroll
            for (int w = 0; w < W; w++) {
                unsigned long long pm = (sg ? n[1][w] : n[0][w]) & S.mvirt[w];
                while (pm) {
                    const int a = 64 * w + __ffsll(pm) - 1;
                    pm &= pm - 1;
                    if (np == 0) pso[0] = sg * S.n + a;
                    else pso[1] = sg * S.n + a;
                    np++;
                }
            }
        }
    }
    const int blk = S.nca * S.nav;
    for (int t = threadIdx.x; t < 2 * blk; t += blockDim.x) {
        const int sg = t >= blk, rem = t - sg * blk;
        const int y = rem / S.nav, xo = rem - y * S.nav, x = S.nc + xo;
        if (y >= S.nc && xo < S.na) continue;
        ctr.g();
        double v = __ldg(S.hc + y * S.n + x);
        unsigned long long bits = AOn;
        while (bits) {
            const int b = __ffsll(bits) - 1;
            bits &= bits - 1;
            const int j = S.nc + (b & 31);
            v += eri_g(S, y, x, j, j);
            ctr.g();
            if ((b >= 32) == (sg == 1)) {
                v -= eri_g(S, y, j, j, x);
                ctr.g();
            }
        }
#pragma unroll
        for (int k = 0; k < 2; k++) {
            if (k < nh) {
                v -= g_corr(S, sg, x, y, hso[k]);
                ctr.g(2);
            }
            if (k < np) {
                v += g_corr(S, sg, x, y, pso[k]);
                ctr.g(2);
            }
        }
        gops[t] = v;
    }
}

template <int W>
__device__ __forceinline__ CasWalker cas_constants(const SysDev& S, const unsigned long long (&n)[2][W], double phin) {
    CasWalker cw;
    const unsigned ao0 = active_bits<W>(S, n[0]), ao1 = active_bits<W>(S, n[1]);
    const unsigned amask = (S.na >= 32) ? 0xFFFFFFFFu : ((1u << S.na) - 1u);
    cw.AOn = (unsigned long long)ao0 | ((unsigned long long)ao1 << 32);
    cw.AEn = (unsigned long long)(~ao0 & amask) | ((unsigned long long)(~ao1 & amask) << 32);
    cw.keyn = hash_key(S, ao0, ao1);
    cw.cntO = __popcll(cw.AOn);
    cw.cntE = __popcll(cw.AEn);
    cw.c0 = __ldg(S.c);
    cw.phin = phin;
    return cw;
}

// ------------------------------------------------------------------ the move race

// Philox4x32-10 of counter (exc, step, walker, 0): after two rounds the state is a mix of words that
// depend on the excitation alone and words that depend on the walker alone, so both halves are made
// once (race_walker_words per walker and task, the excitation's per neighbour) and a clock costs the
// last eight rounds, of which the last needs one product: 15 products instead of 20.
#define PHILOX_M0 0xD2511F53u
#define PHILOX_M1 0xCD9E8D57u
#define PHILOX_W0 0x9E3779B9u
#define PHILOX_W1 0xBB67AE85u

struct WarpTask {
    SysDev sys;                         // the system of the task's walkers
    CasWalker cw;
    unsigned long long nsh[4];
    double inv_psin;
    float inv_f;                        // FP32 |1/psi_s(n)| (INFINITY when FP32 cannot carry it)
    int qn;                             // neighbours waiting in the queue
    uint4 wp[MRQ_TGW];                  // per walker: Philox words (x, y) and screen scale (w, FP32)
    unsigned wid[MRQ_TGW], step[MRQ_TGW], slot[MRQ_TGW];
    float bnd[MRQ_TGW];                 // upper bound of the best clock
    RaceBest best[MRQ_TGW];             // the task's best candidate
    double qt[96];                      // queued neighbours: t and excitation
    unsigned qe[96];
};

// the screen's scale of a walker whose best clock is at most `bound`: a neighbour of rate Gamma =
// |t / psi_n| can win only if w = 1 - u < -expm1(-Gamma bound) <= Gamma bound, i.e. if the top 32
// bits of w, as an integer, are below |t| x this scale.  The factor 1.0001 covers the FP32 roundings,
// the floor keeps the scale in the normal range (a larger scale only lets more through).
__device__ __forceinline__ float race_scale(float bound, float inv_f) {
    return fmaxf(bound * inv_f * 1.0001f * 4294967296.0f, 1e-30f);
}

// the screen on the top 32 bits x of the draw (gf: FP32 rate, or |t| when the scale holds 1/psi_n;
// negative: no neighbour, INFINITY: a rate FP32 cannot carry)
__device__ __forceinline__ bool race_pass(unsigned x, float gf, float scale) { return (float)(~x) <= gf * scale; }

__device__ __forceinline__ uint4 race_walker_words(unsigned long long seed, unsigned step, unsigned wid) {
    const unsigned kx = (unsigned)seed, ky = (unsigned)(seed >> 32);
    const unsigned x1 = __umulhi(PHILOX_M1, wid) ^ step ^ kx, y1 = PHILOX_M1 * wid;      // round 1
    uint4 r;
    r.x = y1 ^ (kx + PHILOX_W0);                                                         // round 2
    r.y = __umulhi(PHILOX_M0, x1) ^ (ky + PHILOX_W1);
    r.z = PHILOX_M0 * x1;
    r.w = 0u;
    return r;
}

__device__ __forceinline__ bool atomic_cas128(RaceBest* at, const RaceBest& cmp, const RaceBest& val, RaceBest& old) {
    const unsigned long long c0 = (unsigned long long)cmp.clk | ((unsigned long long)cmp.exc << 32);
    const unsigned long long v0 = (unsigned long long)val.clk | ((unsigned long long)val.exc << 32);
    const unsigned long long c1 = (unsigned long long)__double_as_longlong(cmp.t);
    const unsigned long long v1 = (unsigned long long)__double_as_longlong(val.t);
    unsigned long long o0, o1;
    asm volatile("{\n\t.reg .b128 c, v, d;\n\t"
                 "mov.b128 c, {%2, %3};\n\tmov.b128 v, {%4, %5};\n\t"
                 "atom.global.cas.b128 d, [%6], c, v;\n\t"
                 "mov.b128 {%0, %1}, d;\n\t}"
                 : "=l"(o0), "=l"(o1)
                 : "l"(c0), "l"(c1), "l"(v0), "l"(v1), "l"(at)
                 : "memory");
    old.clk = (unsigned)o0;
    old.exc = (unsigned)(o0 >> 32);
    old.t = __longlong_as_double((long long)o1);
    return o0 == c0 && o1 == c1;
}

// one 128-bit access: a vector load is four scalar ones to the memory model, and could mix the clock and
// excitation of one candidate with the t of another
__device__ __forceinline__ RaceBest load_best128(const RaceBest* at) {
    unsigned long long o0, o1;
    asm volatile("{\n\t.reg .b128 d;\n\t"
                 "ld.relaxed.gpu.global.b128 d, [%2];\n\t"
                 "mov.b128 {%0, %1}, d;\n\t}"
                 : "=l"(o0), "=l"(o1)
                 : "l"(at)
                 : "memory");
    RaceBest b;
    b.clk = (unsigned)o0;
    b.exc = (unsigned)(o0 >> 32);
    b.t = __longlong_as_double((long long)o1);
    return b;
}

// Whether two FP32 clocks leave the order of the exact ones open.  Their relative error is below 1e-5 within
// FP32's normal range; below and above it (rates near 1e38 or 1e-38 and beyond) the exact clocks always decide.
__device__ __forceinline__ bool clocks_near(float a, float b) {
    const float lo = fminf(a, b), hi = fmaxf(a, b);
    return !(lo < hi * 0.9999f) | (hi < 1e-30f) | (lo > 1e37f);
}

// FP32 upper bound of the clock whose FP32 image is a.  Images below the normal range may have lost all their
// bits, so the bound never falls below 1e-37 (which keeps race_scale away from 0 times infinity, too).
__device__ __forceinline__ float race_bound(float a) { return fmaxf(a * 1.0001f, 1e-37f); }

// Whether a candidate (FP32 clock a; draw k, rate g, excitation) beats `cur`: by the FP32 clocks, near ties
// by the exact FP64 ones, then by the smaller excitation
__device__ __forceinline__ bool race_better(const WarpTask& wt, int j, float a, unsigned long long k, double g, unsigned exc,
                                            const RaceBest& cur) {
    if (cur.exc == 0xFFFFFFFFu) return true;
    const float ca = __uint_as_float(cur.clk);
    if (!clocks_near(a, ca)) return a < ca;
    const double tm = race_clock_f64(k, g);
    const double tb = race_clock_f64(race_bits(wt.sys.seed, cur.exc, wt.step[j], wt.wid[j]), fabs(cur.t * wt.inv_psin));
    return tm < tb || (tm == tb && exc < cur.exc);
}

// Some lane's neighbour passed walker j's screen: of those that pass the closer one (race_may_win) take
// the smallest clock (near ties by the exact FP64 clocks, then the smaller excitation) as the task's best
// candidate if it beats that.  Runs a handful of times per walker and task and touches shared memory only;
// the tasks' candidates meet in race_publish.
__device__ __noinline__ void race_slow(WarpTask& wt, int j, double t, unsigned exc, int lane) {
    const unsigned long long seed = wt.sys.seed;
    const unsigned step = wt.step[j], wid = wt.wid[j];
    const unsigned long long k = race_bits(seed, exc, step, wid);
    const double g = fabs(t * wt.inv_psin);
    const float gf = abs_f32_of(g);
    const bool ok = g > 0.0 && race_may_win(k, gf, wt.bnd[j]);
    float a = INFINITY;
    if (ok) {
        const float w = (float)(9007199254740991ull - k) * 1.1102230246251565e-16f;
        if (gf > 0.0f) a = (w > 0.5f ? -logf((float)(k + 1) * 1.1102230246251565e-16f) : -log1pf(-w)) / gf;
        else a = (float)race_clock_f64(k, g);
    }
    float amin = a;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amin = fminf(amin, __shfl_xor_sync(0xffffffffu, amin, o));
    unsigned near = __ballot_sync(0xffffffffu, ok && clocks_near(a, amin));
    if (near == 0u) return;
    int src = __ffs(near) - 1;
    if (near & (near - 1u)) {
        double tc = INFINITY;
        unsigned e = 0xFFFFFFFFu;
        if (near >> lane & 1u) {
            tc = race_clock_f64(k, g);
            e = exc;
        }
        double tm = tc;
        unsigned em = e;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double t2 = __shfl_xor_sync(0xffffffffu, tm, o);
            const unsigned e2 = __shfl_xor_sync(0xffffffffu, em, o);
            if (t2 < tm || (t2 == tm && e2 < em)) {
                tm = t2;
                em = e2;
            }
        }
        src = __ffs(__ballot_sync(0xffffffffu, (near >> lane & 1u) && tc == tm && e == em)) - 1;
        if (src < 0) src = __ffs(near) - 1;
    }
    if (lane == src && race_better(wt, j, a, k, g, exc, wt.best[j])) {
        wt.best[j].clk = __float_as_uint(a);
        wt.best[j].exc = exc;
        wt.best[j].t = t;
        const float up = race_bound(a);
        if (up < wt.bnd[j]) {
            wt.bnd[j] = up;
            wt.wp[j].w = __float_as_uint(race_scale(up, wt.inv_f));
        }
    }
    __syncwarp();
}

// the task's best candidates against the walkers' (one walker per lane): replaced by a 128-bit
// compare-and-swap, and the bounds lowered for the tasks that begin later
__device__ __noinline__ void race_publish(const WarpTask& wt, RaceBest* best, unsigned* bound, int count, int lane) {
    if (lane >= count || wt.best[lane].exc == 0xFFFFFFFFu) return;
    const RaceBest mine = wt.best[lane];
    const float a = __uint_as_float(mine.clk);
    const unsigned long long k = race_bits(wt.sys.seed, mine.exc, wt.step[lane], wt.wid[lane]);
    const double g = fabs(mine.t * wt.inv_psin);
    RaceBest* const at = best + (int)wt.slot[lane];
    RaceBest cur = load_best128(at), old;
    while (race_better(wt, lane, a, k, g, mine.exc, cur)) {     // every turn but the last, another task's candidate won
        if (atomic_cas128(at, cur, mine, old)) break;
        cur = old;
    }
    atomicMin(bound + (int)wt.slot[lane], __float_as_uint(race_bound(a)));
}

// the FP32 |t| of the screen
__device__ __forceinline__ float race_rate(double t) {
    if ((__double_as_longlong(t) << 1) == 0) return -1.0f;          // no neighbour: never passes
    const float gf = abs_f32_of(t);
    return gf == 0.0f ? INFINITY : gf;                              // outside FP32: the exact clock decides
}

// 64 neighbours (two per lane; t = 0: none) against the clocks of the task's walkers; returns the
// walkers that some neighbour may win.  Bound by the integer pipes: 15 products and about 20 logic
// operations per neighbour and walker.  Two neighbours per lane share a walker's words and the loop; the
// rare candidates are settled by the caller, so that the loop holds no call and spills nothing.
__device__ __noinline__ unsigned race_round(const WarpTask& wt, double t0, unsigned exc0, double t1, unsigned exc1,
                                            int count) {
    const float gf0 = race_rate(t0), gf1 = race_rate(t1);
    const unsigned kx = (unsigned)wt.sys.seed, ky = (unsigned)(wt.sys.seed >> 32);
    const unsigned za = __umulhi(PHILOX_M0, exc0) ^ ky, wa = PHILOX_M0 * exc0;
    const unsigned zb = __umulhi(PHILOX_M0, exc1) ^ ky, wb = PHILOX_M0 * exc1;
    const unsigned ha = __umulhi(PHILOX_M1, za), la = PHILOX_M1 * za;
    const unsigned hb = __umulhi(PHILOX_M1, zb), lb = PHILOX_M1 * zb;
    unsigned hits = 0;
    for (int j = 0; j < count; j++) {
        const uint4 a = wt.wp[j];
        unsigned c0 = ha ^ a.x, c1 = la, c2 = wa ^ a.y, c3 = a.z;
        unsigned d0 = hb ^ a.x, d1 = lb, d2 = wb ^ a.y, d3 = a.z;
#pragma unroll
        for (int r = 2; r < 9; r++) {
            const unsigned k0 = kx + (unsigned)r * PHILOX_W0, k1 = ky + (unsigned)r * PHILOX_W1;
            const unsigned long long p0 = (unsigned long long)PHILOX_M0 * c0, p1 = (unsigned long long)PHILOX_M1 * c2;
            const unsigned long long q0 = (unsigned long long)PHILOX_M0 * d0, q1 = (unsigned long long)PHILOX_M1 * d2;
            c0 = (unsigned)(p1 >> 32) ^ c1 ^ k0;
            c1 = (unsigned)p1;
            c2 = (unsigned)(p0 >> 32) ^ c3 ^ k1;
            c3 = (unsigned)p0;
            d0 = (unsigned)(q1 >> 32) ^ d1 ^ k0;
            d1 = (unsigned)q1;
            d2 = (unsigned)(q0 >> 32) ^ d3 ^ k1;
            d3 = (unsigned)q0;
        }
        const unsigned k9 = kx + 9u * PHILOX_W0;
        const unsigned x = __umulhi(PHILOX_M1, c2) ^ c1 ^ k9, y = __umulhi(PHILOX_M1, d2) ^ d1 ^ k9;
        const float scale = __uint_as_float(a.w);
        if (__any_sync(0xffffffffu, race_pass(x, gf0, scale) || race_pass(y, gf1, scale))) hits |= 1u << j;
    }
    return hits;
}

// neighbours of a walk step: queued so that the sums and the race run with full lanes
struct StepSink {
    WarpTask& wt;
    RaceBest* best;
    unsigned* bound;
    int count, lane;
    bool primary;             // this task group stores the determinant's sums
    double sA, sT, sD;        // sum |t|, sum t, sum t_D   (t = H_nm psi_s(m), t_D = (H_D)_nm psi_s(m))
    template <int W>
    __device__ __forceinline__ void post(bool valid, int, const unsigned long long (&)[2][W], double hnm, double hd,
                                         double, double psim, unsigned exc) {
        if (valid) sD += hd * psim;
        push(valid, hnm * psim, exc);
    }
    __device__ __forceinline__ void push(bool valid, double t, unsigned exc) {
        const bool on = valid && (__double_as_longlong(t) << 1) != 0;
        const unsigned m = __ballot_sync(0xffffffffu, on);
        int qn = wt.qn;
        if (on) {
            const int at = qn + __popc(m & ((1u << lane) - 1u));
            wt.qt[at] = t;
            wt.qe[at] = exc;
        }
        qn += __popc(m);
        __syncwarp();
        if (qn >= 64) {
            take(wt.qt[lane], wt.qe[lane], wt.qt[32 + lane], wt.qe[32 + lane]);
            qn -= 64;
            const double t2 = wt.qt[64 + lane];
            const unsigned e2 = wt.qe[64 + lane];
            __syncwarp();
            if (lane < qn) {
                wt.qt[lane] = t2;
                wt.qe[lane] = e2;
            }
        }
        if (lane == 0) wt.qn = qn;
        __syncwarp();
    }
    __device__ __forceinline__ void take(double t0, unsigned e0, double t1, unsigned e1) {
        if (primary) {
            sA += fabs(t0);
            sT += t0;
            sA += fabs(t1);
            sT += t1;
        }
        for (unsigned hits = race_round(wt, t0, e0, t1, e1, count); hits; hits &= hits - 1) {
            const int j = __ffs(hits) - 1;
            race_slow(wt, j, t0, e0, lane);
            race_slow(wt, j, t1, e1, lane);
        }
    }
    __device__ __forceinline__ void finish() {
        const int qn = wt.qn;
        if (qn > 0)
            take(lane < qn ? wt.qt[lane] : 0.0, lane < qn ? wt.qe[lane] : 0u, 32 + lane < qn ? wt.qt[32 + lane] : 0.0,
                 32 + lane < qn ? wt.qe[32 + lane] : 0u);
        __syncwarp();
        race_publish(wt, best, bound, count, lane);
        __syncwarp();
    }
};

// the debug evaluation's neighbours: sums, and records when asked for
struct DebugSink {
    mrq_neighbour* nbout;
    long long nbase, max_nb;
    double inv_psin;
    double sA, sT, sD;
    template <int W>
    __device__ __forceinline__ void post(bool valid, int ri, const unsigned long long (&m)[2][W], double hnm, double hd,
                                         double om, double psim, unsigned exc) {
        if (!valid) return;
        const double t = hnm * psim;
        sA += fabs(t);
        sT += t;
        sD += hd * psim;
        if (nbout != nullptr && nbase + ri < max_nb) {
            unsigned long long w4[4];
            det_words<W>(m, w4);
            write_rec(nbout + nbase + ri, w4, W, hnm, hd, om, psim, fabs(t * inv_psin), exc);
        }
    }
};

// ------------------------------------------------------------------ kernels of a walk step

template <int W>
__device__ __forceinline__ void load_det(const Walker* w, unsigned long long (&n)[2][W]) {
#pragma unroll
    for (int sg = 0; sg < 2; sg++)
#pragma unroll
        for (int k = 0; k < W; k++) n[sg][k] = w->d[sg][k];
}

__device__ __forceinline__ void copy_sys(SysDev* dst, const SysDev* src, int t, int nt) {
    for (int k = t; k < (int)(sizeof(SysDev) / sizeof(int)); k += nt)
        reinterpret_cast<int*>(dst)[k] = reinterpret_cast<const int*>(src)[k];
}

// Distinct determinants of the walkers of system blockIdx.x (slots of the segment), by one block: an
// open-addressing table whose entries hold the first walker seen on a determinant (full determinants
// are compared, so a hash collision costs a probe only).  The table has at least twice as many entries
// as walkers, so a probe always ends.  Task groups and members come out in no fixed order; nothing
// computed from them depends on it.
template <int W>
__global__ void __launch_bounds__(1024) k_group(const WalkSet ws, const WalkScratch sc) {
    const int sys = blockIdx.x;
    const long long off = ws.offsets[sys];
    const long long lo = max(off, sc.seg0) - off, hi = min(ws.offsets[sys + 1], sc.seg1) - off;
    const int n = (int)max(0LL, hi - lo);
    const Walker* const wk = ws.walkers[sys] + lo;
    const int base = (int)(off + lo - sc.seg0);          // first slot of the system in the segment
    const SysDev& S = ws.systems[sys];
    __shared__ int s_members;
    if (threadIdx.x == 0) s_members = 0;
    if (gridDim.x == 1 && threadIdx.x < CTL_N) sc.ctl[threadIdx.x] = 0;
    int tsz = 2;
    while (tsz < 2 * n) tsz <<= 1;
    int* const rep = sc.rep + 4LL * base;
    int* const cnt = sc.cnt + 4LL * base;
    int* const start = sc.start + 4LL * base;
    if (n > 0)
        for (int k = threadIdx.x; k < tsz; k += blockDim.x) {
            rep[k] = -1;
            cnt[k] = 0;
        }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        unsigned long long d[2][W];
        load_det<W>(wk + i, d);
        unsigned long long hh = 0;
#pragma unroll
        for (int sg = 0; sg < 2; sg++)
#pragma unroll
            for (int w = 0; w < W; w++) hh = mix64(hh ^ d[sg][w]);
        int k = (int)(hh & (unsigned long long)(tsz - 1));
        for (int probe = 0; probe < tsz; probe++) {
            const int prev = atomicCAS(rep + k, -1, i);
            bool same = prev < 0;
            if (!same) {
                unsigned long long o[2][W];
                load_det<W>(wk + prev, o);
                same = true;
#pragma unroll
                for (int sg = 0; sg < 2; sg++)
#pragma unroll
                    for (int w = 0; w < W; w++) same = same && o[sg][w] == d[sg][w];
            }
            if (same) break;
            k = (k + 1) & (tsz - 1);
        }
        sc.tab_of[base + i] = k;
        sc.pos_of[base + i] = atomicAdd(cnt + k, 1);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < (n > 0 ? tsz : 0); k += blockDim.x) {
        const int c = cnt[k];
        if (c == 0) continue;
        const int st = atomicAdd(&s_members, c);
        start[k] = st;
        unsigned long long d[2][W];
        load_det<W>(wk + rep[k], d);
        bool cas = true;
#pragma unroll
        for (int sg = 0; sg < 2; sg++)
#pragma unroll
            for (int w = 0; w < W; w++) cas = cas && (d[sg][w] & S.mcore[w]) == S.mcore[w] && (d[sg][w] & S.mvirt[w]) == 0;
        const int ntg = (c + sc.tgw - 1) / sc.tgw;
        const int at = atomicAdd(sc.ctl + (cas ? CTL_TGC : CTL_TGF), ntg), grp = atomicAdd(sc.ctl + (cas ? CTL_GC : CTL_GF), 1);
        TaskGroup* const tg = cas ? sc.tgc : sc.tgf;
        const int det = cas ? grp : (int)(sc.nseg - 1 - grp);
        GroupMeta m;
        m.d[0][0] = m.d[0][1] = m.d[1][0] = m.d[1][1] = 0;
#pragma unroll
        for (int sg = 0; sg < 2; sg++)
#pragma unroll
            for (int w = 0; w < W; w++) m.d[sg][w] = d[sg][w];
        m.psi = wk[rep[k]].psi;
        m.inv_psi = m.psi != 0.0 ? 1.0 / m.psi : 0.0;
        m.phi = m.psi / __ldg(S.c);
        m.hnn = m.hdnn = 0.0;
        m.label = det_label<W>(S, d, m.h, m.p);
        m.sys = sys;
        m.pad = 0;
        sc.meta[det] = m;
        for (int q = 0; q < ntg; q++) {
            TaskGroup t;
            t.sys = sys;
            t.first = base + st + q * sc.tgw;
            t.count = min(sc.tgw, c - q * sc.tgw);
            t.group = det;
            t.primary = q == 0;
            t.pad = 0;
            tg[at + q] = t;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        sc.members[base + start[sc.tab_of[base + i]] + sc.pos_of[base + i]] = (int)lo + i;
        RaceBest b;
        b.clk = 0x7F800000u;
        b.exc = 0xFFFFFFFFu;
        b.t = 0.0;
        sc.best[base + i] = b;
        sc.bound[base + i] = 0x7F800000u;
    }
}

// Constants of every distinct determinant, one block each: diagonals, single-excitation operator
template <int W>
__global__ void __launch_bounds__(128) k_prep(const WalkSet ws, const WalkScratch sc) {
    __shared__ SysDev S;
    __shared__ WarpLists lists;
    int cur = -1;
    const int ntc = sc.ctl[CTL_TGC], ntg = ntc + sc.ctl[CTL_TGF];
    for (int g = blockIdx.x; g < ntg; g += gridDim.x) {
        const TaskGroup tg = g < ntc ? sc.tgc[g] : sc.tgf[g - ntc];
        if (!tg.primary) continue;
        __syncthreads();
        if (tg.sys != cur) {
            copy_sys(&S, ws.systems + tg.sys, threadIdx.x, blockDim.x);
            cur = tg.sys;
            __syncthreads();
        }
        GroupMeta& meta = sc.meta[tg.group];
        const long long ln = meta.label;
        if (ln < 0) continue;
        unsigned long long n[2][W];
#pragma unroll
        for (int sg = 0; sg < 2; sg++)
#pragma unroll
            for (int w = 0; w < W; w++) n[sg][w] = meta.d[sg][w];
        if (threadIdx.x < 32) {
            double hnn, hdnn;
            build_lists<W>(S, n, lists, meta.h, meta.p, threadIdx.x);
            diagonals<W>(S, lists, n, threadIdx.x, hnn, hdnn);
            if (threadIdx.x == 0) {
                meta.hnn = hnn;
                meta.hdnn = hdnn;
            }
        }
        NoCtr ctr;
        if (meta.psi != 0.0) walker_operator<W>(S, n, ln == 0, sc.gops + (long long)tg.group * sc.gstride, ctr);
    }
}

// ---- warp tasks of k_int, k_pairs and k_fois

// the next task of a warp
__device__ __forceinline__ int next_task(int* counter, int lane) {
    int id = 0;
    if (lane == 0) id = atomicAdd(counter, 1);
    return __shfl_sync(0xffffffffu, id, 0);
}

// the system of a warp's task, in its shared memory
__device__ __forceinline__ void task_system(WarpTask& wt, const WalkSet& ws, int sys, int& cur, int lane) {
    __syncwarp();
    if (sys != cur) {
        copy_sys(&wt.sys, ws.systems + sys, lane, 32);
        cur = sys;
        __syncwarp();
    }
}

// walker `lane` of a task: its Philox words and its screen, from the bound of its best clock so far
__device__ __forceinline__ void race_walker(WarpTask& wt, int lane, unsigned step, unsigned wid, int slot, const unsigned* bound,
                                            float inv_f) {
    uint4 a = race_walker_words(wt.sys.seed, step, wid);
    const float b = __uint_as_float(__ldcg(bound + slot));
    a.w = __float_as_uint(race_scale(b, inv_f));
    wt.bnd[lane] = b;
    wt.wp[lane] = a;
    wt.wid[lane] = wid;
    wt.step[lane] = step;
    wt.slot[lane] = (unsigned)slot;
    wt.best[lane].exc = 0xFFFFFFFFu;
}

// FP32 |1/psi_s(n)| of the screen; INFINITY (every neighbour passes) where FP32 cannot carry it
__device__ __forceinline__ float race_inv(double inv) {
    const float f = abs_f32_of(inv);
    return f > 0.0f ? f : INFINITY;
}

// the determinant of a task group and the Philox words and screens of its walkers; false when it cannot
// be evaluated (outside the first-order space, or psi_s = 0)
template <int W>
__device__ __forceinline__ bool task_begin(WarpTask& wt, const WalkSet& ws, const WalkScratch& sc, const TaskGroup& tg,
                                           int lane) {
    const GroupMeta* const meta = sc.meta + tg.group;
    if (meta->label < 0 || !(meta->psi != 0.0)) return false;
    if (lane < 2 * W) wt.nsh[lane] = meta->d[lane / W][lane % W];
    const double inv = meta->inv_psi;
    const float inv_f = race_inv(inv);
    if (lane < tg.count) {
        const int i = sc.members[tg.first + lane];
        const Walker* const wk = ws.walkers[tg.sys] + i;
        race_walker(wt, lane, wk->step, wk->wid, (int)(ws.offsets[tg.sys] + i - sc.seg0), sc.bound, inv_f);
    }
    if (lane == 0) {
        wt.inv_psin = inv;
        wt.inv_f = inv_f;
        wt.qn = 0;
    }
    __syncwarp();
    return true;
}

// partial sums of a task, stored by the determinant's primary group (D: with the H_D numerator)
template <bool D>
__device__ __forceinline__ void task_sums(const WalkScratch& sc, const TaskGroup& tg, int slice, double sA, double sT,
                                          double sD, int lane) {
    if (!tg.primary) return;
    sA = warp_sum(sA);
    sT = warp_sum(sT);
    if (D) sD = warp_sum(sD);
    if (lane == 0) {
        double* const p = sc.part + ((long long)tg.group * (sc.ns_max + MRQ_ACT_SLICES) + slice) * 3;
        p[0] = sA;
        p[1] = sT;
        p[2] = sD;
    }
}

// neighbours inside the CAS.  They carry most of the total rate, so they run first: the later kernels
// start with nearly final screens.
template <int W>
__global__ void __launch_bounds__(256, 3) k_int(const WalkSet ws, const WalkScratch sc) {
    __shared__ WarpTask tasks[8];
    const int lane = threadIdx.x & 31;
    WarpTask& wt = tasks[threadIdx.x >> 5];
    const SysDev& S = wt.sys;
    int cur = -1;
    const int ntg = sc.ctl[CTL_TGC];
    NoCtr ctr;
    for (;;) {
        const int id = next_task(sc.ctl + CTL_INT, lane);
        if (id >= ntg * MRQ_INT_SLICES) break;
        const int slice = id / ntg;
        const TaskGroup tg = sc.tgc[id - slice * ntg];
        task_system(wt, ws, tg.sys, cur, lane);
        double sA = 0.0, sT = 0.0;
        if (task_begin<W>(wt, ws, sc, tg, lane)) {
            const unsigned long long(&n)[2][W] = *reinterpret_cast<const unsigned long long(*)[2][W]>(wt.nsh);
            if (lane == 0) wt.cw = cas_constants<W>(S, n, sc.meta[tg.group].phi);
            __syncwarp();
            StepSink sink{wt, sc.best, sc.bound, tg.count, lane, tg.primary != 0, 0.0, 0.0, 0.0};
            for (int u = slice; u < S.cas_units; u += MRQ_INT_SLICES) cas_internal_unit<W>(S, wt.cw, n, u, lane, sink, ctr);
            sink.finish();
            sA = sink.sA;
            sT = sink.sT;
        }
        task_sums<false>(sc, tg, sc.ns_max + slice, sA, sT, 0.0, lane);
    }
}

// ---- first-order determinants

// Neighbours that move active electrons only (the determinant's own label), one per lane: each has an
// active remnant of its own, so there is no list to share.
template <int W>
__global__ void __launch_bounds__(256, 3) k_fois_act(const WalkSet ws, const WalkScratch sc) {
    __shared__ WarpTask tasks[8];
    const int lane = threadIdx.x & 31;
    WarpTask& wt = tasks[threadIdx.x >> 5];
    const SysDev& S = wt.sys;
    int cur = -1;
    const int ntg = sc.ctl[CTL_TGF];
    NoCtr ctr;
    for (;;) {
        const int id = next_task(sc.ctl + CTL_ACT, lane);
        if (id >= ntg * MRQ_ACT_SLICES) break;
        const int slice = id / ntg;
        const TaskGroup tg = sc.tgf[id - slice * ntg];
        task_system(wt, ws, tg.sys, cur, lane);
        StepSink sink{wt, sc.best, sc.bound, tg.count, lane, tg.primary != 0, 0.0, 0.0, 0.0};
        if (task_begin<W>(wt, ws, sc, tg, lane)) {
            const unsigned long long(&n)[2][W] = *reinterpret_cast<const unsigned long long(*)[2][W]>(wt.nsh);
            const double* const gops = sc.gops + (long long)tg.group * sc.gstride;
            const double cl = __ldg(S.c + sc.meta[tg.group].label);
            const unsigned amask = (S.na >= 32) ? 0xFFFFFFFFu : ((1u << S.na) - 1u);
            const unsigned ao0 = active_bits<W>(S, n[0]), ao1 = active_bits<W>(S, n[1]);
            const unsigned long long oa = ao0, ob = (unsigned long long)ao1 << 32;
            const unsigned long long ea = ~ao0 & amask, eb = (unsigned long long)(~ao1 & amask) << 32;
            const int total = active_neighbours(__popcll(oa), __popcll(ob), __popcll(ea), __popcll(eb));
            for (int base = 32 * slice; base < total; base += 32 * MRQ_ACT_SLICES) {
                double t = 0.0;
                unsigned exc = 0;
                if (base + lane < total) {
                    unsigned long long Xb, Yb, m[2][W];
                    const int r = active_neighbour(S, oa, ob, ea, eb, base + lane, Xb, Yb);
                    int rem[2], add[2];
                    act_list(S, Xb, rem);
                    act_list(S, Yb, add);
#pragma unroll
                    for (int sg = 0; sg < 2; sg++)
#pragma unroll
                        for (int w = 0; w < W; w++) m[sg][w] = n[sg][w];
                    apply_exc<W>(m, S, rem, add, r);
                    const double hnm = r == 1 ? single_elem<W>(S, n, rem[0], add[0], ctr)
                                              : hb_screen(S, double_elem<W>(S, n, rem[0], rem[1], add[0], add[1], ctr));
                    const int r2 = r == 1 ? rem[0] : rem[1], a2 = r == 1 ? add[0] : add[1];
                    const double psim = cl * reach_back<W>(S, m, ctr, MRQ_EMPTY_KEY, 0.0, SglFromWalker{gops, r, rem[0], r2, add[0], a2});
                    sink.sD += (r == 1 ? hd_single_elem<W>(S, n, rem[0], add[0], ctr) : hnm) * psim;
                    t = hnm * psim;
                    exc = exc_code(rem[0], r2, add[0], a2);
                }
                sink.push(true, t, exc);
            }
            sink.finish();
        }
        task_sums<true>(sc, tg, sc.ns_max + slice, sink.sA, sink.sT, sink.sD, lane);
    }
}

// A neighbour of a first-order determinant n moves active electrons X_a -> Y_a and outer ones: core
// electrons X_c and virtual electrons X_v out, core holes Y_c filled, virtual orbitals Y_v entered.  A
// unit is a pair (X_a, Y_a) - one active remnant - and its groups run over the outer patterns; the
// neighbours of a group differ in the orbitals of X_c and Y_v only and share one candidate list.

// core holes and virtual electrons of a first-order determinant and what they leave free
struct FoisOuter {
    int h, p, ha, pa;                 // holes, virtual electrons, alpha ones
    int hs[2], ps[2];                 // spin orbitals, sorted
    int ct[2][2], vt[2][2];           // taken core / virtual positions per spin, ascending (large: none)
    int fc[2], fv[2];                 // free ones
};

template <int W>
__device__ __forceinline__ void fois_outer(const SysDev& S, const unsigned long long (&n)[2][W], FoisOuter& o) {
    int hs[2], ps[2], h, p;
    outer_orbitals<W>(S, n, h, p, hs, ps);
    const int voff = S.nc + S.na, none = 1 << 20;
    const int ha = (h >= 1 && hs[0] < S.n) + (h == 2 && hs[1] < S.n), pa = (p >= 1 && ps[0] < S.n) + (p == 2 && ps[1] < S.n);
    o.h = h;
    o.p = p;
    o.ha = ha;
    o.pa = pa;
    o.hs[0] = hs[0];
    o.hs[1] = hs[1];
    o.ps[0] = ps[0];
    o.ps[1] = ps[1];
    o.ct[0][0] = ha >= 1 ? hs[0] : none;
    o.ct[0][1] = ha == 2 ? hs[1] : none;
    o.ct[1][0] = h - ha >= 1 ? (ha ? hs[1] : hs[0]) - S.n : none;
    o.ct[1][1] = h - ha == 2 ? hs[1] - S.n : none;
    o.vt[0][0] = pa >= 1 ? ps[0] - voff : none;
    o.vt[0][1] = pa == 2 ? ps[1] - voff : none;
    o.vt[1][0] = p - pa >= 1 ? (pa ? ps[1] : ps[0]) - S.n - voff : none;
    o.vt[1][1] = p - pa == 2 ? ps[1] - S.n - voff : none;
    o.fc[0] = S.nc - ha;
    o.fc[1] = S.nc - (h - ha);
    o.fv[0] = S.nv - pa;
    o.fv[1] = S.nv - (p - pa);
}

// the i-th orbital that is neither a nor b (a < b)
__device__ __forceinline__ int skip_two(int i, int a, int b) {
    i += i >= a;
    i += i >= b;
    return i;
}

// choices of cnt orbitals, nal of them alpha, among f0 alpha and f1 beta ones
__device__ __forceinline__ int free_count(int cnt, int nal, int f0, int f1) {
    if (cnt == 0) return 1;
    if (cnt == 1) return nal ? f0 : f1;
    return nal == 1 ? f0 * f1 : (nal == 2 ? f0 * (f0 - 1) / 2 : f1 * (f1 - 1) / 2);
}

// the idx-th choice: sorted spin orbitals; `taken` positions of each spin are left out, orbitals start at off
__device__ __forceinline__ void free_decode(const SysDev& S, int cnt, int nal, const int* f, const int (*taken)[2], int off,
                                            int idx, int& x0, int& x1) {
    if (cnt == 1) {
        const int sg = nal ? 0 : 1;
        x0 = sg * S.n + off + skip_two(idx, taken[sg][0], taken[sg][1]);
    } else if (cnt == 2) {
        int i, j, s0 = 0, s1 = 1;
        if (nal == 1) {
            i = idx / f[1];
            j = idx - i * f[1];
        } else {
            s0 = s1 = nal == 2 ? 0 : 1;
            lex_decode_tab(S.colex, idx, f[s0], i, j);
        }
        x0 = s0 * S.n + off + skip_two(i, taken[s0][0], taken[s0][1]);
        x1 = s1 * S.n + off + skip_two(j, taken[s1][0], taken[s1][1]);
    }
}

__device__ __forceinline__ void put2(int x, int& k, int& a, int& b) {
    if (k == 0) a = x;
    else b = x;
    k++;
}

// Groups of the wave's determinants, one block each: threads take the units in order, count their
// groups and neighbours, and a block scan gives every group its number, which therefore depends on the
// determinant alone (the sums of k_fois run in that order).
template <int W>
__global__ void __launch_bounds__(256) k_fgroups(const WalkSet ws, const WalkScratch sc) {
    const int ng = min(sc.fwave, sc.ctl[CTL_GF] - sc.fwave0);
    __shared__ FoisOuter o;
    __shared__ int s_sum[2][8], s_base[2];
    __shared__ long long s_row;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int g = blockIdx.x; g < ng; g += gridDim.x) {
        const int det = (int)(sc.nseg - 1 - (sc.fwave0 + g));
        const GroupMeta& meta = sc.meta[det];
        const SysDev& S = ws.systems[meta.sys];
        __syncthreads();
        if (meta.label < 0 || !(meta.psi != 0.0)) {
            if (threadIdx.x == 0) sc.fg_of[g] = make_int2(0, 0);
            continue;
        }
        unsigned long long n[2][W];
#pragma unroll
        for (int sg = 0; sg < 2; sg++)
#pragma unroll
            for (int w = 0; w < W; w++) n[sg][w] = meta.d[sg][w];
        if (threadIdx.x == 0) {
            fois_outer<W>(S, n, o);
            s_base[0] = s_base[1] = 0;
        }
        const unsigned ao0 = active_bits<W>(S, n[0]), ao1 = active_bits<W>(S, n[1]);
        const unsigned amask = (S.na >= 32) ? 0xFFFFFFFFu : ((1u << S.na) - 1u);
        const unsigned long long AO = (unsigned long long)ao0 | ((unsigned long long)ao1 << 32);
        const unsigned long long AE = (unsigned long long)(~ao0 & amask) | ((unsigned long long)(~ao1 & amask) << 32);
        const int cntO = __popcll(AO), cntE = __popcll(AE);
        int units = 0;
        for (int k = 0; k < 8; k++) units += nsub(cntO, k / 3) * nsub(cntE, k % 3);
        FGroup* const fg = sc.fg + (long long)g * sc.fg_max;
        __syncthreads();
        // pass 0 counts, then the determinant takes its place in the row buffer; pass 1 writes
        for (int pass = 0; pass < 2; pass++) {
            for (int u0 = 0; u0 < units; u0 += blockDim.x) {
                const int u = u0 + threadIdx.x;
                int ngr = 0, nnb = 0, at = 0, row = 0;
                for (int emit = 0; emit <= pass; emit++) {
                    if (emit) {
                        // exclusive scan of (groups, neighbours) over the block
                        int x = ngr, y = nnb;
#pragma unroll
                        for (int d = 1; d < 32; d <<= 1) {
                            const int x2 = __shfl_up_sync(0xffffffffu, x, d), y2 = __shfl_up_sync(0xffffffffu, y, d);
                            if (lane >= d) {
                                x += x2;
                                y += y2;
                            }
                        }
                        if (lane == 31) {
                            s_sum[0][warp] = x;
                            s_sum[1][warp] = y;
                        }
                        __syncthreads();
                        at = s_base[0] + x - ngr;
                        row = s_base[1] + y - nnb;
                        for (int w = 0; w < warp; w++) {
                            at += s_sum[0][w];
                            row += s_sum[1][w];
                        }
                        __syncthreads();
                        if (threadIdx.x == blockDim.x - 1) {
                            s_base[0] = at + ngr;
                            s_base[1] = row + nnb;
                        }
                    }
                    if (u < units) {
                        int k = 0, pair = u;
                        for (; k < 7; k++) {
                            const int w = nsub(cntO, k / 3) * nsub(cntE, k % 3);
                            if (pair < w) break;
                            pair -= w;
                        }
                        const int ka = k / 3, kb = k % 3, nYa = nsub(cntE, kb), xa = pair / nYa, ya = pair - xa * nYa;
                        const unsigned long long Xb = subset_bits(S.colex, AO, cntO, ka, xa);
                        const unsigned long long Yb = subset_bits(S.colex, AE, cntE, kb, ya);
                        const int da = __popcll(Xb & 0xFFFFFFFFull) - __popcll(Yb & 0xFFFFFFFFull);
                        for (int r = max(1, max(ka, kb)); r <= 2; r++) {
                            const int ko = r - ka, vo = r - kb;              // outer electrons removed / added
                            if (ko == 0 && vo == 0) continue;                // active only: k_fois_act
                            const int na_ = min(ko, o.p) + 1, nb_ = min(vo, o.h) + 1;
                            for (int pat = 0; pat < na_ * nb_ * 4; pat++) {
                                const int av = (pat >> 2) / nb_, bc = (pat >> 2) - av * nb_, xs = pat & 1, ys = (pat >> 1) & 1;
                                if ((xs && !(av == 1 && o.p == 2)) || (ys && !(bc == 1 && o.h == 2))) continue;
                                const int ac = ko - av, bv = vo - bc, c = o.h + ac - bc, v = o.p - av + bv;
                                if (c > 2 || v > 2) continue;
                                const int xva = av == 2 ? o.pa : (av == 1 ? o.ps[xs] < S.n : 0);
                                const int yca = bc == 2 ? o.ha : (bc == 1 ? o.hs[ys] < S.n : 0);
                                for (int sac = 0; sac <= ac; sac++) {
                                    const int sbv = da + xva + sac - yca;
                                    if (sbv < 0 || sbv > bv) continue;
                                    const int ni = free_count(ac, sac, o.fc[0], o.fc[1]) * free_count(bv, sbv, o.fv[0], o.fv[1]);
                                    if (!emit) {
                                        ngr += (ni + MRQ_FG_NB - 1) / MRQ_FG_NB;
                                        nnb += ni;
                                        continue;
                                    }
                                    for (int q = 0; q < ni; q += MRQ_FG_NB) {
                                        FGroup f;
                                        f.ao = (AO & ~Xb) | Yb;
                                        f.off = s_row + row;
                                        f.det = det;
                                        f.q0 = q;
                                        f.nq = min(MRQ_FG_NB, ni - q);
                                        f.c = (unsigned char)c;
                                        f.v = (unsigned char)v;
                                        f.scn = (unsigned char)(o.ha + sac - yca);
                                        f.sv = (unsigned char)(o.pa - xva + sbv);
                                        f.ac = (unsigned char)ac;
                                        f.sac = (unsigned char)sac;
                                        f.bv = (unsigned char)bv;
                                        f.sbv = (unsigned char)sbv;
                                        f.av = (unsigned char)av;
                                        f.bc = (unsigned char)bc;
                                        f.xs = (unsigned char)xs;
                                        f.ys = (unsigned char)ys;
                                        fg[at++] = f;
                                        row += f.nq;
                                    }
                                }
                            }
                        }
                    }
                }
                if (pass == 0) {
                    const int x = __reduce_add_sync(0xffffffffu, nnb);
                    if (lane == 0) atomicAdd(&s_base[1], x);
                }
                __syncthreads();
            }
            if (pass == 0) {
                if (threadIdx.x == 0) {
                    s_row = (long long)atomicAdd(reinterpret_cast<unsigned long long*>(sc.ctl + CTL_FCUR),
                                                 (unsigned long long)((s_base[1] + 3) & ~3));
                    s_base[1] = 0;
                }
                __syncthreads();
            }
        }
        if (threadIdx.x == 0) {
            sc.fg_of[g] = make_int2(g * sc.fg_max, s_base[0]);
            atomicMax(sc.ctl + CTL_FG, s_base[0]);
        }
    }
}

// psi_s of the groups' neighbours, a warp task each: the candidate list once, then its sum per neighbour
// (bound by the building of the short lists' candidates: hash reads and integer work)
template <int W, int MINB>
__global__ void __launch_bounds__(MRQ_MAXNW * 32, MINB) k_frows(const WalkSet ws, const WalkScratch sc, int lbytes, int cap) {
    extern __shared__ __align__(16) unsigned char smem_dyn[];
    const int lane = threadIdx.x & 31;
    unsigned char* const mine = smem_dyn + (size_t)(threadIdx.x >> 5) * lbytes;
    SysDev& S = *reinterpret_cast<SysDev*>(mine);
    FoisOuter& o = *reinterpret_cast<FoisOuter*>(mine + (sizeof(SysDev) + 15) / 16 * 16);
    double* const cphi = reinterpret_cast<double*>(mine + (sizeof(SysDev) + 15) / 16 * 16 + (sizeof(FoisOuter) + 15) / 16 * 16);
    unsigned* const ccode = reinterpret_cast<unsigned*>(cphi + cap);
    const int ng = min(sc.fwave, sc.ctl[CTL_GF] - sc.fwave0);
    if (ng <= 0) return;
    int cur = -1;
    const long long ntask = (long long)ng * sc.ctl[CTL_FG];
    NoCtr ctr;
    for (;;) {
        const int id = next_task(sc.ctl + CTL_FGTASK, lane);
        if (id >= ntask) break;
        const int g = id % ng, k = id / ng;
        const int2 of = sc.fg_of[g];
        if (k >= of.y) continue;
        const FGroup f = sc.fg[of.x + k];
        const GroupMeta& meta = sc.meta[f.det];
        __syncwarp();
        if (meta.sys != cur) {
            copy_sys(&S, ws.systems + meta.sys, lane, 32);
            cur = meta.sys;
            __syncwarp();
        }
        if (lane == 0) {
            unsigned long long n[2][W];
#pragma unroll
            for (int sg = 0; sg < 2; sg++)
#pragma unroll
                for (int w = 0; w < W; w++) n[sg][w] = meta.d[sg][w];
            fois_outer<W>(S, n, o);
        }
        __syncwarp();
        double* const row = sc.frows + f.off;
        if (f.c == 0 && f.v == 0) {                       // a CAS determinant: the group holds one neighbour
            if (lane == 0) row[0] = __ldg(S.c) * hash_lookup(S, hash_key(S, (unsigned)f.ao, (unsigned)(f.ao >> 32)));
            continue;
        }
        int n1;
        const int count = row_list<W>(S, f.ao, f.c, f.v, f.scn, f.sv, cphi, ccode, n1, lane, ctr);
        const int nvc = free_count(f.bv, f.sbv, o.fv[0], o.fv[1]);
        const int h0 = o.hs[0], h1 = o.hs[1], p0 = o.ps[0], p1 = o.ps[1];
        const int yc = f.bc == 1 ? (f.ys ? h1 : h0) : -1, xv = f.av == 1 ? (f.xs ? p1 : p0) : -1;
        for (int qb = 0; qb < f.nq; qb += 32) {
            const int nr = min(32, f.nq - qb), fl = split_of(nr), lf = __ffs(fl) - 1;
            const int qi = lane >> lf, part = lane & (fl - 1);
            const int q = f.q0 + qb + min(qi, nr - 1), ic = q / nvc;
            int x0 = 0, x1 = 0, y0 = 0, y1 = 0, H0 = 0, H1 = 0, P0 = 0, P1 = 0, i = 0, j = 0, par;
            free_decode(S, f.ac, f.sac, o.fc, o.ct, 0, ic, x0, x1);
            free_decode(S, f.bv, f.sbv, o.fv, o.vt, S.nc + S.na, q - ic * nvc, y0, y1);
            if (o.h >= 1 && f.bc < 2 && yc != h0) put2(h0, i, H0, H1);
            if (o.h == 2 && f.bc < 2 && yc != h1) put2(h1, i, H0, H1);
            if (f.ac >= 1) put2(x0, i, H0, H1);
            if (f.ac == 2) put2(x1, i, H0, H1);
            if (o.p >= 1 && f.av < 2 && xv != p0) put2(p0, j, P0, P1);
            if (o.p == 2 && f.av < 2 && xv != p1) put2(p1, j, P0, P1);
            if (f.bv >= 1) put2(y0, j, P0, P1);
            if (f.bv == 2) put2(y1, j, P0, P1);
            if (f.c == 2 && H0 > H1) { const int t = H0; H0 = H1; H1 = t; }
            if (f.v == 2 && P0 > P1) { const int t = P0; P0 = P1; P1 = t; }
            const double s = row_overlap(S, f.ao, f.c, f.v, H0, H1, P0, P1, cphi, ccode, n1, count, part, fl, par);
            if (qi < nr && part == 0) row[qb + qi] = __ldg(S.c + row_label(S, f.c, f.v, H0, H1, P0, P1)) * neg_if(s, par);
        }
        __syncwarp();
    }
}

// the groups' neighbours: elements times the overlaps of k_frows, and the race
template <int W, int MINB>
__global__ void __launch_bounds__(256, MINB) k_fois(const WalkSet ws, const WalkScratch sc) {
    __shared__ WarpTask tasks[8];
    __shared__ FoisOuter outer[8];
    const int lane = threadIdx.x & 31;
    WarpTask& wt = tasks[threadIdx.x >> 5];
    FoisOuter& o = outer[threadIdx.x >> 5];
    const SysDev& S = wt.sys;
    if (sc.ctl[CTL_GF] <= sc.fwave0) return;
    int cur = -1;
    const int ntg = sc.ctl[CTL_TGF];
    NoCtr ctr;
    for (;;) {
        const int id = next_task(sc.ctl + CTL_FOIS, lane);
        if (id >= ntg * MRQ_FOIS_SLICES) break;
        const int slice = id / ntg;
        const TaskGroup tg = sc.tgf[id - slice * ntg];
        const int g = (int)(sc.nseg - 1 - tg.group) - sc.fwave0;
        if (g < 0 || g >= sc.fwave) continue;
        task_system(wt, ws, tg.sys, cur, lane);
        StepSink sink{wt, sc.best, sc.bound, tg.count, lane, tg.primary != 0, 0.0, 0.0, 0.0};
        if (task_begin<W>(wt, ws, sc, tg, lane)) {
            const unsigned long long(&n)[2][W] = *reinterpret_cast<const unsigned long long(*)[2][W]>(wt.nsh);
            if (lane == 0) fois_outer<W>(S, n, o);
            __syncwarp();
            const unsigned long long AO =
                (unsigned long long)active_bits<W>(S, n[0]) | ((unsigned long long)active_bits<W>(S, n[1]) << 32);
            const double* const gops = sc.gops + (long long)tg.group * sc.gstride;
            const int2 of = sc.fg_of[g];
            for (int k = slice; k < of.y; k += MRQ_FOIS_SLICES) {
                const FGroup f = sc.fg[of.x + k];
                const unsigned long long Xb = AO & ~f.ao, Yb = f.ao & ~AO;
                // the fixed orbitals removed and added
                int rf0 = 0, rf1 = 0, af0 = 0, af1 = 0, nrf = 0, naf = 0;
                if (Xb) put2(act_so(S, __ffsll(Xb) - 1), nrf, rf0, rf1);
                if (Xb & (Xb - 1)) put2(act_so(S, 63 - __clzll(Xb)), nrf, rf0, rf1);
                if (f.av >= 1) put2(f.av == 1 ? o.ps[f.xs] : o.ps[0], nrf, rf0, rf1);
                if (f.av == 2) put2(o.ps[1], nrf, rf0, rf1);
                if (Yb) put2(act_so(S, __ffsll(Yb) - 1), naf, af0, af1);
                if (Yb & (Yb - 1)) put2(act_so(S, 63 - __clzll(Yb)), naf, af0, af1);
                if (f.bc >= 1) put2(f.bc == 1 ? o.hs[f.ys] : o.hs[0], naf, af0, af1);
                if (f.bc == 2) put2(o.hs[1], naf, af0, af1);
                const int nvc = free_count(f.bv, f.sbv, o.fv[0], o.fv[1]);
                const bool one = nrf + f.ac == 1;
                const double* const row = sc.frows + f.off;
                for (int qb = 0; qb < f.nq; qb += 32) {
                    const bool on = qb + lane < f.nq;
                    double t = 0.0;
                    unsigned exc = 0;
                    if (on) {
                        const double psim = __ldcg(row + qb + lane);
                        const int q = f.q0 + qb + lane, ic = q / nvc;
                        int x0 = 0, x1 = 0, y0 = 0, y1 = 0, r0 = rf0, r1 = rf1, a0 = af0, a1 = af1, i = nrf, j = naf;
                        free_decode(S, f.ac, f.sac, o.fc, o.ct, 0, ic, x0, x1);
                        free_decode(S, f.bv, f.sbv, o.fv, o.vt, S.nc + S.na, q - ic * nvc, y0, y1);
                        if (f.ac >= 1) put2(x0, i, r0, r1);
                        if (f.ac == 2) put2(x1, i, r0, r1);
                        if (f.bv >= 1) put2(y0, j, a0, a1);
                        if (f.bv == 2) put2(y1, j, a0, a1);
                        if (one) {
                            r1 = r0;
                            a1 = a0;
                            t = (in_walker_block(S, r0, a0)
                                     ? single_from_walker<W>(S, SglFromWalker{gops, 0, 0, 0, 0, 0}, n, r0, a0, ctr)
                                     : single_elem<W>(S, n, r0, a0, ctr)) * psim;
                        } else {
                            if (r0 > r1) { const int z = r0; r0 = r1; r1 = z; }
                            if (a0 > a1) { const int z = a0; a0 = a1; a1 = z; }
                            t = hb_screen(S, double_elem<W>(S, n, r0, r1, a0, a1, ctr)) * psim;
                        }
                        exc = exc_code(r0, r1, a0, a1);
                    }
                    sink.push(on, t, exc);
                }
            }
            sink.finish();
        }
        task_sums<false>(sc, tg, slice, sink.sA, sink.sT, 0.0, lane);
    }
}

// ---- rows of a wave of CAS determinants

// entries of the row (c core holes, v virtual electrons) of a remnant with d more active alpha electrons
// than a CAS determinant: the groups (sc, sv = sc - d) one after the other
__device__ __forceinline__ int row_len(const SysDev& S, int c, int v, int d) {
    int len = 0;
    for (int sc = 0; sc <= c; sc++) {
        const int sv = sc - d;
        if (sv < 0 || sv > v) continue;
        len += shape_count(S.nc, c, sc) * shape_count(S.nv, v, sv);
    }
    return len;
}

// Rows stay known through a launch's steps (they depend on the loaded system and its coefficients only;
// every launch begins with none): most determinants of a step were there the step before.  A wave that
// may not fit behind the known rows forgets them first.
__global__ void k_rows_begin(const WalkScratch sc) {
    sc.kctl[KNOWN_ROWS] = 0;
    sc.kctl[KNOWN_EPOCH]++;
    *reinterpret_cast<unsigned long long*>(sc.kctl + KNOWN_CUR) = 0ull;
}
__global__ void k_wave_begin(const WalkScratch sc) {
    if (sc.wave0 == 0) *sc.seen = max(*sc.seen, sc.ctl[CTL_GC]);
    const long long ng = min(sc.wave_groups, sc.ctl[CTL_GC] - sc.wave0);
    if (ng <= 0) return;
    sc.ctl[CTL_PAIRS] = sc.ctl[CTL_ROWTASK] = sc.ctl[CTL_BIG] = sc.ctl[CTL_SMALL] = 0;
    unsigned long long* const cur = reinterpret_cast<unsigned long long*>(sc.kctl + KNOWN_CUR);
    if ((long long)*cur + ng * sc.row_worst > sc.wave_groups * sc.row_worst ||
        sc.kctl[KNOWN_ROWS] + ng * sc.nref_max > (long long)sc.wave_groups * sc.nref_max) {
        sc.kctl[KNOWN_ROWS] = 0;
        sc.kctl[KNOWN_EPOCH]++;
        *cur = 0ull;
    }
}

__device__ __forceinline__ unsigned long long row_hash(unsigned long long ao, int key) {
    return mix64(ao + 0x9E3779B97F4A7C15ull * (unsigned)(key + 1));
}

// the row references of every determinant of the wave: remnant and class, and the row where it is known
template <int W>
__global__ void __launch_bounds__(256) k_refs(const WalkSet ws, const WalkScratch sc) {
    const int ng = min(sc.wave_groups, sc.ctl[CTL_GC] - sc.wave0);
    if (ng <= 0) return;
    const unsigned epoch = (unsigned)sc.kctl[KNOWN_EPOCH], known = (unsigned)sc.kctl[KNOWN_ROWS];
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < sc.table_size; k += gridDim.x * blockDim.x) sc.table[k] = -1;
    for (int g = blockIdx.x; g < ng; g += gridDim.x) {
        const GroupMeta& meta = sc.meta[sc.wave0 + g];
        const SysDev& S = ws.systems[meta.sys];
        unsigned long long n[2][W];
#pragma unroll
        for (int sg = 0; sg < 2; sg++)
#pragma unroll
            for (int w = 0; w < W; w++) n[sg][w] = meta.d[sg][w];
        const unsigned ao0 = active_bits<W>(S, n[0]), ao1 = active_bits<W>(S, n[1]);
        const unsigned amask = (S.na >= 32) ? 0xFFFFFFFFu : ((1u << S.na) - 1u);
        const unsigned long long AO = (unsigned long long)ao0 | ((unsigned long long)ao1 << 32);
        const unsigned long long AE = (unsigned long long)(~ao0 & amask) | ((unsigned long long)(~ao1 & amask) << 32);
        const int cntO = __popcll(AO), cntE = __popcll(AE);
        const long long at = (long long)g * sc.nref_max;
        for (int q = threadIdx.x; q < sc.nref_max; q += blockDim.x) {
            unsigned char cls = MRQ_NOROW;
            if (q < S.ref_off[8]) {
                int k = 0;
                while (k < 7 && q >= S.ref_off[k + 1]) k++;
                const int ka = k / 3, kb = k % 3, two = ka + kb == 1;       // (0,1) and (1,0) pairs own two rows
                const int loc = q - S.ref_off[k], pair = two ? loc >> 1 : loc;
                const int r = (ka + kb == 0 || (two && !(loc & 1))) ? 1 : 2;
                const int nYa = nsub(cntE, kb), xa = pair / nYa, ya = pair - xa * nYa;
                const unsigned long long Xb = subset_bits(S.colex, AO, cntO, ka, xa);
                const unsigned long long Yb = subset_bits(S.colex, AE, cntE, kb, ya);
                const int d = __popcll(Yb & 0xFFFFFFFFull) - __popcll(Xb & 0xFFFFFFFFull);
                const int c = r - ka, v = r - kb;
                const unsigned long long ao = (AO & ~Xb) | Yb;
                sc.ref_ao[at + q] = ao;
                if (row_len(S, c, v, d) > 0) {
                    cls = (unsigned char)(3 * c + v);
                    const int key = 9 * meta.sys + cls;
                    int h = (int)(row_hash(ao, key) & (unsigned)(sc.ktab_size - 1));
                    for (int probe = 0; probe < sc.ktab_size; probe++) {
                        const unsigned long long e = sc.ktab[h];
                        if ((unsigned)(e >> 32) != epoch) break;
                        const unsigned id = (unsigned)e;
                        if (id < known && sc.k_ao[id] == ao && sc.k_key[id] == key) {
                            cls |= MRQ_KNOWN;
                            sc.ref_rep[at + q] = (int)(at + q);
                            sc.row_off[at + q] = sc.k_off[id];
                            break;
                        }
                        h = (h + 1) & (sc.ktab_size - 1);
                    }
                }
            }
            sc.ref_cls[at + q] = cls;
        }
    }
}

// Distinct new rows: every reference whose row is not known finds or becomes the owner of its (system,
// class, remnant) in an open-addressing table with at least twice as many entries as references; owners
// get a place in the row buffer (which holds the worst case of a wave, every row distinct) and enter the
// table of known rows, which k_refs reads in later waves and steps.
__global__ void __launch_bounds__(256) k_insert(const WalkSet ws, const WalkScratch sc) {
    const int ng = min(sc.wave_groups, sc.ctl[CTL_GC] - sc.wave0);
    if (ng <= 0) return;
    const int total = ng * sc.nref_max, lane = threadIdx.x & 31;
    for (int base = (blockIdx.x * blockDim.x + threadIdx.x) & ~31; base < total; base += gridDim.x * blockDim.x) {
        const int i = base + lane;
        bool owner = false;
        int len = 0;
        int key = 0;
        unsigned long long ao = 0;
        if (i < total && !(sc.ref_cls[i] & MRQ_KNOWN)) {              // (MRQ_NOROW has that bit too)
            const int cls = sc.ref_cls[i], sys = sc.meta[sc.wave0 + i / sc.nref_max].sys;
            key = 9 * sys + cls;
            ao = sc.ref_ao[i];
            int k = (int)(row_hash(ao, key) & (unsigned)(sc.table_size - 1));
            for (int probe = 0; probe < sc.table_size; probe++) {
                const int prev = atomicCAS(sc.table + k, -1, i);
                if (prev < 0) {
                    owner = true;
                    sc.ref_rep[i] = i;
                    break;
                }
                if (sc.ref_ao[prev] == ao && sc.ref_cls[prev] == cls && sc.meta[sc.wave0 + prev / sc.nref_max].sys == sys) {
                    sc.ref_rep[i] = prev;
                    break;
                }
                k = (k + 1) & (sc.table_size - 1);
            }
            if (owner) {
                const SysDev& S = ws.systems[sys];
                const int c = cls / 3, v = cls - 3 * c;
                len = row_len(S, c, v, __popcll(ao & 0xFFFFFFFFull) - (S.nalpha - S.nc));
                len = (len + 3) & ~3;                    // rows start on 32-byte sectors
            }
        }
        // one atomic per warp for the places in the buffer and in the task list
        int x = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        const unsigned big = __ballot_sync(0xffffffffu, owner && len > MRQ_BIG_ROW);
        const unsigned small = __ballot_sync(0xffffffffu, owner && len <= MRQ_BIG_ROW);
        const int pieces = owner && len > MRQ_BIG_ROW ? (len + MRQ_BIG_ROW - 1) / MRQ_BIG_ROW : 0;
        int y = pieces;
        if (big) {
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int z = __shfl_up_sync(0xffffffffu, y, o);
                if (lane >= o) y += z;
            }
        }
        unsigned long long cur = 0;
        int nb = 0, ns = 0, nk = 0;
        if (lane == 31 && x > 0) cur = atomicAdd(reinterpret_cast<unsigned long long*>(sc.kctl + KNOWN_CUR), (unsigned long long)x);
        if (lane == 0 && (big | small)) nk = atomicAdd(sc.kctl + KNOWN_ROWS, __popc(big | small));
        if (lane == 31 && big) nb = atomicAdd(sc.ctl + CTL_BIG, y);
        if (lane == 0 && small) ns = atomicAdd(sc.ctl + CTL_SMALL, __popc(small));
        cur = __shfl_sync(0xffffffffu, cur, 31);
        nb = __shfl_sync(0xffffffffu, nb, 31) + y - pieces;
        ns = __shfl_sync(0xffffffffu, ns, 0);
        nk = __shfl_sync(0xffffffffu, nk, 0);
        if (owner) {
            const long long off = (long long)cur + x - len;
            sc.row_off[i] = off;
            const unsigned lt = (1u << lane) - 1u;
            const int id = nk + __popc((big | small) & lt);
            sc.k_ao[id] = ao;
            sc.k_key[id] = key;
            sc.k_off[id] = off;
            const unsigned long long mine = ((unsigned long long)(unsigned)sc.kctl[KNOWN_EPOCH] << 32) | (unsigned)id;
            int h = (int)(row_hash(ao, key) & (unsigned)(sc.ktab_size - 1));
            for (int probe = 0; probe < sc.ktab_size;) {
                const unsigned long long e = *reinterpret_cast<volatile unsigned long long*>(sc.ktab + h);
                if ((e >> 32) != (mine >> 32) && atomicCAS(sc.ktab + h, e, mine) == e) break;
                if ((e >> 32) == (mine >> 32)) {
                    h = (h + 1) & (sc.ktab_size - 1);
                    probe++;
                }
            }
            for (int k2 = 0; k2 < pieces; k2++) sc.ulist[nb + k2] = make_int2(i, k2);
            if (pieces == 0) sc.ulist[sc.ulist_size - 1 - (ns + __popc(small & lt))] = make_int2(i, 0);
        }
    }
}

// The distinct rows, a warp task each (long ones in pieces).  Entry q of a group (core choice slow, virtual choice fast)
// holds c_l O(m) (-1)^(core-hole positions of m): the sign that H_nm of the same neighbour carries too,
// so k_pairs multiplies the two as they are.
// Bound by FP64 (2 FMA per clock and SM): one read and one FMA per candidate.
template <int W, int MINB>
__global__ void __launch_bounds__(MRQ_MAXNW * 32, MINB) k_rows(const WalkSet ws, const WalkScratch sc, int lbytes, int cap) {
    extern __shared__ __align__(16) unsigned char smem_dyn[];
    const int lane = threadIdx.x & 31;
    unsigned char* const mine = smem_dyn + (size_t)(threadIdx.x >> 5) * lbytes;
    SysDev& S = *reinterpret_cast<SysDev*>(mine);
    double* const cphi = reinterpret_cast<double*>(mine + (sizeof(SysDev) + 15) / 16 * 16);
    unsigned* const ccode = reinterpret_cast<unsigned*>(cphi + cap);
    if (sc.ctl[CTL_GC] <= sc.wave0) return;
    int cur = -1;
    const int nbig = sc.ctl[CTL_BIG], ntask = nbig + sc.ctl[CTL_SMALL];
    NoCtr ctr;
    for (;;) {
        const int id = next_task(sc.ctl + CTL_ROWTASK, lane);
        if (id >= ntask) break;
        const int2 task = id < nbig ? sc.ulist[id] : sc.ulist[sc.ulist_size - 1 - (id - nbig)];
        const int i = task.x, lo = task.y * MRQ_BIG_ROW, hi = lo + MRQ_BIG_ROW;      // entries of the row
        const int sys = sc.meta[sc.wave0 + i / sc.nref_max].sys;
        __syncwarp();
        if (sys != cur) {
            copy_sys(&S, ws.systems + sys, lane, 32);
            cur = sys;
            __syncwarp();
        }
        const unsigned long long AO = sc.ref_ao[i];
        const int c = sc.ref_cls[i] / 3, v = sc.ref_cls[i] - 3 * c;
        const int d = __popcll(AO & 0xFFFFFFFFull) - (S.nalpha - S.nc);
        double* row = sc.rows + sc.row_off[i];
        int base = 0;
        for (int scn = 0; scn <= c; scn++) {
            const int sv = scn - d;
            if (sv < 0 || sv > v) continue;
            const int nvc = shape_count(S.nv, v, sv), ni = shape_count(S.nc, c, scn) * nvc;
            const int q0 = max(lo, base) - base, q1 = min(hi, base + ni) - base;
            base += ni;
            if (q0 >= q1) {
                row += ni;
                continue;
            }
            int n1;
            const int count = row_list<W>(S, AO, c, v, scn, sv, cphi, ccode, n1, lane, ctr);
            const unsigned long long mvc = ~0ull / (unsigned long long)nvc + 1ull;     // q / nvc by its high product
            for (int qb = q0; qb < q1; qb += 32) {
                const int nr = min(32, q1 - qb), f = split_of(nr), lf = __ffs(f) - 1;
                const int qi = lane >> lf, part = lane & (f - 1);
                const int q = qb + min(qi, nr - 1);
                const int ic = nvc == 1 ? q : (int)__umul64hi((unsigned long long)q, mvc);
                int xc[2] = {0, 0}, yv[2] = {0, 0}, par;
                shape_decode(S, S.nc, c, scn, 0, ic, xc, S.mag_c);
                shape_decode(S, S.nv, v, sv, S.nc + S.na, q - ic * nvc, yv, S.mag_v);
                const double s = row_overlap(S, AO, c, v, xc[0], xc[1], yv[0], yv[1], cphi, ccode, n1, count, part, f, par);
                if (qi < nr && part == 0) row[q] = __ldg(S.c + row_label(S, c, v, xc[0], xc[1], yv[0], yv[1])) * s;
            }
            __syncwarp();
            row += ni;
        }
    }
}

// The neighbours of the (X_a, Y_a) pairs of CAS determinants.  A group's neighbour is (core choice,
// virtual choice); its element lies at an affine place of the physicists' table (or of the walker's
// single-excitation operator, r = 1), its overlap times c_l at its place of the group's row, and its
// excitation code is affine too, so a neighbour costs two reads, one product and the two sums.  The
// sign of H_nm (-1)^(core-hole positions) is the same for the whole group.  (No active electron
// moved and r = 2: the only reference determinant reached is the walker's, t = c_l H_nm^2 phi_0(n).)
template <int W, int MINB>
__global__ void __launch_bounds__(256, MINB) k_pairs(const WalkSet ws, const WalkScratch sc) {
    __shared__ WarpTask tasks[8];
    const int lane = threadIdx.x & 31;
    WarpTask& wt = tasks[threadIdx.x >> 5];
    const SysDev& S = wt.sys;
    if (sc.ctl[CTL_GC] <= sc.wave0) return;
    int cur = -1;
    const int ntg = sc.ctl[CTL_TGC];
    for (;;) {
        const int id = next_task(sc.ctl + CTL_PAIRS, lane);
        if (id >= (long long)ntg * sc.ns_max) break;
        const int slice = id / ntg;
        const TaskGroup tg = sc.tgc[id - slice * ntg];
        if (tg.group < sc.wave0 || tg.group >= sc.wave0 + sc.wave_groups) continue;
        task_system(wt, ws, tg.sys, cur, lane);
        if (slice >= S.nslice) continue;
        StepSink sink{wt, sc.best, sc.bound, tg.count, lane, tg.primary != 0, 0.0, 0.0, 0.0};
        if (task_begin<W>(wt, ws, sc, tg, lane)) {
            const unsigned long long(&n)[2][W] = *reinterpret_cast<const unsigned long long(*)[2][W]>(wt.nsh);
            const unsigned ao0 = active_bits<W>(S, n[0]), ao1 = active_bits<W>(S, n[1]);
            const unsigned amask = (S.na >= 32) ? 0xFFFFFFFFu : ((1u << S.na) - 1u);
            const unsigned long long AO = (unsigned long long)ao0 | ((unsigned long long)ao1 << 32);
            const unsigned long long AE = (unsigned long long)(~ao0 & amask) | ((unsigned long long)(~ao1 & amask) << 32);
            const int cntO = __popcll(AO), cntE = __popcll(AE), nc = S.nc, nv = S.nv, voff = S.nc + S.na;
            const long long refs = (long long)(tg.group - sc.wave0) * sc.nref_max;
            const double phin = sc.meta[tg.group].phi;
            for (int u = S.cas_units + slice; u < S.unit_off[8]; u += S.nslice) {
                int k = 0;
                while (k < 7 && u >= S.unit_off[k + 1]) k++;
                const int ka = k / 3, kb = k % 3, nch = S.nch[k];
                const int loc = u - S.unit_off[k], pair = loc / nch, ch = loc - pair * nch;
                const int nYa = nsub(cntE, kb), xa = pair / nYa, ya = pair - xa * nYa;
                const unsigned long long Xb = subset_bits(S.colex, AO, cntO, ka, xa);
                const unsigned long long Yb = subset_bits(S.colex, AE, cntE, kb, ya);
                const int d = __popcll(Yb & 0xFFFFFFFFull) - __popcll(Xb & 0xFFFFFFFFull);
                const int tot = pair_total(S, ka, kb, d);
                const int lo = (int)((long long)ch * tot / nch), hi = (int)((long long)(ch + 1) * tot / nch);
                const int xa0 = Xb ? act_so(S, __ffsll(Xb) - 1) : 0, xa1 = ka == 2 ? act_so(S, 63 - __clzll(Xb)) : 0;
                const int ya0 = Yb ? act_so(S, __ffsll(Yb) - 1) : 0, ya1 = kb == 2 ? act_so(S, 63 - __clzll(Yb)) : 0;
                int base = 0;
                int ref = S.ref_off[k] + (ka + kb == 1 ? 2 * pair : pair);
                for (int r = max(1, max(ka, kb)); r <= 2; r++) {
                    const int c = r - ka, v = r - kb;
                    if (c == 0 && v == 0) continue;
                    const bool self = c == 2 && v == 2;
                    const double* row = sc.rows;
                    if (!self) {
                        if (sc.ref_cls[refs + ref] != MRQ_NOROW) row += sc.row_off[sc.ref_rep[refs + ref]];
                        ref++;
                    }
                    for (int scn = 0; scn <= c; scn++) {
                        const int sv = scn - d;
                        if (sv < 0 || sv > v) continue;
                        const int nvc = shape_count(nv, v, sv), ni = shape_count(nc, c, scn) * nvc;
                        const int q0 = max(lo, base) - base, q1 = min(hi, base + ni) - base;
                        if (ni > 0 && q0 < q1) {
                            // the group's first neighbour, and how element and code change from it
                            int xc0, xc1, yv0, yv1, rm0, rm1, ad0, ad1;
                            unsigned long long m[2][W];
                            group_neighbour<W>(S, n, nc, nv, voff, c, scn, v, sv, 0, 0, ka, xa0, xa1, kb, ya0, ya1, r, xc0, xc1,
                                               yv0, yv1, rm0, rm1, ad0, ad1, m);
                            const int cp0 = xc0 - (xc0 >= S.n ? S.n : 0), cp1 = xc1 - (xc1 >= S.n ? S.n : 0);
                            const int vp0 = yv0 - (yv0 >= S.n ? S.n : 0) - voff, vp1 = yv1 - (yv1 >= S.n ? S.n : 0) - voff;
                            const double* H;
                            unsigned cs0 = 0, cs1 = 0, vs0 = 0, vs1 = 0, ce0 = 0, ce1 = 0, ve0 = 0, ve1 = 0, hb, eb;
                            int odd = (c >= 1 ? cp0 : 0) + (c == 2 ? cp1 : 0);
                            const unsigned sv1 = (unsigned)S.nav, sq = sv1 * sv1, sp = sq * (unsigned)S.nca;
                            if (r == 1) {
                                const int sx = rm0 >= S.n, px = rm0 - sx * S.n, py = ad0 - sx * S.n;
                                H = sc.gops + (long long)tg.group * sc.gstride;
                                hb = (unsigned)((sx * S.nca + px) * S.nav + (py - nc));
                                odd += popc_sel<W>(n, sx, min(px, py), max(px, py));
                                eb = exc_code(rm0, rm0, ad0, ad0);
                                cs0 = sv1;
                                vs0 = 1u;
                                ce0 = 0x101u;
                                ve0 = 0x1010000u;
                            } else {
                                const int s1 = rm0 >= S.n, s2 = rm1 >= S.n;
                                int p1 = rm0 - s1 * S.n, p2 = rm1 - s2 * S.n;
                                int a1 = ad0 - (ad0 >= S.n) * S.n, a2 = ad1 - (ad1 >= S.n) * S.n;
                                int o = popc_sel<W>(n, s1, min(p1, a1), max(p1, a1));
                                if (s1 == s2) {
                                    unsigned long long t[W];
#pragma unroll
                                    for (int w = 0; w < W; w++) t[w] = s1 ? n[1][w] : n[0][w];
                                    flip<W>(t, p1);
                                    flip<W>(t, a1);
                                    o += popc_between<W>(t, min(p2, a2), max(p2, a2));
                                } else {
                                    o += popc_sel<W>(n, s2, min(p2, a2), max(p2, a2));
                                }
                                odd += o;
                                H = S.tab;
                                eb = exc_code(rm0, rm1, ad0, ad1);
                                const bool cfirst = c == 2 || (c == 1 && rm0 == xc0), vfirst = v == 2 || (v == 1 && ad0 == yv0);
                                cs0 = cfirst ? sp : sq;
                                cs1 = sq;
                                ce0 = cfirst ? 0x1u : 0x100u;
                                ce1 = 0x100u;
                                vs0 = vfirst ? sv1 : 1u;
                                vs1 = 1u;
                                ve0 = vfirst ? 0x10000u : 0x1000000u;
                                ve1 = 0x1000000u;
                                if (v == 1 && vfirst) {
                                    // <pq|rs> = <qp|sr>: the virtual index last, so that a warp reads consecutive words
                                    int t = p1;
                                    p1 = p2;
                                    p2 = t;
                                    t = a1;
                                    a1 = a2;
                                    a2 = t;
                                    cs0 = cfirst ? sq : sp;
                                    cs1 = sp;                  // (c = 2: the two holes are of opposite spin)
                                    vs0 = 1u;
                                }
                                hb = (s1 == s2 ? S.tab_half : 0u) + (unsigned)p1 * sp + (unsigned)p2 * sq +
                                     (unsigned)(a1 - nc) * sv1 + (unsigned)(a2 - nc);
                            }
                            if (c < 2) cs1 = ce1 = 0u;
                            if (v < 2) vs1 = ve1 = 0u;
                            if (c < 1) cs0 = ce0 = 0u;
                            if (v < 1) vs0 = ve0 = 0u;
                            hb -= (unsigned)cp0 * cs0 + (unsigned)cp1 * cs1 + (unsigned)vp0 * vs0 + (unsigned)vp1 * vs1;
                            eb -= (unsigned)cp0 * ce0 + (unsigned)cp1 * ce1 + (unsigned)vp0 * ve0 + (unsigned)vp1 * ve1;
                            const unsigned long long mvc = ~0ull / (unsigned long long)nvc + 1ull;
                            auto element = [&](int q, double& t, unsigned& exc) {
                                const int ic = nvc == 1 ? q : (int)__umul64hi((unsigned long long)q, mvc), iv = q - ic * nvc;
                                int i0 = ic, i1 = 0, j0 = iv, j1 = 0;
                                if (c == 2) {
                                    if (scn == 1) {
                                        i0 = S.mag_c ? (int)__umul64hi((unsigned long long)ic, S.mag_c) : ic;
                                        i1 = ic - i0 * nc;
                                    } else {
                                        lex_decode_tab(S.colex, ic, nc, i0, i1);
                                    }
                                }
                                if (v == 2) {
                                    if (sv == 1) {
                                        j0 = S.mag_v ? (int)__umul64hi((unsigned long long)iv, S.mag_v) : iv;
                                        j1 = iv - j0 * nv;
                                    } else {
                                        lex_decode_tab(S.colex, iv, nv, j0, j1);
                                    }
                                }
                                const double h = H[hb + (unsigned)i0 * cs0 + (unsigned)i1 * cs1 + (unsigned)j0 * vs0 + (unsigned)j1 * vs1];
                                exc = eb + (unsigned)i0 * ce0 + (unsigned)i1 * ce1 + (unsigned)j0 * ve0 + (unsigned)j1 * ve1;
                                if (self) {
                                    const int h0 = scn == 0 ? nc + i0 : i0, h1 = scn == 2 ? i1 : nc + i1;
                                    const int p0 = sv == 0 ? nv + j0 : j0, p1 = sv == 2 ? j1 : nv + j1;
                                    t = h * (h * phin) * __ldg(S.c + set_rank(2, h0, h1, 2 * nc) * S.nPs + set_rank(2, p0, p1, 2 * nv));
                                } else {
                                    t = neg_if(h * __ldcg(row + q), odd);
                                }
                            };
                            for (int qb = q0; qb < q1; qb += 64) {
                                double t0, t1;
                                unsigned e0, e1;
                                element(min(qb + lane, q1 - 1), t0, e0);
                                element(min(qb + 32 + lane, q1 - 1), t1, e1);
                                if (q1 - qb >= 64) {
                                    sink.take(t0, e0, t1, e1);
                                } else {
                                    sink.push(qb + lane < q1, t0, e0);
                                    if (qb + 32 < q1) sink.push(qb + 32 + lane < q1, t1, e1);
                                }
                            }
                        }
                        base += ni;
                        if (!self) row += ni;
                    }
                }
            }
            sink.finish();
        }
        task_sums<false>(sc, tg, slice, sink.sA, sink.sT, 0.0, lane);
    }
}

// apply the excitation code of the race's winner to n
template <int W>
__device__ __forceinline__ void apply_code(unsigned long long (&m)[2][W], const SysDev& S, unsigned exc) {
    const int r1 = exc & 255u, r2 = (exc >> 8) & 255u, a1 = (exc >> 16) & 255u, a2 = (exc >> 24) & 255u;
    int s = r1 >= S.n;
    flip_reg<W>(m, s, r1 - s * S.n);
    s = a1 >= S.n;
    flip_reg<W>(m, s, a1 - s * S.n);
    if (r2 != r1) {
        s = r2 >= S.n;
        flip_reg<W>(m, s, r2 - s * S.n);
        s = a2 >= S.n;
        flip_reg<W>(m, s, a2 - s * S.n);
    }
}

// The step's end, one warp per task group: the determinant's sums over its slices (in slice order
// within a lane, then a fixed tree), each walker's record (k_accum adds them) and move, and psi_s at
// the new determinant - a function of that determinant alone, so that walkers that meet on it agree
// bit for bit.
template <int W>
__global__ void __launch_bounds__(MRQ_MAXNW * 32) k_move(const WalkSet ws, const WalkScratch sc, int accumulate, int lbytes,
                                                         int cap) {
    extern __shared__ __align__(16) unsigned char smem_dyn[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    double* const cphi = reinterpret_cast<double*>(smem_dyn + (size_t)warp * lbytes);
    unsigned* const ccode = reinterpret_cast<unsigned*>(cphi + cap);
    const int ntc = sc.ctl[CTL_TGC], ntg = ntc + sc.ctl[CTL_TGF];
    for (int g = blockIdx.x * nw + warp; g < ntg; g += gridDim.x * nw) {
        const TaskGroup tg = g < ntc ? sc.tgc[g] : sc.tgf[g - ntc];
        const SysDev& S = ws.systems[tg.sys];
        const GroupMeta meta = sc.meta[tg.group];
        const double inv_psin = meta.inv_psi;
        double A = 0.0, T = 0.0, D = 0.0;
        const double* const part = sc.part + (long long)tg.group * (sc.ns_max + MRQ_ACT_SLICES) * 3;
        const int ns = g < ntc ? S.nslice : MRQ_FOIS_SLICES;
        for (int k = lane; k < ns; k += 32) {
            A += part[3 * k];
            T += part[3 * k + 1];
            D += part[3 * k + 2];
        }
        if (lane < (g < ntc ? MRQ_INT_SLICES : MRQ_ACT_SLICES)) {
            A += part[3 * (sc.ns_max + lane)];
            T += part[3 * (sc.ns_max + lane) + 1];
            D += part[3 * (sc.ns_max + lane) + 2];
        }
        A = warp_sum(A);
        T = warp_sum(T);
        D = warp_sum(D);
        const double rate = fabs(inv_psin) * A;
        unsigned long long m[2][W];
#pragma unroll
        for (int sg = 0; sg < 2; sg++)
#pragma unroll
            for (int w = 0; w < W; w++) m[sg][w] = meta.d[sg][w];
        Walker* wk = nullptr;
        bool moved = false;
        long long lm = 0;
        if (lane < tg.count) {
            const int i = sc.members[tg.first + lane];
            wk = ws.walkers[tg.sys] + i;
            wk->rl = -1;
            const RaceBest b = sc.best[ws.offsets[tg.sys] + i - sc.seg0];
            if (meta.label < 0 || !(rate > 0.0) || b.exc == 0xFFFFFFFFu) {
                atomicOr(S.err, meta.label < 0 ? MRQ_ERR_LABEL : MRQ_ERR_NOMOVE);
            } else {
                moved = true;
                if (accumulate && (long long)wk->step >= S.burn_in) {
                    wk->rl = meta.label;
                    wk->rtype = 3 * meta.h + meta.p;
                    wk->rw = 1.0 / rate;
                    wk->rEL = meta.hnn + inv_psin * T;
                    wk->rnum = meta.label > 0 ? meta.hdnn + inv_psin * D : 0.0;
                }
                apply_code<W>(m, S, b.exc);
                int h, p;
                lm = det_label<W>(S, m, h, p);
            }
        }
        double psi = 0.0;
        if (moved && lm == 0) psi = __ldg(S.c) * hash_lookup(S, hash_key(S, active_bits<W>(S, m[0]), active_bits<W>(S, m[1])));
        unsigned todo = __ballot_sync(0xffffffffu, moved && lm > 0);
        while (todo) {
            const int src = __ffs(todo) - 1;
            todo &= todo - 1;
            unsigned long long x[2][W];
#pragma unroll
            for (int sg = 0; sg < 2; sg++)
#pragma unroll
                for (int w = 0; w < W; w++) x[sg][w] = __shfl_sync(0xffffffffu, m[sg][w], src);
            const double o = reach_back_warp<W>(S, x, cphi, ccode, lane);
            if (lane == src) psi = __ldg(S.c + lm) * o;
        }
        if (moved) {
#pragma unroll
            for (int sg = 0; sg < 2; sg++)
#pragma unroll
                for (int w = 0; w < W; w++) wk->d[sg][w] = m[sg][w];
            wk->psi = psi;
            wk->step++;
        }
    }
}

// Accumulate the last step's walker records (Eq. 12, Eq. 16; weight w = 1/S): one warp per
// (system, group), walkers of the group in id order.  The label-0 (CAS) sums are warp sums in a fixed
// order; other labels are added by their lanes at once, walkers that share a label one after the other
// in lane order - the same result on every run.
__global__ void __launch_bounds__(1024) k_accum(const WalkSet ws) {
    const int sys = blockIdx.x;
    const int g = blockIdx.y * 32 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const SysDev& S = ws.systems[sys];
    if (g >= S.G) return;
    Walker* const wk = ws.walkers[sys];
    const long long nw = ws.offsets[sys + 1] - ws.offsets[sys];
    const long long L = S.nlab;
    double n0 = 0.0, a0 = 0.0, b0 = 0.0, wsum = 0.0, esum = 0.0;
    unsigned count = 0;                       // lane t < MRQ_NTYPES: steps at type t
    const double c0 = S.c[0];
    for (long long base = g; base < nw; base += 32LL * S.G) {
        const long long i = base + (long long)lane * S.G;
        long long l = -1;
        double w = 0.0, EL = 0.0, num = 0.0;
        int type = -1;
        if (i < nw) {
            l = wk[i].rl;
            w = wk[i].rw;
            EL = wk[i].rEL;
            num = wk[i].rnum;
            if (l >= 0) type = wk[i].rtype;
        }
#pragma unroll
        for (int t = 0; t < MRQ_NTYPES; t++) {
            const unsigned m = __ballot_sync(0xffffffffu, type == t);
            if (lane == t) count += __popc(m);
        }
        if (l >= 0) {
            wsum += w;
            esum += w * EL;
        }
        if (l == 0) {
            n0 += w / (c0 * c0);
            a0 += (w * EL) / c0;
            b0 += w / c0;
        }
        unsigned todo = __ballot_sync(0xffffffffu, l > 0);
        const unsigned peers = __match_any_sync(0xffffffffu, l) & todo;
        while (todo) {
            const bool mine = (todo >> lane & 1u) && (peers & todo & ((1u << lane) - 1u)) == 0u;   // first of its label left
            if (mine) {
                const double cl = S.c[l], c2 = cl * cl;
                const long long at = (long long)g * L + l;
                S.accN[at] += w / c2;
                S.accU[at] += (w * num) / c2;
                S.accA[at] += (w * EL) / cl;
                S.accB[at] += w / cl;
            }
            todo &= ~__ballot_sync(0xffffffffu, mine);
            __syncwarp();
        }
    }
    n0 = warp_sum(n0);
    a0 = warp_sum(a0);
    b0 = warp_sum(b0);
    wsum = warp_sum(wsum);
    esum = warp_sum(esum);
    if (lane < MRQ_NTYPES && count) atomicAdd(S.type_steps + lane, (unsigned long long)count);
    if (lane == 0) {
        const long long at = (long long)g * L;
        S.accN[at] += n0;
        S.accA[at] += a0;
        S.accB[at] += b0;
        S.accW[g] += wsum;
        S.accE[g] += esum;
    }
}

// The race alone, for parity: the neighbours (t, excitation) of one determinant against nw walkers' clocks, the
// neighbours in rounds of 64 dealt to `slices` warp tasks per group of MRQ_TGW walkers, as in a walk step.
__global__ void __launch_bounds__(256) k_debug_race(const unsigned* __restrict__ exc, const double* __restrict__ t, long long n,
                                                    double inv_psi, unsigned long long seed, const unsigned* __restrict__ wid,
                                                    const unsigned* __restrict__ step, int nw, int slices, RaceBest* best,
                                                    unsigned* bound) {
    __shared__ WarpTask tasks[8];
    const int lane = threadIdx.x & 31;
    WarpTask& wt = tasks[threadIdx.x >> 5];
    const long long id = (long long)blockIdx.x * 8 + (threadIdx.x >> 5);
    const long long first = id / slices * MRQ_TGW;
    if (first >= nw) return;
    const int count = (int)min((long long)MRQ_TGW, nw - first);
    if (lane == 0) {
        wt.sys.seed = seed;
        wt.inv_psin = inv_psi;
        wt.inv_f = race_inv(inv_psi);
        wt.qn = 0;
    }
    __syncwarp();
    if (lane < count) race_walker(wt, lane, step[first + lane], wid[first + lane], (int)(first + lane), bound, wt.inv_f);
    __syncwarp();
    StepSink sink{wt, best, bound, count, lane, false, 0.0, 0.0, 0.0};
    for (long long q = 64 * (id % slices); q < n; q += 64LL * slices) {
        const long long q0 = q + lane, q1 = q0 + 32;
        const double t0 = q0 < n ? t[q0] : 0.0, t1 = q1 < n ? t[q1] : 0.0;
        const unsigned e0 = q0 < n ? exc[q0] : 0u, e1 = q1 < n ? exc[q1] : 0u;
        if (q + 64 <= n) {
            sink.take(t0, e0, t1, e1);
        } else {
            sink.push(q0 < n, t0, e0);
            sink.push(q1 < n, t1, e1);
        }
    }
    sink.finish();
}

// ------------------------------------------------------------------ debug evaluation (parity)

// shared state of a debug block (dynamic shared memory: this, the operator, one list per warp)
struct DebugSh {
    SysDev sys;
    WarpLists lists;
    double wsum[3][MRQ_VW];
    unsigned long long ctr[4];      // gathers, probes, candidates, terms
    double hnn, hdnn;
    CasWalker cw;
    unsigned long long nsh[4];
};

__host__ __device__ __forceinline__ size_t debug_smem_bytes(int nw, int cap, int gstride) {
    return (sizeof(DebugSh) + 15) / 16 * 16 + ((size_t)gstride * sizeof(double) + 15) / 16 * 16 +
           (size_t)nw * cand_list_bytes(cap);
}
__host__ __device__ __forceinline__ size_t frows_warp_bytes(int cap) {
    return (sizeof(SysDev) + 15) / 16 * 16 + (sizeof(FoisOuter) + 15) / 16 * 16 + cand_list_bytes(cap);
}
__host__ __device__ __forceinline__ size_t rows_warp_bytes(int cap) {
    return (sizeof(SysDev) + 15) / 16 * 16 + cand_list_bytes(cap);
}

// Local quantities of arbitrary determinants: one block per determinant, every neighbour with the lists of its own
// group or lane (cas_pair_unit, fois_unit).  The walk shares rows and groups between determinants instead; the two
// meet in the tests, which hold the walk's per-walker sums against this evaluation and both against the oracle.
template <int W>
__global__ void __launch_bounds__(MRQ_MAXNW * 32, 2) k_debug2(const SysDev* __restrict__ sys,
                                                              const unsigned long long* __restrict__ dets, long long ndet,
                                                              mrq_local* __restrict__ out, long long max_nb,
                                                              mrq_neighbour* __restrict__ nb, long long* nb_prefix,
                                                              int prefix_stride) {
    extern __shared__ __align__(16) unsigned char smem_dyn[];
    DebugSh& cs = *reinterpret_cast<DebugSh*>(smem_dyn);
    const long long i = blockIdx.x;
    if (i >= ndet) return;
    const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5, nw = blockDim.x >> 5;
    copy_sys(&cs.sys, sys, threadIdx.x, blockDim.x);
    if (threadIdx.x < 4) cs.ctr[threadIdx.x] = 0;
    __syncthreads();
    const SysDev& S = cs.sys;
    unsigned long long n[2][W];
#pragma unroll
    for (int w = 0; w < W; w++) {
        n[0][w] = dets[i * 2 * W + w];
        n[1][w] = dets[i * 2 * W + W + w];
    }
    int h, p;
    const long long ln = det_label<W>(S, n, h, p);
    mrq_local r;
    memset(&r, 0, sizeof r);
    r.label = ln;
    r.type = 3 * h + p;
    if (ln < 0) {
        if (threadIdx.x == 0) out[i] = r;
        return;
    }
    double psin;
    NoCtr nc0;
    if (ln == 0) psin = __ldg(S.c) * hash_lookup(S, hash_key(S, active_bits<W>(S, n[0]), active_bits<W>(S, n[1])), nc0);
    else psin = __ldg(S.c + ln) * reach_back<W>(S, n, nc0);
    Ctr ctr;
    mrq_neighbour* const rec = nb ? nb + i * max_nb : nullptr;
    long long* const prefix = nb_prefix ? nb_prefix + i * (long long)prefix_stride : nullptr;
    unsigned char* const lists = smem_dyn + (sizeof(DebugSh) + 15) / 16 * 16;
    double* const gops = reinterpret_cast<double*>(lists);
    double* const cphi = reinterpret_cast<double*>(lists + ((size_t)S.gstride * sizeof(double) + 15) / 16 * 16 +
                                                   (size_t)wi * cand_list_bytes(S.cand_cap));
    unsigned* const ccode = reinterpret_cast<unsigned*>(cphi + S.cand_cap);
    const double c0 = __ldg(S.c), inv_psin = psin != 0.0 ? 1.0 / psin : 0.0;
    const bool cas = ln == 0 && psin != 0.0;
    if (wi == 0) {
        double hnn, hdnn;
        build_lists<W>(S, n, cs.lists, h, p, lane);
        diagonals<W>(S, cs.lists, n, lane, hnn, hdnn);
        if (lane == 0) {
            cs.hnn = hnn;
            cs.hdnn = hdnn;
            if (cas) cs.cw = cas_constants<W>(S, n, psin / c0);
#pragma unroll
            for (int sg = 0; sg < 2; sg++)
#pragma unroll
                for (int w = 0; w < W; w++) cs.nsh[sg * W + w] = n[sg][w];
        }
    }
    if (psin != 0.0) walker_operator<W>(S, n, cas, gops, ctr);
    const unsigned long long(&nsh)[2][W] = *reinterpret_cast<const unsigned long long(*)[2][W]>(cs.nsh);
    __syncthreads();
    const int total_fois = cas ? 0 : cs.lists.bstart[cs.lists.nb];
    const int units = cas ? S.unit_off[8] : (total_fois + MRQ_FOIS_CH - 1) / MRQ_FOIS_CH;
    if (rec != nullptr && cas) {              // neighbour offsets of the units
        for (int u = threadIdx.x; u < units; u += blockDim.x) prefix[u] = cas_unit_count(S, cs.cw, u);
        __syncthreads();
        if (threadIdx.x == 0) {
            long long run = 0;
            for (int u = 0; u < units; u++) {
                const long long c = prefix[u];
                prefix[u] = run;
                run += c;
            }
        }
        __syncthreads();
    }
    const unsigned long long self_key =
        ln == 0 ? hash_key(S, active_bits<W>(S, n[0]), active_bits<W>(S, n[1])) : MRQ_EMPTY_KEY;
    const double phi_self = ln == 0 ? psin / c0 : 0.0;
    for (int vw = wi; vw < MRQ_VW; vw += nw) {
        DebugSink sink{rec, 0, max_nb, inv_psin, 0.0, 0.0, 0.0};
        for (int u = vw; u < units; u += MRQ_VW) {
            if (cas) {
                sink.nbase = rec != nullptr ? prefix[u] : 0;
                if (u < S.cas_units) cas_internal_unit<W>(S, cs.cw, nsh, u, lane, sink, ctr);
                else cas_pair_unit<W>(S, cs.cw, gops, cphi, ccode, nsh, u, lane, sink, ctr);
            } else {
                fois_unit<W>(S, cs.lists, psin != 0.0 ? gops : nullptr, nsh, ln, c0, self_key, phi_self, u * MRQ_FOIS_CH,
                             min(total_fois, (u + 1) * MRQ_FOIS_CH), lane, sink, ctr);
            }
        }
        const double sA = warp_sum(sink.sA), sT = warp_sum(sink.sT), sD = warp_sum(sink.sD);
        if (lane == 0) {
            cs.wsum[0][vw] = sA;
            cs.wsum[1][vw] = sT;
            cs.wsum[2][vw] = sD;
        }
    }
    {
        unsigned long long v[4] = {ctr.gathers, ctr.probes, ctr.cands, ctr.terms};
#pragma unroll
        for (int k = 0; k < 4; k++) {
            unsigned long long x = v[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
            if (lane == 0) atomicAdd(&cs.ctr[k], x);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double A = 0.0, T = 0.0, D = 0.0;
        for (int k = 0; k < MRQ_VW; k++) {
            A += cs.wsum[0][k];
            T += cs.wsum[1][k];
            D += cs.wsum[2][k];
        }
        r.n_gathers = (long long)cs.ctr[0];
        r.n_probes = (long long)cs.ctr[1];
        r.n_candidates = (long long)cs.ctr[2];
        r.n_terms = (long long)cs.ctr[3];
        r.S = fabs(inv_psin) * A;
        r.e_local = cs.hnn + inv_psin * T;
        r.num = ln > 0 ? cs.hdnn + inv_psin * D : 0.0;
        r.h_nn = cs.hnn;
        r.hd_nn = cs.hdnn;
        r.psi = psin;
        r.n_neighbours = cas ? (long long)S.cas_nb_total : (long long)total_fois;
        out[i] = r;
    }
}
