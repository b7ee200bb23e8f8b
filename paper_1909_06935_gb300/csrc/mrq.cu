// mrq.cu - GB300 (sm_103a) kernels and host runtime of the stochastic SC-NEVPT2(s) /
// SC-MRCI(s) local-estimator path (arXiv:1909.06935), behind the C ABI of include/mrq.h.
//
// Hot path (mrq_walk.cuh), per step and distinct determinant of the walkers:
//   classify it (label, Sec. II A) -> enumerate every single and double excitation that stays in
//   CAS u FOIS -> per lane: <n|H|m> by Slater-Condon, psi_s(m) by a hash probe (m in the CAS) or
//   reach-back O(m) = <m|H|phi0> (Eq. 6-7, Sec. II D) -> rates Gamma_nm = |H_nm psi_s(m)/psi_s(n)|,
//   E_L (Eq. 5), the H_D numerator (Eq. 16) -> fixed-order sums -> accumulate with weight 1/S ->
//   every walker moves by the first-reaction (competing exponential clocks) form of Gillespie's
//   algorithm.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <chrono>
#include <cstring>
#include <mutex>
#include <thread>
#include <vector>

#include "../../include/mrq.h"
#include "mrq_device.cuh"
#include "mrq_internal.h"

// ============================================================================ per-warp state

struct Walker {
    unsigned long long d[2][2];   // [spin][word]
    double psi;                   // psi_s of the current determinant
    unsigned step;                // steps taken by this walker so far
    unsigned wid;                 // walker id (Philox counter word)
    int sys;                      // index into the system table
    int group;                    // accumulator group
    // the last step's contribution, written by the walk and added by k_accum
    long long rl;                 // label of the determinant the step was taken at (-1: nothing to add)
    double rw, rEL, rnum;         // residence weight 1/S, E_L, H_D numerator
    int rtype;                    // 3h + p
    int rpad;
};

static_assert(sizeof(SysDev) % sizeof(int) == 0, "SysDev is copied word by word");

struct WarpLists {
    unsigned char ol[2][MRQ_MAXN];   // occupied orbitals per spin, ascending (core|active|virtual)
    unsigned char el[2][MRQ_MAXN];   // empty orbitals per spin
    short os[2][4], es[2][4];        // class starts: [spin][class], [3] = count
    int bstart[MRQ_MAXB + 1];        // block prefix offsets
    unsigned bdesc[MRQ_MAXB];        // block descriptors
    int nb;
};

// pair tables for same-spin doubles: (X1, X2) with X1 <= X2
__constant__ unsigned char c_pair_a[6] = {0, 0, 0, 1, 1, 2};
__constant__ unsigned char c_pair_b[6] = {0, 1, 2, 1, 2, 2};

__device__ __forceinline__ int pairs_of(int k1, int k2, bool same) { return same ? k1 * (k1 - 1) / 2 : k1 * k2; }

// enumeration speed of an orbital class: active slowest (0), core (1), virtual fastest (2)
__device__ __forceinline__ int cls_pri(int c) { return c == 1 ? 0 : (c == 0 ? 1 : 2); }

// pair index -> (i < j), ordered by j then i (used for the occupied-pair diagonal sums)
__device__ __forceinline__ void tri_decode(int op, int& i, int& j) {
    int jj = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)op)) * 0.5f);
    while (jj * (jj - 1) / 2 > op) jj--;
    while ((jj + 1) * jj / 2 <= op) jj++;
    j = jj;
    i = op - jj * (jj - 1) / 2;
}

// Build occupied/empty lists (class-partitioned) and the valid excitation blocks of det d.
template <int W>
__device__ void build_lists(const SysDev& S, const unsigned long long (&d)[2][W], WarpLists& sh, int h, int p,
                            int lane) {
    const int n = S.n;
    for (int sg = 0; sg < 2; sg++) {
        int no = 0, ne = 0;
        for (int base = 0; base < n; base += 32) {
            int q = base + lane;
            bool valid = q < n;
            bool o = valid && bit_of<W>(d[sg], q);
            unsigned bo = __ballot_sync(0xffffffffu, o);
            unsigned be = __ballot_sync(0xffffffffu, valid && !o);
            unsigned lt = (1u << lane) - 1u;
            if (o) sh.ol[sg][no + __popc(bo & lt)] = (unsigned char)q;
            if (valid && !o) sh.el[sg][ne + __popc(be & lt)] = (unsigned char)q;
            no += __popc(bo);
            ne += __popc(be);
        }
        if (lane == 0) {
            int oc = 0, oa = 0, ov = 0;
#pragma unroll
            for (int w = 0; w < W; w++) {
                oc += __popcll(d[sg][w] & S.mcore[w]);
                oa += __popcll(d[sg][w] & S.mact[w]);
                ov += __popcll(d[sg][w] & S.mvirt[w]);
            }
            sh.os[sg][0] = 0;
            sh.os[sg][1] = oc;
            sh.os[sg][2] = oc + oa;
            sh.os[sg][3] = oc + oa + ov;
            sh.es[sg][0] = 0;
            sh.es[sg][1] = S.nc - oc;
            sh.es[sg][2] = S.nc - oc + S.na - oa;
            sh.es[sg][3] = n - (oc + oa + ov);
        }
    }
    __syncwarp();
    // candidate blocks: 18 singles, 72 same-spin doubles, 81 opposite-spin doubles
    int run = 0, carry = 0;
    for (int base = 0; base < MRQ_MAXB; base += 32) {
        int ci = base + lane;
        int size = 0, kind = 0, sg = 0, X1 = 0, X2 = 0, Y1 = 0, Y2 = 0;
        unsigned order = 0;
        if (ci < MRQ_MAXB) {
            if (ci < 18) {
                kind = 0; sg = ci / 9; X1 = (ci % 9) / 3; Y1 = ci % 3;
                size = (sh.os[sg][X1 + 1] - sh.os[sg][X1]) * (sh.es[sg][Y1 + 1] - sh.es[sg][Y1]);
            } else if (ci < 90) {
                int c = ci - 18;
                kind = 1; sg = c / 36;
                int px = (c % 36) / 6, py = c % 6;
                X1 = c_pair_a[px]; X2 = c_pair_b[px]; Y1 = c_pair_a[py]; Y2 = c_pair_b[py];
                int k1 = sh.os[sg][X1 + 1] - sh.os[sg][X1], k2 = sh.os[sg][X2 + 1] - sh.os[sg][X2];
                int e1 = sh.es[sg][Y1 + 1] - sh.es[sg][Y1], e2 = sh.es[sg][Y2 + 1] - sh.es[sg][Y2];
                size = pairs_of(k1, k2, X1 == X2) * pairs_of(e1, e2, Y1 == Y2);
            } else {
                int c = ci - 90;
                kind = 2; X1 = c / 27; Y1 = (c / 9) % 3; X2 = (c / 3) % 3; Y2 = c % 3;
                size = (sh.os[0][X1 + 1] - sh.os[0][X1]) * (sh.es[0][Y1 + 1] - sh.es[0][Y1]) *
                       (sh.os[1][X2 + 1] - sh.os[1][X2]) * (sh.es[1][Y2 + 1] - sh.es[1][Y2]);
            }
            // digit order inside the block: active indices slowest, core next, virtual fastest, so
            // that the lanes of one warp iteration share the active remnant of their neighbours
            if (kind == 0) {
                order = cls_pri(X1) > cls_pri(Y1) ? 1u : 0u;                         // occ fastest?
            } else if (kind == 1) {
                int po = min(cls_pri(X1), cls_pri(X2)), pe = min(cls_pri(Y1), cls_pri(Y2));
                order = (pe < po ? 1u : 0u) | ((X1 != X2 && cls_pri(X1) > cls_pri(X2)) ? 2u : 0u) |
                        ((Y1 != Y2 && cls_pri(Y1) > cls_pri(Y2)) ? 4u : 0u);
            } else {
                int cl[4] = {X1, Y1, X2, Y2}, perm[4] = {0, 1, 2, 3};
                for (int a = 1; a < 4; a++)       // stable insertion sort by class priority
                    for (int b2 = a; b2 > 0 && cls_pri(cl[perm[b2]]) < cls_pri(cl[perm[b2 - 1]]); b2--) {
                        int t = perm[b2]; perm[b2] = perm[b2 - 1]; perm[b2 - 1] = t;
                    }
                order = (unsigned)perm[0] | ((unsigned)perm[1] << 2) | ((unsigned)perm[2] << 4) |
                        ((unsigned)perm[3] << 6);
            }
            int dh = (X1 == 0) - (Y1 == 0), dp = (Y1 == 2) - (X1 == 2);
            if (kind != 0) {
                dh += (X2 == 0) - (Y2 == 0);
                dp += (Y2 == 2) - (X2 == 2);
            }
            if (h + dh > 2 || p + dp > 2) size = 0;
        }
        unsigned vm = __ballot_sync(0xffffffffu, size > 0);
        // inclusive scan of sizes (invalid lanes contribute 0) -> global prefix via the carry
        int x = size;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (size > 0) {
            int k = run + __popc(vm & ((1u << lane) - 1u));
            sh.bdesc[k] = (unsigned)kind | ((unsigned)sg << 2) | ((unsigned)X1 << 4) | ((unsigned)X2 << 6) |
                          ((unsigned)Y1 << 8) | ((unsigned)Y2 << 10) | (order << 12);
            sh.bstart[k + 1] = carry + x;
        }
        carry += __shfl_sync(0xffffffffu, x, 31);
        run += __popc(vm);
    }
    if (lane == 0) {
        sh.nb = run;
        sh.bstart[0] = 0;
    }
    __syncwarp();
}

// pair index -> (i < j) in lexicographic order (i slowest, j fastest) among k items
__device__ __forceinline__ void lex_decode(int op, int k, int& i, int& j) {
    int ti, tj;
    tri_decode(k * (k - 1) / 2 - 1 - op, ti, tj);
    i = k - 1 - tj;
    j = k - 1 - ti;
}

// pair within one class (lexicographic) or across two classes (rev: first index fastest)
__device__ __forceinline__ void pair_decode(int op, bool same, int k1, int k2, bool rev, int& i, int& j) {
    if (same) lex_decode(op, k1, i, j);
    else if (rev) { j = op / k1; i = op - j * k1; }
    else { i = op / k2; j = op - i * k2; }
}

// decode neighbour `loc` of block `desc` into removed r1<=r2 and added a1<=a2 spin orbitals
__device__ __forceinline__ void decode_exc(const WarpLists& sh, int n, unsigned desc, int loc, int& kind, int& r1,
                                           int& r2, int& a1, int& a2) {
    kind = desc & 3;
    int sg = (desc >> 2) & 1, X1 = (desc >> 4) & 3, X2 = (desc >> 6) & 3, Y1 = (desc >> 8) & 3,
        Y2 = (desc >> 10) & 3;
    const unsigned order = desc >> 12;
    if (kind == 0) {
        int nX = sh.os[sg][X1 + 1] - sh.os[sg][X1], nY = sh.es[sg][Y1 + 1] - sh.es[sg][Y1];
        int i, a;
        if (order & 1u) { a = loc / nX; i = loc - a * nX; }
        else { i = loc / nY; a = loc - i * nY; }
        r1 = r2 = sg * n + sh.ol[sg][sh.os[sg][X1] + i];
        a1 = a2 = sg * n + sh.el[sg][sh.es[sg][Y1] + a];
    } else if (kind == 1) {
        int k1 = sh.os[sg][X1 + 1] - sh.os[sg][X1], k2 = sh.os[sg][X2 + 1] - sh.os[sg][X2];
        int e1 = sh.es[sg][Y1 + 1] - sh.es[sg][Y1], e2 = sh.es[sg][Y2 + 1] - sh.es[sg][Y2];
        int nOP = pairs_of(k1, k2, X1 == X2), nEP = pairs_of(e1, e2, Y1 == Y2);
        int op, ep;
        if (order & 1u) { ep = loc / nOP; op = loc - ep * nOP; }
        else { op = loc / nEP; ep = loc - op * nEP; }
        int i, j, a, b;
        pair_decode(op, X1 == X2, k1, k2, (order & 2u) != 0, i, j);
        pair_decode(ep, Y1 == Y2, e1, e2, (order & 4u) != 0, a, b);
        r1 = sg * n + sh.ol[sg][sh.os[sg][X1] + i];
        r2 = sg * n + sh.ol[sg][sh.os[sg][X2] + j];
        a1 = sg * n + sh.el[sg][sh.es[sg][Y1] + a];
        a2 = sg * n + sh.el[sg][sh.es[sg][Y2] + b];
    } else {
        // digits 0: alpha occupied (X1), 1: alpha empty (Y1), 2: beta occupied (X2), 3: beta empty (Y2)
        int rad[4] = {sh.os[0][X1 + 1] - sh.os[0][X1], sh.es[0][Y1 + 1] - sh.es[0][Y1],
                      sh.os[1][X2 + 1] - sh.os[1][X2], sh.es[1][Y2 + 1] - sh.es[1][Y2]};
        int x[4];
#pragma unroll
        for (int d = 3; d >= 0; d--) {
            int id = (order >> (2 * d)) & 3u;
            int q = loc / rad[id];
            x[id] = loc - q * rad[id];
            loc = q;
        }
        r1 = sh.ol[0][sh.os[0][X1] + x[0]];
        a1 = sh.el[0][sh.es[0][Y1] + x[1]];
        r2 = n + sh.ol[1][sh.os[1][X2] + x[2]];
        a2 = n + sh.el[1][sh.es[1][Y2] + x[3]];
    }
}

__device__ __forceinline__ bool active_only(unsigned desc) {
    int kind = desc & 3, X1 = (desc >> 4) & 3, X2 = (desc >> 6) & 3, Y1 = (desc >> 8) & 3, Y2 = (desc >> 10) & 3;
    if (kind == 0) return X1 == 1 && Y1 == 1;
    return X1 == 1 && X2 == 1 && Y1 == 1 && Y2 == 1;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// <d|H|d> and <d|H_D|d> (lane-parallel over occupied pairs); label >= 0 required for H_D
template <int W>
__device__ void diagonals(const SysDev& S, const WarpLists& sh, const unsigned long long (&d)[2][W], int lane,
                          double& hnn, double& hdnn) {
    const int na_ = sh.os[0][3], nb_ = sh.os[1][3], N = na_ + nb_;
    double h = 0.0, hd = 0.0;
    for (int k = lane; k < N; k += 32) {
        int p = k < na_ ? sh.ol[0][k] : sh.ol[1][k - na_];
        h += __ldg(S.h1 + p * S.n + p);
        int cls = p < S.nc ? 0 : (p < S.nc + S.na ? 1 : 2);
        if (cls == 1) hd += __ldg(S.hc + p * S.n + p);
        else if (cls == 2) hd += __ldg(S.eps + p);
    }
    // core holes
    for (int sg = 0; sg < 2; sg++) {
        for (int k = lane; k < S.nc - sh.os[sg][1]; k += 32) hd -= __ldg(S.eps + sh.el[sg][k]);
    }
    const int npair = N * (N - 1) / 2;
    for (int q = lane; q < npair; q += 32) {
        int j, i;
        tri_decode(q, i, j);
        int si = i >= na_, sj = j >= na_;
        int p1 = si ? sh.ol[1][i - na_] : sh.ol[0][i];
        int p2 = sj ? sh.ol[1][j - na_] : sh.ol[0][j];
        double v = eri_g(S, p1, p1, p2, p2);
        if (si == sj) v -= eri_g(S, p1, p2, p2, p1);
        h += v;
        bool a1 = p1 >= S.nc && p1 < S.nc + S.na, a2 = p2 >= S.nc && p2 < S.nc + S.na;
        if (a1 && a2) hd += v;
    }
    hnn = warp_sum(h) + S.e_nuc;
    hdnn = warp_sum(hd) + S.e_core;
}

// ============================================================================ the walk

#include "mrq_cas.cuh"

// The walkers of one launch: one or several systems, each with its own walker array; slot numbers
// run over all systems (system k owns slots [offsets[k], offsets[k+1])).
struct WalkSet {
    const SysDev* systems;
    Walker* const* walkers;
    const long long* offsets;
    int nsys;
    long long nslots;
};

#include "mrq_walk.cuh"

__global__ void k_walkers_init(Walker* w, long long nslots, unsigned long long d0, unsigned long long d1,
                               unsigned long long d2, unsigned long long d3, double psi, int sys, int G) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nslots) return;
    Walker x;
    x.d[0][0] = d0; x.d[0][1] = d1; x.d[1][0] = d2; x.d[1][1] = d3;
    x.psi = psi;
    x.step = 0;
    x.wid = (unsigned)i;
    x.sys = sys;
    x.group = (int)(i % G);
    x.rl = -1;
    x.rw = x.rEL = x.rnum = 0.0;
    x.rtype = 0;
    x.rpad = 0;
    w[i] = x;
}

// ============================================================================ setup kernels

// insert reference determinants (and validate them: full core, empty virtuals, electron counts)
template <int W>
__global__ void k_hash_build(const SysDev* __restrict__ sys, HashSlot* __restrict__ hash, const unsigned long long* dets,
                             const double* coeffs, long long nref, int* err) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nref) return;
    const SysDev S = *sys;
    unsigned long long d[2][W];
#pragma unroll
    for (int w = 0; w < W; w++) {
        d[0][w] = dets[i * 2 * W + w];
        d[1][w] = dets[i * 2 * W + W + w];
    }
    int ca = 0, cb = 0;
    bool bad = false;
#pragma unroll
    for (int w = 0; w < W; w++) {
        ca += __popcll(d[0][w]);
        cb += __popcll(d[1][w]);
        unsigned long long all = S.mcore[w] | S.mact[w] | S.mvirt[w];
        for (int sg = 0; sg < 2; sg++) {
            if ((d[sg][w] & S.mcore[w]) != S.mcore[w]) bad = true;
            if (d[sg][w] & S.mvirt[w]) bad = true;
            if (d[sg][w] & ~all) bad = true;
        }
    }
    if (ca != S.nalpha || cb != S.nbeta) bad = true;
    if (bad) {
        atomicOr(err, 8);
        return;
    }
    unsigned long long key = hash_key(S, active_bits<W>(S, d[0]), active_bits<W>(S, d[1]));
    unsigned long long hidx = mix64(key) & S.hmask;
    for (int k = 0; k < S.max_probe; k++) {
        unsigned long long prev = atomicCAS(&hash[hidx].key, MRQ_EMPTY_KEY, key);
        if (prev == MRQ_EMPTY_KEY) {
            hash[hidx].val = coeffs[i];
            return;
        }
        if (prev == key) {
            atomicOr(err, 16);   // duplicate determinant
            return;
        }
        hidx = (hidx + 1) & S.hmask;
    }
    atomicOr(err, 32);   // probe bound exceeded
}

__global__ void k_hash_clear(HashSlot* hash, unsigned long long cap) {
    unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < cap) {
        hash[i].key = MRQ_EMPTY_KEY;
        hash[i].val = 0.0;
    }
}

// half-unpacked integral table E[P(p,q)][r][s] from the 8-fold packed input
__global__ void k_expand_eri(const double* __restrict__ eri, double* __restrict__ eri4, int n) {
    const long long npair = (long long)n * (n + 1) / 2;
    const long long total = npair * n * n;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        long long P = t / ((long long)n * n);
        int rs = (int)(t - P * n * n);
        int r = rs / n, s = rs - r * n;
        long long Q = r >= s ? (long long)r * (r + 1) / 2 + s : (long long)s * (s + 1) / 2 + r;
        long long i = P >= Q ? P * (P + 1) / 2 + Q : Q * (Q + 1) / 2 + P;
        eri4[t] = eri[i];
    }
}

// physicists' tables on the (core+active) x (core+active) x (active+virtual) x (active+virtual)
// block: T[p][q][r][s] = <pq|rs> = (pr|qs) and, after tab_half entries, <pq||rs>
__global__ void k_build_tab(const SysDev* __restrict__ sys, double* __restrict__ tab) {
    const SysDev S = *sys;
    const long long a = S.nca, v = S.nav, half = a * a * v * v;
    for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < half; t += (long long)gridDim.x * blockDim.x) {
        const int s = (int)(t % v) + S.nc, r = (int)((t / v) % v) + S.nc;
        const int q = (int)((t / (v * v)) % a), p = (int)(t / (v * v * a));
        const double d = eri_g(S, p, r, q, s), x = eri_g(S, p, s, q, r);
        tab[t] = hb_screen(S, d);                 // every double the CAS path takes reads one entry
        tab[half + t] = hb_screen(S, d - x);
    }
}

// terms of the single-excitation operator (SysDev::sgl)
__global__ void k_build_sgl(const SysDev* __restrict__ sys, double* __restrict__ sgl) {
    const SysDev S = *sys;
    const int blk = S.nca * S.nav, half = S.na * blk;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < half; t += gridDim.x * blockDim.x) {
        const int j = S.nc + t / blk, y = (t % blk) / S.nav, x = S.nc + t % S.nav;
        const double d = eri_g(S, y, x, j, j);
        sgl[t] = d - eri_g(S, y, j, j, x);
        sgl[half + t] = d;
    }
}

// hc_pq = h_pq + sum_i [2(pq|ii) - (pi|iq)]
__global__ void k_core_fock(const SysDev* __restrict__ sys, double* hc) {
    const SysDev S = *sys;
    int pq = blockIdx.x * blockDim.x + threadIdx.x;
    if (pq >= S.n * S.n) return;
    int p = pq / S.n, q = pq % S.n;
    double v = __ldg(S.h1 + pq);
    for (int i = 0; i < S.nc; i++) v += 2.0 * eri_g(S, p, q, i, i) - eri_g(S, p, i, i, q);
    hc[pq] = v;
}

// block-level deterministic sum of `nv` values per thread into out[blockIdx.x * nv + k]
template <int NV>
__device__ void block_sum_store(double (&v)[NV], double* out) {
    __shared__ double red[32][NV];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int k = 0; k < NV; k++) {
        double x = warp_sum(v[k]);
        if (lane == 0) red[wid][k] = x;
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        double s = 0.0;
        for (int w = 0; w < nw; w++) s += red[w][threadIdx.x];
        out[(long long)blockIdx.x * NV + threadIdx.x] = s;
    }
    __syncthreads();
}

#define MRQ_REF_BLOCKS 304       // blocks of k_ref_sum

// <k|H|k> of every reference determinant: e_nuc + sum_p [h_pp + 1/2 sum_q ((pp|qq) - delta (pq|qp))], one
// running sum per determinant (its rounding is that of E0 against the perturbers' energies), one thread
// each, and every determinant's integrals in the same order, so that a warp's reads coincide or nearly do
template <int W>
__global__ void __launch_bounds__(128) k_ref_diag(const SysDev* __restrict__ sys, const unsigned long long* __restrict__ dets,
                                                  long long nref, double* __restrict__ e) {
    const SysDev& S = *sys;
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nref) return;
    unsigned long long d[2][W];
#pragma unroll
    for (int w = 0; w < W; w++) {
        d[0][w] = dets[i * 2 * W + w];
        d[1][w] = dets[i * 2 * W + W + w];
    }
    double hdiag = S.e_nuc;
#pragma unroll
    for (int sg = 0; sg < 2; sg++)
#pragma unroll
        for (int w = 0; w < W; w++) {
            unsigned long long om = d[sg][w];
            while (om) {
                const int p1 = 64 * w + __ffsll(om) - 1;
                om &= om - 1;
                hdiag += __ldg(S.h1 + p1 * S.n + p1);
#pragma unroll
                for (int sg2 = 0; sg2 < 2; sg2++)
#pragma unroll
                    for (int w2 = 0; w2 < W; w2++) {
                        unsigned long long om2 = d[sg2][w2];
                        while (om2) {
                            const int p2 = 64 * w2 + __ffsll(om2) - 1;
                            om2 &= om2 - 1;
                            hdiag += 0.5 * eri_g(S, p1, p1, p2, p2);
                            if (sg == sg2) hdiag -= 0.5 * eri_g(S, p1, p2, p2, p1);
                        }
                    }
            }
        }
    e[i] = hdiag;
}

// E0 numerator per reference determinant k: e[k] <- c_k^2 H_kk + 2 sum_{k' > k} c_k H_kk' c_k', one warp each.
// A pair is taken at the determinant of the smaller key (H is symmetric).  The opposite-spin doubles, most
// of the pairs, run over a list of the alpha singles and one of the beta singles that raise the key, in
// shared memory: a pair costs one probe, one integral and one FMA.  The other excitations are decoded one
// per lane.  Bound by the random reads.  (One thread per determinant took 2.5 ms on 63,504 determinants,
// a warp decoding every excitation 1.9 ms.)
#define MRQ_REF_SINGLES 256          // singles of one spin of <= 32 active orbitals
template <int W>
__global__ void __launch_bounds__(256) k_ref_energy(const SysDev* __restrict__ sys, const unsigned long long* __restrict__ dets,
                                                    const double* __restrict__ coeffs, long long nref, double* __restrict__ e) {
    __shared__ SysDev S;
    __shared__ uint2 list[8][2][MRQ_REF_SINGLES];      // new string; integral index, sign in bit 31
    for (int k = threadIdx.x; k < (int)(sizeof(SysDev) / sizeof(int)); k += blockDim.x)
        reinterpret_cast<int*>(&S)[k] = reinterpret_cast<const int*>(sys)[k];
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, n = S.n;
    const long long nwarp = (long long)gridDim.x * (blockDim.x >> 5);
    const unsigned am = (S.na >= 32) ? 0xFFFFFFFFu : ((1u << S.na) - 1u);
    NoCtr z;
    for (long long i = (long long)blockIdx.x * (blockDim.x >> 5) + warp; i < nref; i += nwarp) {
        unsigned long long d[2][W];
#pragma unroll
        for (int w = 0; w < W; w++) {
            d[0][w] = dets[i * 2 * W + w];
            d[1][w] = dets[i * 2 * W + W + w];
        }
        const double ck = coeffs[i];
        const unsigned ao0 = active_bits<W>(S, d[0]), ao1 = active_bits<W>(S, d[1]);
        const unsigned long long oa = ao0, ob = (unsigned long long)ao1 << 32, AO = oa | ob;
        const unsigned long long ea = ~ao0 & am, eb = (unsigned long long)(~ao1 & am) << 32;
        const unsigned long long key = hash_key(S, ao0, ao1);
        double sum = 0.0;
        int cnt[2];
        __syncwarp();
#pragma unroll
        for (int sg = 0; sg < 2; sg++) {
            const unsigned o = sg ? ao1 : ao0, em = ~o & am;
            const int co = __popc(o), ce = __popc(em), tot = co * ce;
            int run = 0;
            for (int base = 0; base < tot; base += 32) {
                const int q = base + lane;
                bool on = q < tot;
                unsigned str = 0, idx = 0;
                if (on) {
                    const int x = nth_bit64(o, q / ce), y = nth_bit64(em, q % ce);
                    str = o ^ (1u << x) ^ (1u << y);
                    const int odd = __popc(o & ((1u << max(x, y)) - 1u) & ~((2u << min(x, y)) - 1u)) & 1;
                    const int p = S.nc + y, r = S.nc + x;
                    idx = sg == 0 ? (unsigned)pair_idx(p, r) * (unsigned)(n * n) : (unsigned)(p * n + r);
                    idx |= (unsigned)odd << 31;
                    on = sg == 0 || str > o;                      // the beta string decides the key's order
                }
                const unsigned m = __ballot_sync(0xffffffffu, on);
                if (on) list[warp][sg][run + __popc(m & ((1u << lane) - 1u))] = make_uint2(str, idx);
                run += __popc(m);
            }
            cnt[sg] = run;
        }
        __syncwarp();
        for (int q = lane; q < cnt[0] * cnt[1]; q += 32) {
            const int ib = q / cnt[0];
            const uint2 a = list[warp][0][q - ib * cnt[0]], b = list[warp][1][ib];
            const double c = hash_lookup(S, hash_key(S, a.x, b.x));
            if (c != 0.0)
                sum += 2.0 * (ck * c) * neg_if(__ldg(S.eri4 + ((a.y & 0x7FFFFFFFu) + (b.y & 0x7FFFFFFFu))), (int)((a.y ^ b.y) >> 31));
        }
        // singles and same-spin doubles
        const int same = active_neighbours(__popcll(oa), __popcll(ob), __popcll(ea), __popcll(eb)) -
                         __popcll(oa) * __popcll(ob) * __popcll(ea) * __popcll(eb);
        for (int q = lane; q < same; q += 32) {
            unsigned long long Xb, Yb;
            const int r = active_neighbour(S, oa, ob, ea, eb, q, Xb, Yb);
            const unsigned long long km = (AO & ~Xb) | Yb;
            const unsigned long long kk = hash_key(S, (unsigned)km, (unsigned)(km >> 32));
            if (kk < key) continue;
            const double c = hash_lookup(S, kk);
            if (c == 0.0) continue;
            int rem[2], add[2];
            act_list(S, Xb, rem);
            act_list(S, Yb, add);
            double h;
            if (r == 1) {
                const int sx = rem[0] >= n, px = rem[0] - sx * n, py = add[0] - sx * n;
                h = __ldg(S.hc + py * n + px);
                const double* const col = S.sgl + py * S.nav + (px - S.nc);
                for (unsigned long long bits = AO; bits; bits &= bits - 1) {
                    const int b = __ffsll(bits) - 1;
                    h += __ldg(col + (long long)((b & 31) + (((b >= 32) == (sx == 1)) ? 0 : S.na)) * S.nca * S.nav);
                }
                h = neg_if(h, popc_sel<W>(d, sx, min(px, py), max(px, py)));
            } else {
                h = double_elem<W>(S, d, rem[0], rem[1], add[0], add[1], z);
            }
            sum += 2.0 * (ck * c) * h;
        }
        sum = warp_sum(sum);
        if (lane == 0) e[i] = ck * ck * e[i] + sum;
    }
}

// sums of the determinants' numerators and of c_k^2, partials per block
__global__ void __launch_bounds__(128) k_ref_sum(const double* __restrict__ e, const double* __restrict__ coeffs, long long nref,
                                                 double* partial) {
    double acc[2] = {0.0, 0.0};
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nref; i += (long long)gridDim.x * blockDim.x) {
        acc[0] += e[i];
        acc[1] += coeffs[i] * coeffs[i];
    }
    block_sum_store<2>(acc, partial);
}

// spin-summed active 1-RDM element gamma_tu (unnormalised): block (t, u; slice) over a slice of the
// determinants, partial sums added in order by k_setup_finish
#define MRQ_RDM_SLICES 16
template <int W>
__global__ void __launch_bounds__(256) k_ref_rdm(const SysDev* __restrict__ sys, const unsigned long long* __restrict__ dets,
                                                 const double* __restrict__ coeffs, long long nref, double* partial) {
    const SysDev& S = *sys;
    const int t = blockIdx.x / S.na, u = blockIdx.x % S.na;
    double acc[1] = {0.0};
    for (long long i = (long long)blockIdx.y * blockDim.x + threadIdx.x; i < nref; i += (long long)gridDim.y * blockDim.x) {
        unsigned long long d[2][W];
#pragma unroll
        for (int w = 0; w < W; w++) {
            d[0][w] = dets[i * 2 * W + w];
            d[1][w] = dets[i * 2 * W + W + w];
        }
        const double ck = coeffs[i];
        const unsigned ao[2] = {active_bits<W>(S, d[0]), active_bits<W>(S, d[1])};
        for (int sg = 0; sg < 2; sg++) {
            // <phi0| a+_t a_u |phi0>: d has u occupied; k' = d - u + t
            if (!((ao[sg] >> u) & 1u)) continue;
            if (t == u) {
                acc[0] += ck * ck;
                continue;
            }
            if ((ao[sg] >> t) & 1u) continue;
            unsigned k0 = ao[0], k1 = ao[1];
            (sg ? k1 : k0) ^= (1u << t) | (1u << u);
            double c = hash_lookup(S, hash_key(S, k0, k1));
            if (c != 0.0) acc[0] += ck * c * sgn_single<W>(d[sg], S.nc + u, S.nc + t);
        }
    }
    __shared__ double red[32];
    double x = warp_sum(acc[0]);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x + 31) / 32; w++) s += red[w];
        partial[(long long)blockIdx.x * gridDim.y + blockIdx.y] = s;
    }
}

// reduce E0 partials (fixed order), normalise gamma, eps_p = F_pp, E_core; writes scal[0..4]
__global__ void __launch_bounds__(1024) k_setup_finish(const SysDev* __restrict__ sys, const double* __restrict__ partial,
                                                       const double* __restrict__ rdm, double* gamma, double* eps,
                                                       double* scal) {
    const SysDev& S = *sys;
    __shared__ double s_part[2][MRQ_REF_BLOCKS], s_sum[2], s_pair[64 * 64], s_ec;      // n_core <= 64
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = threadIdx.x; i < 2 * MRQ_REF_BLOCKS; i += blockDim.x) s_part[i & 1][i >> 1] = partial[i];
    for (int k = threadIdx.x; k < S.nc * S.nc; k += blockDim.x) {
        const int i = k / S.nc, j = k - i * S.nc;
        s_pair[k] = 2.0 * eri_g(S, i, i, j, j) - eri_g(S, i, j, j, i);
    }
    __syncthreads();
    if (threadIdx.x < 64 && lane == 0) {     // two running sums over the blocks
        double a = 0.0;
        for (int i = 0; i < MRQ_REF_BLOCKS; i++) a += s_part[warp][i];
        s_sum[warp] = a;
    }
    __syncthreads();
    const double num = s_sum[0], norm = s_sum[1];
    if (threadIdx.x == 0) {              // the core energy: one running sum over the orbitals
        double ec = S.e_nuc;
        for (int i = 0; i < S.nc; i++) {
            ec += 2.0 * __ldg(S.h1 + i * S.n + i);
            for (int j = 0; j < S.nc; j++) ec += s_pair[i * S.nc + j];
        }
        s_ec = ec;
    }
    const int na = S.na;
    for (int k = threadIdx.x; k < na * na; k += blockDim.x) {
        double g = 0.0;
        for (int q = 0; q < MRQ_RDM_SLICES; q++) g += rdm[k * MRQ_RDM_SLICES + q];
        gamma[k] = g / norm;
    }
    __syncthreads();
    for (int p = warp; p < S.n; p += nw) {               // a warp per orbital, lanes over (t, u)
        double v = 0.0;
        for (int k = lane; k < na * na; k += 32) {
            const int t = S.nc + k / na, u = S.nc + k % na;
            v += gamma[k] * (eri_g(S, p, p, t, u) - 0.5 * eri_g(S, p, t, u, p));
        }
        v = warp_sum(v);
        if (lane == 0) eps[p] = __ldg(S.hc + p * S.n + p) + v;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double se = 0.0;
        for (int i = 0; i < S.nc; i++) se += eps[i];
        scal[0] = num / norm;
        scal[1] = norm;
        scal[2] = s_ec;
        scal[3] = se;
    }
}

__global__ void k_default_coeffs(double* c, long long n) {
    for (long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x; l < n; l += (long long)gridDim.x * blockDim.x)
        c[l] = l == 0 ? 1.0 : 0.1;
}

// the race's screen and exact clock for given (k, rate, best clock) triples (parity of the move
// selection's screen); the screen takes the FP32 images exactly as the walk forms them
__global__ void k_race_screen(const unsigned long long* __restrict__ k, const double* __restrict__ rate,
                              const double* __restrict__ tbest, long long n, unsigned char* __restrict__ pass,
                              double* __restrict__ exact) {
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float btf = isinf(tbest[i]) ? INFINITY : (float)tbest[i];
    const float gf = abs_f32_of(rate[i]);
    pass[i] = race_pass((unsigned)(k[i] >> 21), gf > 0.0f ? gf : INFINITY, race_scale(race_bound(btf), 1.0f)) &&
              race_may_win(k[i], gf, race_bound(btf));
    exact[i] = race_clock_f64(k[i], rate[i]);
}

// index of the largest |c| (first on ties), one block
__global__ void k_argmax_abs(const double* c, long long n, long long* out) {
    __shared__ double bv[1024];
    __shared__ long long bi[1024];
    double v = -1.0;
    long long idx = 0;
#pragma unroll 8
    for (long long i = threadIdx.x; i < n; i += blockDim.x) {
        double a = fabs(c[i]);
        if (a > v) { v = a; idx = i; }
    }
    bv[threadIdx.x] = v;
    bi[threadIdx.x] = idx;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            double v2 = bv[threadIdx.x + s];
            long long i2 = bi[threadIdx.x + s];
            if (v2 > bv[threadIdx.x] || (v2 == bv[threadIdx.x] && i2 < bi[threadIdx.x])) {
                bv[threadIdx.x] = v2;
                bi[threadIdx.x] = i2;
            }
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = bi[0];
}

// ============================================================================ finalize (Eq. 14-15)

static const long long FIN_CHUNK = 8192;    // labels per partial sum
#define FIN_Q 5    // per type: kept ratio, e2, screened count, screened ratio, visited count
#define FIN_NV (MRQ_NTYPES * FIN_Q)

__device__ __forceinline__ int label_type(long long l, long long nPs, int nc2, int nv2) {
    long long rh = l / nPs, rp = l - rh * nPs;
    int h = rh == 0 ? 0 : (rh <= nc2 ? 1 : 2);
    int p = rp == 0 ? 0 : (rp <= nv2 ? 1 : 2);
    return 3 * h + p;
}

// The visited labels of every chunk, in label order: list[chunk ...], how many in list[nlab + chunk].
// A walk visits few of its labels (a few thousand of 256,038 at 56 orbitals), so one pass over the
// accumulators finds them and the G + 1 jackknife variants read only those.  Bound by the one read
// of accN (G x labels).
__global__ void __launch_bounds__(1024) k_fin_list(const SysDev* __restrict__ sys, long long chunk, int* __restrict__ list) {
    const int G = sys->G;
    const long long L = sys->nlab, lo = blockIdx.x * chunk, hi = min(L, lo + chunk);
    const double* const accN = sys->accN;
    __shared__ int s_w[32];
    int run = 0;
    for (long long base = lo; base < hi; base += 1024) {
        const long long l = base + threadIdx.x;
        bool seen = false;
        if (l > 0 && l < hi) {
            unsigned long long any = 0;              // some bit of some group's sum (the sign aside) is set
#pragma unroll 8
            for (int g = 0; g < G; g++) any |= (unsigned long long)__double_as_longlong(accN[(long long)g * L + l]) << 1;
            seen = any != 0;
        }
        const unsigned m = __ballot_sync(0xffffffffu, seen);
        if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = __popc(m);
        __syncthreads();
        int at = run, all = 0;
        for (int w = 0; w < 32; w++) {
            if (w < (int)(threadIdx.x >> 5)) at += s_w[w];
            all += s_w[w];
        }
        if (seen) list[lo + at + __popc(m & ((1u << (threadIdx.x & 31)) - 1u))] = (int)l;
        run += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) list[L + blockIdx.x] = run;
}

// block (v, chunk): visited labels of the chunk under variant v (v < G: group v left out; v == G: all)
__global__ void __launch_bounds__(256) k_fin_labels(const SysDev* __restrict__ sys, double tau, int nchunk, long long chunk,
                                                    const int* __restrict__ list, double* partial) {
    const SysDev& S = *sys;
    const int v = blockIdx.x / nchunk, ch = blockIdx.x % nchunk;
    const int G = S.G;
    const long long L = S.nlab;
    const int n = list[L + ch];
    __shared__ double s_n0;
    if (threadIdx.x == 0) {
        double a = 0.0;
        for (int g = 0; g < G; g++) a += S.accN[(long long)g * L];
        if (v < G) a -= S.accN[(long long)v * L];
        s_n0 = a;
    }
    __syncthreads();
    const double n0 = s_n0;
    double acc[FIN_NV];
#pragma unroll
    for (int k = 0; k < FIN_NV; k++) acc[k] = 0.0;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const long long l = list[(long long)ch * chunk + k];
        double Nl = 0.0, Ul = 0.0;
        for (int g = 0; g < G; g++) {
            Nl += S.accN[(long long)g * L + l];
            Ul += S.accU[(long long)g * L + l];
        }
        if (v < G) {
            Nl -= S.accN[(long long)v * L + l];
            Ul -= S.accU[(long long)v * L + l];
        }
        if (!(Nl > 0.0)) continue;
        const int t = label_type(l, S.nPs, 2 * S.nc, 2 * S.nv);
        const double ratio = Nl / n0;
        double q[FIN_Q] = {0.0, 0.0, 0.0, 0.0, 1.0};
        if (ratio >= tau) {
            const double El = Ul / Nl;
            q[0] = ratio;
            q[1] = ratio / (S.e0 - El);
        } else {
            q[2] = 1.0;
            q[3] = ratio;
        }
#pragma unroll
        for (int tt = 0; tt < MRQ_NTYPES; tt++)
            if (tt == t) {
#pragma unroll
                for (int j = 0; j < FIN_Q; j++) acc[tt * FIN_Q + j] += q[j];
            }
    }
    if (n == 0) {                    // no visited label: zeros without the reduction
        for (int k = threadIdx.x; k < FIN_NV; k += blockDim.x) partial[(long long)blockIdx.x * FIN_NV + k] = 0.0;
        return;
    }
    block_sum_store<FIN_NV>(acc, partial);
}

// one block: sum chunk partials in order, every reported quantity of every variant (one thread each), then
// one thread per quantity runs the jackknife over the groups and writes the result struct
__global__ void __launch_bounds__(1024) k_fin_reduce(const SysDev* __restrict__ sys, const double* __restrict__ partial,
                                                     int nchunk, mrq_result* res) {
    const SysDev& S = *sys;
    const int G = S.G;
    const long long L = S.nlab;
    __shared__ double vals[65][FIN_NV];   // G <= 64
    __shared__ double sW[64], sE[64], sN[64];
    for (int g = threadIdx.x; g < G; g += blockDim.x) {
        sW[g] = S.accW[g];
        sE[g] = S.accE[g];
        sN[g] = S.accN[(long long)g * L];
    }
    for (int idx = threadIdx.x; idx < (G + 1) * FIN_NV; idx += blockDim.x) {
        int v = idx / FIN_NV, k = idx % FIN_NV;
        double s = 0.0;
#pragma unroll 8
        for (int c = 0; c < nchunk; c++) s += partial[((long long)v * nchunk + c) * FIN_NV + k];
        vals[v][k] = s;
    }
    __syncthreads();
    const double c0 = S.c[0];
    const double f = G > 1 ? (double)(G - 1) / G : NAN;
    // quantity q of variant v: 0 E^(2), 1 E_var, 2 a_0^2, then per type its norm and E^(2)
    constexpr int NQ = 3 + 2 * MRQ_NTYPES;
    __shared__ double x[65][NQ];
    for (int idx = threadIdx.x; idx < (G + 1) * NQ; idx += blockDim.x) {
        const int v = idx / NQ, q = idx - v * NQ;
        double y = 0.0;
        if (q == 0) {
            for (int t = 0; t < MRQ_NTYPES; t++) y += vals[v][t * FIN_Q + 1];
        } else if (q < 3) {
            double Wt = 0.0, Xt = 0.0;
            for (int g = 0; g < G; g++) {
                Wt += sW[g];
                Xt += q == 1 ? sE[g] : sN[g];
            }
            const double Wv = Wt - (v < G ? sW[v] : 0.0), Xv = Xt - (v < G ? (q == 1 ? sE[v] : sN[v]) : 0.0);
            y = q == 1 ? Xv / Wv : c0 * c0 * Xv / Wv;
        } else {
            y = vals[v][(q - 3) / 2 * FIN_Q + (q - 3) % 2];
        }
        x[v][q] = y;
    }
    __syncthreads();
    if (threadIdx.x < NQ) {
        const int q = threadIdx.x;
        const double full = x[G][q];
        double m = 0.0, var = 0.0;
        for (int g = 0; g < G; g++) m += x[g][q];
        m /= G;
        for (int g = 0; g < G; g++) var += (x[g][q] - m) * (x[g][q] - m);
        const double sigma = sqrt(f * var);
        if (q == 0) {
            res->e0 = S.e0;
            res->e2 = full;
            res->e2_sigma = sigma;
        } else if (q == 1) {
            const double a0 = x[G][2];
            res->e_var = full;
            res->e_var_sigma = sigma;
            res->e_mrci_q = full + (1.0 - a0) * (full - S.e0);
        } else if (q == 2) {
            res->a0sq = full;
            res->a0sq_sigma = sigma;
        } else {
            const int t = (q - 3) / 2;
            if ((q - 3) % 2 == 0) {
                res->type_norm[t] = full;
                res->type_norm_sigma[t] = sigma;
                res->type_screened[t] = vals[G][t * FIN_Q + 2];
                res->type_steps[t] = (long long)S.type_steps[t];
            } else {
                res->type_e2[t] = full;
                res->type_e2_sigma[t] = sigma;
            }
        }
    } else if (threadIdx.x == 32) {
        double scr_norm = 0.0, visited = 0.0;
        long long wsteps = 0;
        for (int t = 0; t < MRQ_NTYPES; t++) {
            scr_norm += vals[G][t * FIN_Q + 3];
            visited += vals[G][t * FIN_Q + 4];
            wsteps += (long long)S.type_steps[t];
        }
        res->screened_norm = scr_norm;
        res->n_labels_visited = visited;
        res->walker_steps = wsteps;
    }
}

// ============================================================================ SC-MRCI(s) optimisation (Eq. 8-9)

// grad[l] = (A_l - E B_l) / W over all groups, E = sum E / sum W: <delta_{l,l_n}/c_l (E_L - E)>
__global__ void k_mrci_grad(const SysDev* __restrict__ sys, double* __restrict__ grad, double* __restrict__ energy) {
    const SysDev S = *sys;
    double Wt = 0.0, Et = 0.0;
    for (int g = 0; g < S.G; g++) {
        Wt += S.accW[g];
        Et += S.accE[g];
    }
    const double E = Et / Wt;
    for (long long l = (long long)blockIdx.x * blockDim.x + threadIdx.x; l < S.nlab; l += (long long)gridDim.x * blockDim.x) {
        double a = 0.0, b = 0.0;
        for (int g = 0; g < S.G; g++) {
            a += S.accA[(long long)g * S.nlab + l];
            b += S.accB[(long long)g * S.nlab + l];
        }
        grad[l] = (a - E * b) / Wt;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) *energy = E;
}

// AMSGrad (Reddi, Kale, Kumar, ICLR 2018) on c_l, l >= 1; c_0 stays fixed (the energy does not
// depend on the overall scale of c)
__global__ void k_amsgrad(double* __restrict__ c, const double* __restrict__ g, double* __restrict__ m,
                          double* __restrict__ v, double* __restrict__ vh, long long nlab, double lr, double b1,
                          double b2, double eps) {
    for (long long l = 1 + (long long)blockIdx.x * blockDim.x + threadIdx.x; l < nlab; l += (long long)gridDim.x * blockDim.x) {
        const double gl = g[l];
        const double ml = b1 * m[l] + (1.0 - b1) * gl;
        const double vl = b2 * v[l] + (1.0 - b2) * gl * gl;
        const double vhl = fmax(vh[l], vl);
        m[l] = ml;
        v[l] = vl;
        vh[l] = vhl;
        c[l] -= lr * ml / (sqrt(vhl) + eps);
    }
}

// ============================================================================ fixed scratch for mrq_finalize_noalloc
//
// Partial sums of the finalize kernels for callers that cannot allocate device memory.  Every
// GPU that loads this library holds this array until the process exits.  All calls on a device
// share it: a call overwrites every slot it reads, and two calls whose kernels overlap on the
// GPU race on it.
static __device__ __align__(256) double g_noalloc_scratch[MRQ_NOALLOC_SCRATCH_DOUBLES];

#define MRQ_MAX_DEVICES 64
static double* g_noalloc_ptr[MRQ_MAX_DEVICES];     // device address of g_noalloc_scratch, per device
static std::mutex g_noalloc_mu;                    // guards g_noalloc_ptr (contexts may be created concurrently)

// device address of the fixed finalize scratch on `device` (current), looked up once per device
static double* noalloc_scratch_address(int device) {
    if (device < 0 || device >= MRQ_MAX_DEVICES) return nullptr;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (g_noalloc_ptr[device] == nullptr) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_noalloc_scratch) == cudaSuccess) g_noalloc_ptr[device] = (double*)p;
        else cudaGetLastError();
    }
    return g_noalloc_ptr[device];
}

// ============================================================================ host runtime

#define MRQ_MAX_SMEM (227 * 1024)      // dynamic shared memory of a block, at most

struct mrq_ctx {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    char err[1024] = {0};
    // Hamiltonian
    bool ham = false;
    int n = 0, nc = 0, na = 0, nv = 0, W = 1, nalpha = 0, nbeta = 0;
    double e_nuc = 0.0;
    long long neri = 0;
    double *d_h1 = nullptr, *d_eri = nullptr, *d_eri4 = nullptr, *d_tab = nullptr, *d_sgl = nullptr, *d_hc = nullptr,
           *d_eps = nullptr, *d_gamma = nullptr;
    unsigned short* d_colex = nullptr;
    size_t cap_h1 = 0, cap_eri = 0, cap_eri4 = 0, cap_tab = 0, cap_sgl = 0, cap_hc = 0, cap_eps = 0, cap_gamma = 0;   // bytes
    long long nHs = 0, nPs = 0, nlab = 0;
    // reference
    bool ref = false;
    long long nref = 0;
    HashSlot* d_hash = nullptr;
    unsigned char* d_setup = nullptr;   // the reference's determinants and coefficients and partial sums while it is set up
    size_t cap_hash = 0, cap_c = 0, cap_setup = 0;
    unsigned long long hcap = 0;
    unsigned long long start[4] = {0, 0, 0, 0};
    double start_c = 0.0;
    long long start_idx = 0;
    double e0 = 0, norm0 = 0, e_core = 0, sum_eps_core = 0;
    std::vector<double> eps, gamma;
    // coefficients
    double* d_c = nullptr;
    // walkers / accumulators
    Walker* d_walk = nullptr;
    long long nwalk = 0;
    size_t cap_walk = 0;             // (all cap_*: bytes of a kept buffer, 0 when there is none)
    int G = 0;
    long long burn = 0;
    unsigned long long seed = 0;
    double tau = 1e-10;
    double *d_accN = nullptr, *d_accU = nullptr, *d_accW = nullptr, *d_accE = nullptr;
    double *d_accA = nullptr, *d_accB = nullptr;        // SC-MRCI gradient sums [G][nlab]
    double *d_grad = nullptr, *d_am_m = nullptr, *d_am_v = nullptr, *d_am_vh = nullptr;   // AMSGrad state
    unsigned long long* d_types = nullptr;
    int* d_flist = nullptr;                             // visited labels of the finalize, by chunk, and their counts
    long long acc_lab = 0;
    int acc_G = 0;
    int* d_err = nullptr;                        // error flags; most CAS determinants of a step (WalkScratch::seen)
    int seen = 0;                                // the latter as last read (it sizes the workspace)
    Walker** d_wptr = nullptr;                   // this context's walk set: one walker array
    Walker* h_wset_ptr = nullptr;                // (host staging of the copies above)
    long long h_wset_off[2] = {0, 0};
    long long* d_woff = nullptr;
    // batch tables (a batch launched through this context as the first of its list)
    SysDev* d_bsys = nullptr;
    Walker** d_bwptr = nullptr;
    long long* d_boff = nullptr;
    size_t cap_bsys = 0, cap_bwptr = 0, cap_boff = 0;
    // workspace of this context's walk launches (WalkScratch), kept between calls
    unsigned char* d_work = nullptr;
    size_t work_cap = 0;
    long long work_limit = 1LL << 40;   // mrq_internal_work_limit
    long long row_worst = 0;         // doubles of one CAS determinant's rows when none is shared
    int fg_max = 1;                  // groups of a first-order determinant's neighbours (at most)
    WalkScratch work{};
    size_t ktab_bytes = 0;           // the table of known rows that was cleared last, and its counters
    int* kctl_at = nullptr;
    double* d_partial = nullptr;
    size_t cap_partial = 0;
    mrq_result* d_res = nullptr;
    SysDev hsys{};
    SysDev* d_sys = nullptr;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    cudaStream_t side[2] = {};       // side streams of a walk step, forked from and joined to `stream`
    cudaEvent_t ev_fork = nullptr, ev_prep = nullptr, ev_join[2] = {};
    // launch configuration (mrq_set_launch, mrq_tune_batch)
    int wpb = 0;                     // warps per walk block (0: MRQ_MAXNW)
    int max_nw = MRQ_MAXNW;          // most warps per block whose candidate lists fit shared memory
    int spl = 0;                     // steps per launch (0: every advance is one launch)
    int use_graph = 0;               // batches replay one reporting interval from a CUDA graph
    // everything a captured launch holds by value: the walk set, the workspace's layout and bounds, and the
    // launch shapes.  Compared and copied as bytes (made by graph_key, which clears the padding).
    struct GraphKey {
        const void *sys, *wptr, *off;
        long long nslots;
        int k, wpb, spl, cap, rows_minb, rows_blocks, frows_blocks, pad;
        WalkScratch work;
    };
    // per determinant width and warps per block (8, 4, 2, 1) of a batch launch
    static constexpr int NSLOT = 8;
    cudaGraphExec_t gexec[NSLOT] = {};
    GraphKey gkey[NSLOT] = {};
    int n_sm = 0;                    // SMs of the device
    long long graph_replays = 0;
    long long kernels = 0;           // kernels of walks and finalizes launched so far (mrq_kernel_launches)
    long long gkernels[NSLOT] = {};  // kernels of one replay of a graph
    long long* d_nbpre = nullptr;    // debug records: neighbour offsets of a determinant's units
    size_t cap_nbpre = 0;
    Walker* d_tune = nullptr;        // the tuner's scratch copy of a batch's walkers
    size_t cap_tune = 0;
    std::vector<cudaEvent_t> evs;    // start/stop pairs of the walk launches since the last finalize
    int launches = 0;
    long long launches_total = 0;
    double walk_ms = 0.0;
    long long total_steps = 0;
    // failure detection: host-wait deadline and lowered device bounds (mrq_set_deadline,
    // mrq_debug_set_limits)
    double deadline_s = 0.0;         // 0: host waits have no deadline
    cudaEvent_t ev_wait = nullptr;
    int probe_limit = 0, cap_limit = 0;
    int cand_cap_full = 1;           // the candidate-list capacity the loaded system needs
    double l2_fraction = 0.0;        // mrq_set_l2_window: share of the persisting-L2 carve-out for the tables
    int rows_minb = 2, rows_blocks = 0;   // k_rows: build in use (resident blocks per SM) and grid
    int frows_blocks = 0;            // k_frows' grid
};

static int fail(mrq_ctx* c, int code, const char* fmt, ...) {
    if (c) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(c->err, sizeof c->err, fmt, ap);
        va_end(ap);
    }
    return code;
}

#define CK(call)                                                                                      \
    do {                                                                                              \
        cudaError_t e_ = (call);                                                                      \
        if (e_ != cudaSuccess) {                                                                      \
            cudaGetLastError(); /* a failed allocation is not the next launch's error */              \
            return fail(ctx, e_ == cudaErrorMemoryAllocation ? MRQ_OOM : MRQ_CUDA_ERROR, "%s: %s (%s:%d)", \
                        #call, cudaGetErrorString(e_), __FILE__, __LINE__);                           \
        }                                                                                             \
    } while (0)

// Wait for the context stream.  With a deadline set (mrq_set_deadline) the wait polls an event
// and gives up with MRQ_DEVICE_TIMEOUT once the deadline passes; the device work keeps running
// and the next wait on this context waits for it again.
static int sync_stream(mrq_ctx* ctx) {
    if (!(ctx->deadline_s > 0.0) || ctx->ev_wait == nullptr) {
        CK(cudaStreamSynchronize(ctx->stream));
        return 0;
    }
    CK(cudaEventRecord(ctx->ev_wait, ctx->stream));
    const auto t0 = std::chrono::steady_clock::now();
    for (;;) {
        const cudaError_t e = cudaEventQuery(ctx->ev_wait);
        if (e == cudaSuccess) return 0;
        if (e != cudaErrorNotReady) return fail(ctx, MRQ_CUDA_ERROR, "cudaEventQuery: %s", cudaGetErrorString(e));
        const double dt = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
        if (dt > ctx->deadline_s)
            return fail(ctx, MRQ_DEVICE_TIMEOUT,
                        "device work did not finish within the %.6f s deadline; it keeps running and the next "
                        "call on this context waits for it", ctx->deadline_s);
        std::this_thread::sleep_for(std::chrono::microseconds(20));
    }
}

// Set-up calls wait for earlier work under the deadline, then run their own kernels and copies to
// the end without one (so a timeout never leaves a half-built table or a temporary buffer behind).
struct DeadlinePause {
    mrq_ctx* c;
    double d;
    explicit DeadlinePause(mrq_ctx* ctx) : c(ctx), d(ctx->deadline_s) { ctx->deadline_s = 0.0; }
    ~DeadlinePause() { c->deadline_s = d; }
};

template <typename T>
static void dfree(T*& p) {
    if (p) cudaFree((void*)p);
    p = nullptr;
}

// A device buffer of at least n elements: kept when it is that large already, so that a context that is
// loaded again (a geometry scan) allocates nothing
template <typename T>
static cudaError_t reserve(T*& p, size_t& cap, size_t n) {
    const bool fits = n <= SIZE_MAX / sizeof(T);
    if (p && fits && cap >= n * sizeof(T)) return cudaSuccess;
    dfree(p);
    cap = 0;
    if (!fits) return cudaErrorMemoryAllocation;
    const cudaError_t e = cudaMalloc(&p, n * sizeof(T));
    if (e == cudaSuccess) cap = n * sizeof(T);
    else p = nullptr;
    return e;
}

// Give the walk's workspace back, and with it the graphs captured on it (the caller has waited for the
// context's stream)
static void free_work(mrq_ctx* c) {
    for (int w = 0; w < mrq_ctx::NSLOT; w++) {
        if (c->gexec[w]) cudaGraphExecDestroy(c->gexec[w]);
        c->gexec[w] = nullptr;
    }
    dfree(c->d_work);
    c->work_cap = 0;
    c->ktab_bytes = 0;
}

static void free_reference(mrq_ctx* c) {
    dfree(c->d_hash);
    dfree(c->d_c);
    dfree(c->d_setup);
    c->cap_hash = c->cap_c = c->cap_setup = 0;
    c->ref = false;
}
static void free_accumulators(mrq_ctx* c) {
    dfree(c->d_accN);
    dfree(c->d_accU);
    dfree(c->d_accA);
    dfree(c->d_accB);
    dfree(c->d_accW);
    dfree(c->d_accE);
    dfree(c->d_types);
    dfree(c->d_flist);
    c->acc_lab = 0;
    c->acc_G = 0;
}

// Accumulators of G groups, all or none: a context whose allocation failed holds none and can be started again
static int alloc_accumulators(mrq_ctx* ctx, int G) {
    if (ctx->acc_lab == ctx->nlab && ctx->acc_G == G) return 0;
    free_accumulators(ctx);
    const size_t L = (size_t)ctx->nlab;
    const auto all = [&]() -> int {
        CK(cudaMalloc(&ctx->d_accN, sizeof(double) * L * G));
        CK(cudaMalloc(&ctx->d_accU, sizeof(double) * L * G));
        CK(cudaMalloc(&ctx->d_accA, sizeof(double) * L * G));
        CK(cudaMalloc(&ctx->d_accB, sizeof(double) * L * G));
        CK(cudaMalloc(&ctx->d_accW, sizeof(double) * G));
        CK(cudaMalloc(&ctx->d_accE, sizeof(double) * G));
        CK(cudaMalloc(&ctx->d_types, sizeof(unsigned long long) * MRQ_NTYPES));
        CK(cudaMalloc(&ctx->d_flist, sizeof(int) * (L + (size_t)((ctx->nlab + FIN_CHUNK - 1) / FIN_CHUNK))));
        return 0;
    };
    if (int r = all()) {
        free_accumulators(ctx);
        ctx->nwalk = 0;
        return r;
    }
    ctx->acc_lab = ctx->nlab;
    ctx->acc_G = G;
    return 0;
}

static void free_walkers(mrq_ctx* c) {
    dfree(c->d_walk);
    c->cap_walk = 0;
    c->nwalk = 0;
    free_accumulators(c);
    dfree(c->d_grad);
    dfree(c->d_am_m);
    dfree(c->d_am_v);
    dfree(c->d_am_vh);
    dfree(c->d_partial);
    c->cap_partial = 0;
}
static void free_hamiltonian(mrq_ctx* c) {
    dfree(c->d_h1);
    dfree(c->d_eri);
    dfree(c->d_eri4);
    dfree(c->d_tab);
    dfree(c->d_sgl);
    dfree(c->d_hc);
    dfree(c->d_eps);
    dfree(c->d_gamma);
    dfree(c->d_colex);
    c->cap_h1 = c->cap_eri = c->cap_eri4 = c->cap_tab = c->cap_sgl = c->cap_hc = c->cap_eps = c->cap_gamma = 0;
    c->ham = false;
}

static int push_sys(mrq_ctx* ctx) {
    SysDev& s = ctx->hsys;
    s.accN = ctx->d_accN;
    s.accU = ctx->d_accU;
    s.accA = ctx->d_accA;
    s.accB = ctx->d_accB;
    s.accW = ctx->d_accW;
    s.accE = ctx->d_accE;
    s.type_steps = ctx->d_types;
    s.G = ctx->G;
    s.burn_in = ctx->burn;
    s.seed = ctx->seed;
    s.err = ctx->d_err;
    s.c = ctx->d_c;
    s.hash = ctx->d_hash;
    s.hmask = ctx->hcap ? ctx->hcap - 1 : 0;
    s.e0 = ctx->e0;
    s.e_core = ctx->e_core;
    s.sum_eps_core = ctx->sum_eps_core;
    s.max_probe = ctx->probe_limit > 0 ? std::min(64, ctx->probe_limit) : 64;
    s.cand_cap = ctx->cap_limit > 0 ? std::min(ctx->cand_cap_full, ctx->cap_limit) : ctx->cand_cap_full;
    CK(cudaMemcpyAsync(ctx->d_sys, &s, sizeof(SysDev), cudaMemcpyHostToDevice, ctx->stream));
    return 0;
}

static int check_err_flag(mrq_ctx* ctx, int* flag_out) {
    int f[2] = {0, 0};
    if (int r = sync_stream(ctx)) return r;
    CK(cudaMemcpyAsync(f, ctx->d_err, sizeof f, cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));    // idle already: returns at once
    *flag_out = f[0];
    ctx->seen = f[1];
    return 0;
}

// The other contexts of a batch walk in its first one's workspace; where memory is short they give theirs back
// (their streams have been waited for).
struct WorkPeers {
    mrq_ctx* const* ctxs = nullptr;
    int n = 0;
};

// launch-time options of a walk: warps per block, whether to accumulate, and whether the one-time
// set-up (workspace growth, function attributes) has been done already (inside a stream capture)
struct WalkLaunch {
    int wpb = 8;
    int accumulate = 1;
    bool captured = false;
    WorkPeers peers;                     // (a batch's contexts)
    cudaAccessPolicyWindow l2win = {};   // num_bytes 0: no persisting-L2 window
};

// what a walk set's systems need: the largest candidate-list capacity, single-excitation operator and
// slice count among them
struct WalkNeed {
    int cap = 1, gstride = 0, ns = MRQ_FOIS_SLICES, nref = 1, fg_max = 1;
    long long row_worst = 1, fois_nb = 1;
    long long ncas = 0;              // CAS determinants with walkers, at most: those of the references (psi_s is 0 on others)
    void add(const mrq_ctx* c) {
        const SysDev& s = c->hsys;
        ncas += c->nref;
        nref = std::max(nref, s.ref_off[8]);
        row_worst = std::max(row_worst, c->row_worst);
        fg_max = std::max(fg_max, c->fg_max);
        fois_nb = std::max(fois_nb, s.cas_nb_total + 4);
        cap = std::max(cap, s.cand_cap);
        gstride = std::max(gstride, s.gstride);
        ns = std::max(ns, s.nslice);
    }
};

// Workspace of a launch over nslots walkers.  A launch takes its walkers in segments, and a segment's
// determinants in waves, so that the workspace stays within bounds whatever the number of walkers: a segment's
// arrays hold one entry per walker, a wave's row buffer the worst case that none of its determinants share a row.
// Walkers crowd (56 orbitals: 4,096 walkers on 640 CAS determinants), so a wave starts at a third of the walkers, or
// whatever MRQ_ROW_START holds, and grows in steps of a half to 1.5 times the most CAS determinants that a step of
// this context has had.  (Steps, since a count that creeps up would make it anew again and again: 2 % of the time of a
// running 56-orbital walk.  One determinant for every walker: 8 GiB of rows there instead of 4, and no faster.)
// A workspace takes at most an eighth of the memory that is free when it is made, so that other contexts and
// libraries find room; where that or a lowered limit is less, waves and segments shrink.
#define MRQ_WORK_BYTES (1LL << 30)
#define MRQ_ROW_BYTES (8LL << 30)
#define MRQ_ROW_START (2LL << 30)
#define MRQ_FROW_BYTES (2LL << 30)

// sizes of a workspace and the places of its arrays
struct WorkPlan {
    long long seg, groups, fwave, tsz;
    bool least;                      // the floor: 256 walkers per segment, one determinant per wave
    size_t rep, cnt, start, tab, pos, mem, tgc, tgf, meta, gops, part, best, bound, ctl, ao, cls, rrep, roff, tbl, ul, kt, kao, kkey,
        koff, kctl, fgo, fg, rows, frows, nul, bytes;
};

static WorkPlan work_layout(const WalkNeed& need, long long seg, long long groups, long long fwave) {
    WorkPlan p{};
    p.seg = seg;
    p.groups = groups;
    p.fwave = fwave;
    p.tsz = 2;
    while (p.tsz < 2 * groups * need.nref) p.tsz <<= 1;      // (as many known rows as references of a wave)
    auto take = [&](size_t bytes) {
        const size_t at = p.bytes;
        p.bytes += (bytes + 255) / 256 * 256;
        return at;
    };
    const size_t nr = (size_t)groups * need.nref;
    p.nul = nr + (size_t)(need.row_worst * groups / MRQ_BIG_ROW) + 1;
    p.rep = take(16 * seg);
    p.cnt = take(16 * seg);
    p.start = take(16 * seg);
    p.tab = take(4 * seg);
    p.pos = take(4 * seg);
    p.mem = take(4 * seg);
    p.tgc = take(sizeof(TaskGroup) * seg);
    p.tgf = take(sizeof(TaskGroup) * seg);
    p.meta = take(sizeof(GroupMeta) * seg);
    p.gops = take(8 * (size_t)need.gstride * seg);
    p.part = take(24 * (size_t)(need.ns + MRQ_ACT_SLICES) * seg);
    p.best = take(sizeof(RaceBest) * seg);
    p.bound = take(4 * seg);
    p.ctl = take(4 * CTL_N);
    p.ao = take(8 * nr);
    p.cls = take(nr);
    p.rrep = take(4 * nr);
    p.roff = take(8 * nr);
    p.tbl = take(4 * p.tsz);
    p.ul = take(sizeof(int2) * p.nul);
    p.kt = take(8 * p.tsz);
    p.kao = take(8 * nr);
    p.kkey = take(4 * nr);
    p.koff = take(8 * nr);
    p.kctl = take(4 * KNOWN_N);
    p.fgo = take(8 * fwave);
    p.fg = take(sizeof(FGroup) * (size_t)need.fg_max * fwave);
    p.rows = take(8 * (size_t)need.row_worst * groups);
    p.frows = take(8 * (size_t)need.fois_nb * fwave);
    return p;
}

// the workspace for nslots walkers within `limit` bytes (or the floor); seen: the most CAS determinants of a step
// so far
static WorkPlan work_size(long long nslots, const WalkNeed& need, int seen, long long limit) {
    const long long per = 12 * 4 + 3 * 4 + 2 * (long long)sizeof(TaskGroup) + (long long)sizeof(GroupMeta) +
                          8LL * need.gstride + 24LL * (need.ns + MRQ_ACT_SLICES) + (long long)sizeof(RaceBest) + 4;
    const long long per_group = 8 * need.row_worst + 93LL * need.nref;
    const long long per_fois = 8 * need.fois_nb + (long long)sizeof(FGroup) * need.fg_max + 8;
    const long long seg0 = std::min(256LL, nslots);
    long long seg = std::min(nslots, std::max(seg0, std::min(1LL << 20, std::min(MRQ_WORK_BYTES, limit / 5) / per)));
    long long groups = std::max({1LL, MRQ_ROW_START / per_group, (seg + 2) / 3});
    while (2 * groups < 3LL * seen) groups += (groups + 1) / 2;
    groups = std::min({groups, seg, need.ncas, std::min(MRQ_ROW_BYTES, limit / 5 * 3) / per_group,
                       (1LL << 29) / need.nref});                                  // (reference indices and the table: 32 bits)
    long long fwave = std::min(MRQ_FROW_BYTES, limit / 5) / per_fois;
    fwave = std::min({fwave, seg, (1LL << 30) / need.fg_max});                     // (group indices: 32 bits)
    groups = std::max(1LL, groups);
    fwave = std::max(1LL, fwave);
    for (;;) {
        WorkPlan p = work_layout(need, seg, groups, fwave);
        p.least = groups == 1 && fwave == 1 && seg == seg0;
        if ((long long)p.bytes <= limit || p.least) return p;
        groups = std::max(1LL, groups * 7 / 8);
        fwave = std::max(1LL, fwave * 7 / 8);
        seg = std::max(seg0, seg * 7 / 8);
    }
}

static int work_prepare(mrq_ctx* ctx, long long nslots, const WalkNeed& need, const WorkPeers& peers) {
    const long long limit = ctx->work_limit;
    WorkPlan p = work_size(nslots, need, ctx->seen, limit);
    const auto renew = [&]() { return p.bytes > ctx->work_cap || ((long long)ctx->work_cap > limit && p.bytes < ctx->work_cap); };
    if (renew()) {
        size_t free_b = 0, total_b = 0;
        CK(cudaMemGetInfo(&free_b, &total_b));
        long long room = (long long)((free_b + ctx->work_cap) / 8);
        if ((long long)p.bytes > room) {
            for (int i = 0; i < peers.n; i++) {
                if (peers.ctxs[i] == ctx) continue;
                free_b += peers.ctxs[i]->work_cap;
                free_work(peers.ctxs[i]);
            }
            room = (long long)((free_b + ctx->work_cap) / 8);
        }
        if (room < limit) {
            // (one that is nearly as large stays)
            if ((long long)ctx->work_cap <= limit && (long long)ctx->work_cap >= room - room / 4) room = (long long)ctx->work_cap;
            p = work_size(nslots, need, ctx->seen, room);
        }
        if (renew()) {
            if (int r = sync_stream(ctx)) return r;
            free_work(ctx);
            for (;;) {
                const cudaError_t e = cudaMalloc(&ctx->d_work, p.bytes);
                if (e == cudaSuccess) break;
                ctx->d_work = nullptr;
                if (e != cudaErrorMemoryAllocation || p.least) CK(e);
                cudaGetLastError();
                p = work_size(nslots, need, ctx->seen, (long long)(p.bytes / 2));
            }
            ctx->work_cap = p.bytes;
        }
    }
    unsigned char* const b = ctx->d_work;
    WalkScratch& w = ctx->work;
    w.rep = (int*)(b + p.rep);
    w.cnt = (int*)(b + p.cnt);
    w.start = (int*)(b + p.start);
    w.tab_of = (int*)(b + p.tab);
    w.pos_of = (int*)(b + p.pos);
    w.members = (int*)(b + p.mem);
    w.tgc = (TaskGroup*)(b + p.tgc);
    w.tgf = (TaskGroup*)(b + p.tgf);
    w.meta = (GroupMeta*)(b + p.meta);
    w.gops = (double*)(b + p.gops);
    w.part = (double*)(b + p.part);
    w.best = (RaceBest*)(b + p.best);
    w.bound = (unsigned*)(b + p.bound);
    w.ctl = (int*)(b + p.ctl);
    w.seen = ctx->d_err + 1;
    w.ref_ao = (unsigned long long*)(b + p.ao);
    w.ref_cls = b + p.cls;
    w.ref_rep = (int*)(b + p.rrep);
    w.row_off = (long long*)(b + p.roff);
    w.table = (int*)(b + p.tbl);
    w.ulist = (int2*)(b + p.ul);
    w.ulist_size = (int)p.nul;
    w.rows = (double*)(b + p.rows);
    w.frows = (double*)(b + p.frows);
    w.table_size = (int)p.tsz;
    w.ktab_size = (int)p.tsz;
    w.k_ao = (unsigned long long*)(b + p.kao);
    w.k_key = (int*)(b + p.kkey);
    w.k_off = (long long*)(b + p.koff);
    w.kctl = (int*)(b + p.kctl);
    // a new layout of the workspace: nothing in it is a table of known rows yet
    if (w.ktab != (unsigned long long*)(b + p.kt) || ctx->ktab_bytes != 8 * (size_t)p.tsz || ctx->kctl_at != w.kctl) {
        w.ktab = (unsigned long long*)(b + p.kt);
        ctx->ktab_bytes = 8 * (size_t)p.tsz;
        ctx->kctl_at = w.kctl;
        CK(cudaMemsetAsync(w.ktab, 0, ctx->ktab_bytes, ctx->stream));
        CK(cudaMemsetAsync(w.kctl, 0, sizeof(int) * KNOWN_N, ctx->stream));
    }
    w.fg_of = (int2*)(b + p.fgo);
    w.fg = (FGroup*)(b + p.fg);
    w.nref_max = need.nref;
    w.row_worst = need.row_worst;
    w.wave_groups = (int)p.groups;
    w.wave0 = 0;
    w.fg_max = need.fg_max;
    w.fwave = (int)p.fwave;
    w.fwave0 = 0;
    w.gstride = need.gstride;
    w.ns_max = need.ns;
    w.nseg = p.seg;
    // walkers per task group: 32 when there are many, fewer for small launches, so that the walkers of
    // a crowded determinant spread over more warps (against the determinant's neighbours being formed once
    // per group)
    w.tgw = (int)std::max(4LL, std::min<long long>(p.seg <= 2048 ? 16 : MRQ_TGW, p.seg <= 2048 ? p.seg / 64 : p.seg / 128));
    return 0;
}

// (a kernel's limit is the process's, so it is always set to the most a block may have: contexts on other
// threads launch with other sizes)
template <int W, int B>
static int rows_fits(mrq_ctx* ctx, size_t smem, int threads, int& blocks) {
    CK(cudaFuncSetAttribute(k_rows<W, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, MRQ_MAX_SMEM));
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, k_rows<W, B>, threads, smem));
    return 0;
}

// k_rows' build for this launch: the most resident warps per SM (4 or 2 blocks' worth of MRQ_MAXNW warps)
// that the candidate lists in shared memory allow, and a grid that fills the chip once
static int rows_prepare(mrq_ctx* ctx, int W, int nw, int cap) {
    const size_t smem = nw * rows_warp_bytes(cap);
    const size_t fsm = nw * frows_warp_bytes(cap);
    int b4 = 0, b2 = 0, bf = 0;
    if (W == 1) {
        if (int r = rows_fits<1, 4>(ctx, smem, 32 * nw, b4)) return r;
        if (int r = rows_fits<1, 2>(ctx, smem, 32 * nw, b2)) return r;
        CK(cudaFuncSetAttribute(k_move<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, MRQ_MAX_SMEM));
        CK(cudaFuncSetAttribute(k_frows<1, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, MRQ_MAX_SMEM));
        CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bf, k_frows<1, 3>, 32 * nw, fsm));
    } else {
        if (int r = rows_fits<2, 4>(ctx, smem, 32 * nw, b4)) return r;
        if (int r = rows_fits<2, 2>(ctx, smem, 32 * nw, b2)) return r;
        CK(cudaFuncSetAttribute(k_move<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, MRQ_MAX_SMEM));
        CK(cudaFuncSetAttribute(k_frows<2, 3>, cudaFuncAttributeMaxDynamicSharedMemorySize, MRQ_MAX_SMEM));
        CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bf, k_frows<2, 3>, 32 * nw, fsm));
    }
    ctx->rows_minb = b4 > b2 ? 4 : 2;
    ctx->rows_blocks = std::max(1, std::max(b4, b2)) * ctx->n_sm;
    ctx->frows_blocks = std::max(1, bf) * ctx->n_sm;
    return 0;
}

// warps per block of a context's k_rows and k_move launches: the requested (or default) number, at most
// the most whose candidate lists fit shared memory (large active spaces run with fewer warps)
static int warps_of(const mrq_ctx* ctx) { return std::min(ctx->wpb > 0 ? ctx->wpb : MRQ_MAXNW, ctx->max_nw); }

template <int W>
static int launch_segment(mrq_ctx* ctx, const WalkSet& ws, WalkScratch sc, const WalkNeed& need, int nw, int accumulate,
                          cudaLaunchConfig_t cfg) {
    const long long n = sc.seg1 - sc.seg0;
    const int sms = ctx->n_sm;
    const cudaStream_t st = ctx->stream;
    const size_t lbytes = cand_list_bytes(need.cap), rbytes = rows_warp_bytes(need.cap), fbytes = frows_warp_bytes(need.cap);
    const cudaStream_t st2 = ctx->side[0], st3 = ctx->side[1];
    ctx->kernels += 5;                // k_group, k_prep, k_int, k_fois_act, k_move; the waves' are added below
    if (ws.nsys > 1) CK(cudaMemsetAsync(sc.ctl, 0, sizeof(int) * CTL_N, st));
    k_group<W><<<(unsigned)ws.nsys, 1024, 0, st>>>(ws, sc);
    CK(cudaEventRecord(ctx->ev_fork, st));
    // first side stream: the determinants' constants, the neighbours inside the CAS, the active-only ones of
    // first-order determinants
    CK(cudaStreamWaitEvent(st2, ctx->ev_fork, 0));
    k_prep<W><<<(unsigned)std::min<long long>(n, 8LL * sms), 128, 0, st2>>>(ws, sc);
    CK(cudaEventRecord(ctx->ev_prep, st2));
    k_int<W><<<(unsigned)std::min<long long>(n, 3LL * sms), 256, 0, st2>>>(ws, sc);
    k_fois_act<W><<<(unsigned)std::min<long long>(4 * n, 3LL * sms), 256, 0, st2>>>(ws, sc);
    CK(cudaEventRecord(ctx->ev_join[0], st2));
    // second side stream: the other neighbours of first-order determinants
    CK(cudaStreamWaitEvent(st3, ctx->ev_fork, 0));
    for (long long g = 0; g < n; g += sc.fwave) {
        sc.fwave0 = (int)g;
        ctx->kernels += 3;
        if (g > 0) CK(cudaMemsetAsync(sc.ctl + CTL_FOIS, 0, sizeof(int) * (CTL_N - CTL_FOIS), st3));
        k_fgroups<W><<<(unsigned)std::min<long long>(n, 4LL * sms), 256, 0, st3>>>(ws, sc);
        k_frows<W, 3><<<(unsigned)ctx->frows_blocks, 32 * nw, nw * fbytes, st3>>>(ws, sc, (int)fbytes, need.cap);
        if (g == 0) CK(cudaStreamWaitEvent(st3, ctx->ev_prep, 0));
        k_fois<W, 3><<<3 * sms, 256, 0, st3>>>(ws, sc);
    }
    CK(cudaEventRecord(ctx->ev_join[1], st3));
    // main stream: the CAS determinants' rows and pairs
    for (long long g = 0; g < std::min(n, need.ncas); g += sc.wave_groups) {
        sc.wave0 = (int)g;
        ctx->kernels += 5;
        k_wave_begin<<<1, 1, 0, st>>>(sc);
        k_refs<W><<<(unsigned)std::min<long long>(n, 8LL * sms), 256, 0, st>>>(ws, sc);
        k_insert<<<8 * sms, 256, 0, st>>>(ws, sc);
        cfg.gridDim = dim3((unsigned)ctx->rows_blocks);
        cfg.blockDim = dim3(32 * nw);
        cfg.dynamicSmemBytes = nw * rbytes;
        if (ctx->rows_minb == 4) CK(cudaLaunchKernelEx(&cfg, k_rows<W, 4>, ws, sc, (int)rbytes, need.cap));
        else CK(cudaLaunchKernelEx(&cfg, k_rows<W, 2>, ws, sc, (int)rbytes, need.cap));
        if (g == 0) CK(cudaStreamWaitEvent(st, ctx->ev_prep, 0));
        cfg.gridDim = dim3(4u * sms);
        cfg.blockDim = dim3(256);
        cfg.dynamicSmemBytes = 0;
        CK(cudaLaunchKernelEx(&cfg, k_pairs<W, 4>, ws, sc));
    }
    for (int k = 0; k < 2; k++) CK(cudaStreamWaitEvent(st, ctx->ev_join[k], 0));
    k_move<W><<<(unsigned)std::min<long long>((n + nw - 1) / nw, 4LL * sms), 32 * nw, nw * lbytes, st>>>(
        ws, sc, accumulate, (int)lbytes, need.cap);
    CK(cudaGetLastError());
    return 0;
}

// nsteps walker steps of a walk set (the kernels of mrq_walk.cuh per step); `ctx` provides the stream
// and the workspace.
static int launch_walk(mrq_ctx* ctx, int W, const WalkSet& ws, int nsteps, const WalkNeed& need,
                       const WalkLaunch& L = WalkLaunch()) {
    const int nw = std::min(L.wpb, MRQ_MAXNW);
    if (!L.captured) {
        if (int r = work_prepare(ctx, ws.nslots, need, L.peers)) return r;
        if (int r = rows_prepare(ctx, W, nw, need.cap)) return r;
    }
    const long long seg = ctx->work.nseg;
    cudaLaunchConfig_t cfg = {};
    cfg.stream = ctx->stream;
    cudaLaunchAttribute attr[1];
    if (L.l2win.num_bytes > 0) {            // keep the walk's hottest table resident in L2
        attr[0].id = cudaLaunchAttributeAccessPolicyWindow;
        attr[0].val.accessPolicyWindow = L.l2win;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    k_rows_begin<<<1, 1, 0, ctx->stream>>>(ctx->work);
    CK(cudaGetLastError());
    ctx->kernels++;
    for (int step = 0; step < nsteps; step++) {
        for (long long s0 = 0; s0 < ws.nslots; s0 += seg) {
            WalkScratch sc = ctx->work;
            sc.seg0 = s0;
            sc.seg1 = std::min(ws.nslots, s0 + seg);
            if (int r = W == 1 ? launch_segment<1>(ctx, ws, sc, need, nw, L.accumulate, cfg)
                               : launch_segment<2>(ctx, ws, sc, need, nw, L.accumulate, cfg))
                return r;
        }
        if (L.accumulate) {
            k_accum<<<dim3((unsigned)ws.nsys, 2), 1024, 0, ctx->stream>>>(ws);
            CK(cudaGetLastError());
            ctx->kernels++;
        }
    }
    return 0;
}

// ---------------------------------------------------------------- work plan of the walk (host)

static long long nsub_h(long long k, int size) {
    if (size < 0 || k < size) return 0;
    return size == 0 ? 1 : (size == 1 ? k : k * (k - 1) / 2);
}
static long long shape_h(long long m, int cnt, int nal) {
    if (cnt == 0) return 1;
    if (cnt == 1) return m;
    return nal == 1 ? m * m : m * (m - 1) / 2;
}
// neighbours of one (X_a, Y_a) pair of a CAS walker with alpha(Y_a) - alpha(X_a) = d
static long long pair_total_h(int nc, int nv, int ka, int kb, int d) {
    long long tot = 0;
    for (int r = std::max(1, std::max(ka, kb)); r <= 2; r++) {
        const int c = r - ka, v = r - kb;
        if (c == 0 && v == 0) continue;
        for (int sc = 0; sc <= c; sc++) {
            const int sv = sc - d;
            if (sv < 0 || sv > v) continue;
            tot += shape_h(nc, c, sc) * shape_h(nv, v, sv);
        }
    }
    return tot;
}

// The CAS walkers' work units (the same for every CAS determinant: all hold n_alpha - n_core alpha
// and n_beta - n_core beta active electrons), the largest candidate list of a group (spin-resolved:
// the alpha count of R' fixes that of A'), and the walk block's shared memory.
static int walk_plan(mrq_ctx* ctx, SysDev& s) {
    const int nc = s.nc, na = s.na, nv = s.nv;
    const int nao = s.nalpha - nc, nbo = s.nbeta - nc, cea = na - nao, ceb = na - nbo;
    const int cntO = nao + nbo, cntE = cea + ceb;
    long long cas_nb = nao * (long long)cea + nbo * (long long)ceb + nsub_h(nao, 2) * nsub_h(cea, 2) +
                       nsub_h(nbo, 2) * nsub_h(ceb, 2) + (long long)nao * cea * nbo * ceb;
    long long total = cas_nb;
    long long off = (cas_nb + MRQ_CAS_CH - 1) / MRQ_CAS_CH;
    s.cas_nb = (int)cas_nb;
    s.cas_units = (int)off;
    long long nref = 0;
    for (int k = 0; k < 8; k++) {
        const int ka = k / 3, kb = k % 3;
        const long long npairs = nsub_h(cntO, ka) * nsub_h(cntE, kb);
        long long maxN = 0;
        for (int xal = 0; xal <= ka; xal++)
            for (int yal = 0; yal <= kb; yal++) {
                const long long nx = nsub_h(nao, xal) * nsub_h(nbo, ka - xal);
                const long long ny = nsub_h(cea, yal) * nsub_h(ceb, kb - yal);
                if (nx == 0 || ny == 0) continue;
                const long long N = pair_total_h(nc, nv, ka, kb, yal - xal);
                total += nx * ny * N;
                maxN = std::max(maxN, N);
            }
        const long long nch = std::max(1LL, (maxN + MRQ_UNIT_NB - 1) / MRQ_UNIT_NB);
        s.nch[k] = (int)nch;
        s.unit_off[k] = (int)off;
        off += npairs * nch;
        s.ref_off[k] = (int)nref;
        nref += npairs * (ka + kb == 1 ? 2 : 1);
    }
    s.unit_off[8] = (int)off;
    s.ref_off[8] = (int)nref;
    ctx->row_worst = total - cas_nb + 4 * nref;
    // slices of a determinant's units: about four units each, so that a step on a few hundred
    // determinants is some 10^5 warp tasks and one on a few still spreads over the chip
    s.nslice = 128;
    while (s.nslice < MRQ_NS_MAX && s.nslice * 4 < off) s.nslice <<= 1;
    s.cas_nb_total = total;
    // Groups of a first-order determinant's neighbours: the outer patterns of a pair (X_a, Y_a) of each
    // class, at most (electrons removed: kinds of the virtual ones x alpha core ones; likewise added),
    // for any number of active electrons the determinant may have, and the cuts of long groups.  (A
    // determinant has as many singles and doubles in all as a CAS determinant.)
    {
        static const long long per[8] = {66, 45, 12, 45, 18, 6, 12, 6};
        long long most = 0;
        for (int o = std::max(0, cntO - 2); o <= std::min(2 * na, cntO + 2); o++) {
            long long g = 0;
            for (int k = 0; k < 8; k++) g += nsub_h(o, k / 3) * nsub_h(2 * na - o, k % 3) * per[k];
            most = std::max(most, g);
        }
        most += total / MRQ_FG_NB + 1;
        if (most > (1LL << 28)) return fail(ctx, MRQ_TOO_LARGE, "active space too large for the walk's work plan");
        ctx->fg_max = (int)most;
    }
    if (off > (1LL << 30) || total > (1LL << 40))
        return fail(ctx, MRQ_TOO_LARGE, "active space too large for the walk's work plan");
    // largest candidate list: m's active occupation differs from n's by at most two electrons
    long long cap = 1;
    for (int oa = std::max(0, nao - 2); oa <= std::min(na, nao + 2); oa++)
        for (int ob = std::max(0, nbo - 2); ob <= std::min(na, nbo + 2); ob++) {
            if (std::abs(oa + ob - cntO) > 2) continue;
            const int ea = na - oa, eb = na - ob;
            for (int c = 0; c <= 2; c++)
                for (int v = 0; v <= 2; v++) {
                    if (c == 0 && v == 0) continue;
                    for (int sc = 0; sc <= c; sc++)
                        for (int sv = 0; sv <= v; sv++) {
                            long long t = 0;
                            for (int rr = 1; rr <= 2; rr++) {
                                if (rr == 1 && (c > 1 || v > 1)) continue;
                                const int ne = rr - v, nf = rr - c;
                                if (ne < 0 || nf < 0) continue;
                                for (int i = 0; i <= ne; i++) {
                                    const int j = i + sv - sc;
                                    if (j < 0 || j > nf) continue;
                                    t += nsub_h(oa, i) * nsub_h(ob, ne - i) * nsub_h(ea, j) * nsub_h(eb, nf - j);
                                }
                            }
                            cap = std::max(cap, t);
                        }
                }
        }
    s.gstride = 2 * s.nca * s.nav;
    s.cand_cap = (int)cap;
    ctx->cand_cap_full = (int)cap;
    // the most warps per block (8, 4, 2 or 1) whose candidate lists fit its shared memory; beyond one
    // warp the active space is too large for the walk
    ctx->max_nw = 0;
    for (int nw = MRQ_MAXNW; nw >= 1 && ctx->max_nw == 0; nw >>= 1)
        if (debug_smem_bytes(nw, (int)cap, s.gstride) <= MRQ_MAX_SMEM && nw * frows_warp_bytes((int)cap) <= MRQ_MAX_SMEM)
            ctx->max_nw = nw;
    if (ctx->max_nw == 0)
        return fail(ctx, MRQ_TOO_LARGE, "active space too large for the shared-memory candidate lists");
    return 0;
}

// The persisting-L2 window of a walk launch (mrq_set_l2_window): the physicists' tables, which
// every reach-back term reads, marked persisting up to the device's carve-out (the carve-out is a
// per-process limit of this CUDA context and ends with it).
static int l2_window(mrq_ctx* ctx, cudaAccessPolicyWindow& w) {
    w = cudaAccessPolicyWindow{};
    if (!(ctx->l2_fraction > 0.0) || !ctx->d_tab) return 0;
    int maxwin = 0, maxpersist = 0;
    CK(cudaDeviceGetAttribute(&maxwin, cudaDevAttrMaxAccessPolicyWindowSize, ctx->device));
    CK(cudaDeviceGetAttribute(&maxpersist, cudaDevAttrMaxPersistingL2CacheSize, ctx->device));
    if (maxwin <= 0 || maxpersist <= 0) return 0;
    const size_t tab_bytes = sizeof(double) * 2 * (size_t)ctx->hsys.tab_half;
    const size_t carve = (size_t)(ctx->l2_fraction * (double)maxpersist);
    CK(cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, carve));
    w.base_ptr = ctx->d_tab;
    w.num_bytes = std::min(tab_bytes, (size_t)maxwin);
    w.hitRatio = (float)std::min(1.0, (double)carve / (double)w.num_bytes);
    w.hitProp = cudaAccessPropertyPersisting;
    w.missProp = cudaAccessPropertyStreaming;
    return 0;
}

// Load the code of every kernel of a walk on the current device, once.  A step runs on three streams, and the runtime
// otherwise uploads a kernel's code at its first launch, beside kernels of the other streams that are running.
template <int W>
static cudaError_t load_walk_kernels() {
    const void* const kernels[] = {
        (const void*)k_group<W>, (const void*)k_prep<W>, (const void*)k_int<W>, (const void*)k_fois_act<W>,
        (const void*)k_fgroups<W>, (const void*)k_frows<W, 3>, (const void*)k_fois<W, 3>, (const void*)k_refs<W>,
        (const void*)k_rows<W, 2>, (const void*)k_rows<W, 4>, (const void*)k_pairs<W, 4>, (const void*)k_move<W>,
        (const void*)k_rows_begin, (const void*)k_wave_begin, (const void*)k_insert, (const void*)k_accum,
        (const void*)k_fin_list, (const void*)k_fin_labels, (const void*)k_fin_reduce, (const void*)k_walkers_init};
    for (const void* k : kernels) {
        cudaFuncAttributes a;
        const cudaError_t e = cudaFuncGetAttributes(&a, k);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

static cudaError_t load_kernels(int device) {
    static std::mutex mu;
    static bool done[MRQ_MAX_DEVICES];
    std::lock_guard<std::mutex> lock(mu);
    if (device >= 0 && device < MRQ_MAX_DEVICES && done[device]) return cudaSuccess;
    cudaError_t e = load_walk_kernels<1>();
    if (e == cudaSuccess) e = load_walk_kernels<2>();
    if (e == cudaSuccess && device >= 0 && device < MRQ_MAX_DEVICES) done[device] = true;
    return e;
}

extern "C" {

int mrq_create(mrq_ctx** out, int device) {
    if (!out) return MRQ_INVALID_ARG;
    *out = nullptr;
    mrq_ctx* ctx = new mrq_ctx();
    ctx->device = device;
    cudaError_t e = cudaSetDevice(device);
    if (e != cudaSuccess) {
        delete ctx;
        return MRQ_CUDA_ERROR;
    }
    if (cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking) != cudaSuccess ||
        cudaMalloc(&ctx->d_err, 2 * sizeof(int)) != cudaSuccess || cudaMalloc(&ctx->d_sys, sizeof(SysDev)) != cudaSuccess ||
        cudaMalloc(&ctx->d_res, sizeof(mrq_result)) != cudaSuccess || cudaEventCreate(&ctx->ev0) != cudaSuccess ||
        cudaEventCreate(&ctx->ev1) != cudaSuccess ||
        cudaStreamCreateWithFlags(&ctx->side[0], cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamCreateWithFlags(&ctx->side[1], cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&ctx->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&ctx->ev_prep, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&ctx->ev_join[0], cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&ctx->ev_join[1], cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&ctx->ev_wait, cudaEventDisableTiming) != cudaSuccess) {
        mrq_destroy(ctx);
        return MRQ_CUDA_ERROR;
    }
    ctx->own_stream = true;
    cudaMemset(ctx->d_err, 0, 2 * sizeof(int));
    if (cudaDeviceGetAttribute(&ctx->n_sm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
        load_kernels(device) != cudaSuccess) {
        mrq_destroy(ctx);
        return MRQ_CUDA_ERROR;
    }
    // set-up of the allocation-free finalize: the device address of the fixed scratch array,
    // looked up once per device with that device current (host code cannot use the symbol itself)
    noalloc_scratch_address(device);
    *out = ctx;
    return 0;
}

void mrq_destroy(mrq_ctx* ctx) {
    if (!ctx) return;
    cudaSetDevice(ctx->device);
    if (ctx->stream) cudaStreamSynchronize(ctx->stream);
    free_walkers(ctx);
    free_reference(ctx);
    free_hamiltonian(ctx);
    dfree(ctx->d_err);
    dfree(ctx->d_sys);
    dfree(ctx->d_res);
    free_work(ctx);
    dfree(ctx->d_wptr);
    dfree(ctx->d_woff);
    dfree(ctx->d_bsys);
    dfree(ctx->d_bwptr);
    dfree(ctx->d_boff);
    dfree(ctx->d_tune);
    dfree(ctx->d_nbpre);
    for (auto e : ctx->evs) cudaEventDestroy(e);
    if (ctx->ev0) cudaEventDestroy(ctx->ev0);
    if (ctx->ev1) cudaEventDestroy(ctx->ev1);
    if (ctx->ev_wait) cudaEventDestroy(ctx->ev_wait);
    if (ctx->ev_fork) cudaEventDestroy(ctx->ev_fork);
    if (ctx->ev_prep) cudaEventDestroy(ctx->ev_prep);
    for (int k = 0; k < 2; k++) {
        if (ctx->ev_join[k]) cudaEventDestroy(ctx->ev_join[k]);
        if (ctx->side[k]) cudaStreamDestroy(ctx->side[k]);
    }
    if (ctx->own_stream && ctx->stream) cudaStreamDestroy(ctx->stream);
    delete ctx;
}

const char* mrq_last_error(const mrq_ctx* ctx) { return ctx ? ctx->err : "null context"; }

int mrq_set_stream(mrq_ctx* ctx, void* stream) {
    if (!ctx) return MRQ_INVALID_ARG;
    CK(cudaSetDevice(ctx->device));
    if (int r_ = sync_stream(ctx)) return r_;
    if (stream) {
        if (ctx->own_stream) cudaStreamDestroy(ctx->stream);
        ctx->stream = (cudaStream_t)stream;
        ctx->own_stream = false;
    } else if (!ctx->own_stream) {
        CK(cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking));
        ctx->own_stream = true;
    }
    return 0;
}

int64_t mrq_n_labels(const mrq_ctx* ctx) { return (ctx && ctx->ham) ? ctx->nlab : 0; }

int mrq_load_hamiltonian(mrq_ctx* ctx, int n_core, int n_act, int n_virt, int n_alpha, int n_beta, const double* h1,
                         const double* eri, double e_core) {
    if (!ctx) return MRQ_INVALID_ARG;
    ctx->err[0] = 0;
    const int n = n_core + n_act + n_virt;
    if (n_core < 0 || n_act < 0 || n_virt < 0 || n <= 0 || n > MRQ_MAXN || n_core > 64 || n_act > 32 || !h1 ||
        !eri)
        return fail(ctx, MRQ_INVALID_ARG, "orbital counts out of range (n <= 128, n_core <= 64, n_act <= 32)");
    if (n_alpha < n_core || n_beta < n_core || n_alpha > n_core + n_act || n_beta > n_core + n_act)
        return fail(ctx, MRQ_INVALID_ARG, "electron counts must fill the core and fit the active space");
    CK(cudaSetDevice(ctx->device));
    if (int r_ = sync_stream(ctx)) return r_;
    DeadlinePause pause_(ctx);
    free_walkers(ctx);
    free_work(ctx);                   // the walk workspace of the last system is given back
    CK(cudaMemsetAsync(ctx->d_err, 0, 2 * sizeof(int), ctx->stream));
    ctx->seen = 0;
    ctx->ref = ctx->ham = false;
    ctx->n = n;
    ctx->nc = n_core;
    ctx->na = n_act;
    ctx->nv = n_virt;
    ctx->W = (n + 63) / 64;
    ctx->nalpha = n_alpha;
    ctx->nbeta = n_beta;
    ctx->e_nuc = e_core;
    const long long npair = (long long)n * (n + 1) / 2;
    ctx->neri = npair * (npair + 1) / 2;
    ctx->nHs = 1 + 2LL * n_core + (2LL * n_core) * (2LL * n_core - 1) / 2;
    ctx->nPs = 1 + 2LL * n_virt + (2LL * n_virt) * (2LL * n_virt - 1) / 2;
    ctx->nlab = ctx->nHs * ctx->nPs;
    CK(reserve(ctx->d_h1, ctx->cap_h1, (size_t)n * n));
    CK(reserve(ctx->d_eri, ctx->cap_eri, (size_t)ctx->neri));
    CK(reserve(ctx->d_eri4, ctx->cap_eri4, (size_t)npair * n * n));
    const long long nca = n_core + n_act, nav = n_act + n_virt;
    CK(reserve(ctx->d_tab, ctx->cap_tab, 2 * (size_t)std::max(1LL, nca * nca * nav * nav)));
    CK(reserve(ctx->d_sgl, ctx->cap_sgl, 2 * (size_t)std::max(1LL, n_act * nca * nav)));
    CK(reserve(ctx->d_hc, ctx->cap_hc, (size_t)n * n));
    CK(reserve(ctx->d_eps, ctx->cap_eps, (size_t)n));
    CK(reserve(ctx->d_gamma, ctx->cap_gamma, (size_t)std::max(1, n_act * n_act)));
    if (!ctx->d_colex) {
        // co-lexicographic pair table of up to 128 items: colex[j(j-1)/2 + i] = i | j << 8, i < j
        std::vector<unsigned short> colex(128 * 127 / 2);
        for (int j = 1, q = 0; j < 128; j++)
            for (int i = 0; i < j; i++) colex[q++] = (unsigned short)(i | (j << 8));
        CK(cudaMalloc(&ctx->d_colex, sizeof(unsigned short) * colex.size()));
        CK(cudaMemcpyAsync(ctx->d_colex, colex.data(), sizeof(unsigned short) * colex.size(), cudaMemcpyHostToDevice,
                           ctx->stream));
        CK(cudaStreamSynchronize(ctx->stream));
    }
    CK(cudaMemcpyAsync(ctx->d_h1, h1, sizeof(double) * n * n, cudaMemcpyDefault, ctx->stream));
    CK(cudaMemcpyAsync(ctx->d_eri, eri, sizeof(double) * ctx->neri, cudaMemcpyDefault, ctx->stream));
    SysDev& s = ctx->hsys;
    s = SysDev{};
    s.n = n;
    s.nc = n_core;
    s.na = n_act;
    s.nv = n_virt;
    s.W = ctx->W;
    s.nalpha = n_alpha;
    s.nbeta = n_beta;
    s.nPs = ctx->nPs;
    s.nlab = ctx->nlab;
    for (int w = 0; w < 2; w++) {
        s.mcore[w] = s.mact[w] = s.mvirt[w] = 0;
        for (int q = 64 * w; q < 64 * w + 64 && q < n; q++) {
            unsigned long long b = 1ull << (q - 64 * w);
            if (q < n_core) s.mcore[w] |= b;
            else if (q < n_core + n_act) s.mact[w] |= b;
            else s.mvirt[w] |= b;
        }
    }
    s.eri = ctx->d_eri;
    s.eri4 = ctx->d_eri4;
    s.tab = ctx->d_tab;
    s.sgl = ctx->d_sgl;
    s.nca = (int)nca;
    s.nav = (int)nav;
    s.tab_half = (unsigned)(nca * nca * nav * nav);
    s.colex = ctx->d_colex;
    s.mag_c = n_core > 1 ? ~0ull / (unsigned long long)n_core + 1ull : 0ull;
    s.mag_v = n_virt > 1 ? ~0ull / (unsigned long long)n_virt + 1ull : 0ull;
    s.h1 = ctx->d_h1;
    s.hc = ctx->d_hc;
    s.eps = ctx->d_eps;
    s.e_nuc = e_core;
    s.max_probe = 64;
    s.G = 1;
    if (int r = walk_plan(ctx, s)) return r;
    if (int r = push_sys(ctx)) return r;
    k_expand_eri<<<1216, 256, 0, ctx->stream>>>(ctx->d_eri, ctx->d_eri4, n);
    CK(cudaGetLastError());
    k_build_tab<<<2432, 256, 0, ctx->stream>>>(ctx->d_sys, ctx->d_tab);
    CK(cudaGetLastError());
    k_build_sgl<<<304, 256, 0, ctx->stream>>>(ctx->d_sys, ctx->d_sgl);
    CK(cudaGetLastError());
    k_core_fock<<<(n * n + 127) / 128, 128, 0, ctx->stream>>>(ctx->d_sys, ctx->d_hc);
    CK(cudaGetLastError());
    if (int r_ = sync_stream(ctx)) return r_;
    ctx->ham = true;
    return 0;
}

int mrq_load_reference(mrq_ctx* ctx, int64_t n_det, const uint64_t* dets, const double* coeffs) {
    if (!ctx) return MRQ_INVALID_ARG;
    ctx->err[0] = 0;
    if (!ctx->ham) return fail(ctx, MRQ_NOT_LOADED, "load the Hamiltonian first");
    if (n_det <= 0 || !dets || !coeffs) return fail(ctx, MRQ_INVALID_ARG, "empty reference");
    CK(cudaSetDevice(ctx->device));
    if (int r_ = sync_stream(ctx)) return r_;
    DeadlinePause pause_(ctx);
    free_walkers(ctx);
    ctx->ref = false;
    const int W = ctx->W;
    unsigned long long cap = 16;
    while (cap < 4ull * (unsigned long long)n_det) cap <<= 1;
    ctx->hcap = cap;
    ctx->nref = n_det;
    const int nrdm = ctx->na * ctx->na * MRQ_RDM_SLICES;
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t b_dets = up(sizeof(unsigned long long) * 2 * W * n_det), b_co = up(sizeof(double) * n_det),
                 b_part = up(sizeof(double) * 2 * MRQ_REF_BLOCKS), b_e = b_co, b_rdm = up(sizeof(double) * std::max(1, nrdm)), b_scal = 256;
    CK(reserve(ctx->d_hash, ctx->cap_hash, (size_t)cap));
    CK(reserve(ctx->d_c, ctx->cap_c, (size_t)ctx->nlab));
    CK(reserve(ctx->d_setup, ctx->cap_setup, b_dets + b_co + b_part + b_rdm + 2 * b_scal + b_e));
    unsigned long long* const d_dets = (unsigned long long*)ctx->d_setup;
    double* const d_co = (double*)(ctx->d_setup + b_dets);
    double* const d_part = (double*)(ctx->d_setup + b_dets + b_co);
    double* const d_rdm = (double*)(ctx->d_setup + b_dets + b_co + b_part);
    double* const d_scal = (double*)(ctx->d_setup + b_dets + b_co + b_part + b_rdm);
    long long* const d_idx = (long long*)(ctx->d_setup + b_dets + b_co + b_part + b_rdm + b_scal);
    double* const d_e = (double*)(ctx->d_setup + b_dets + b_co + b_part + b_rdm + 2 * b_scal);
    CK(cudaMemcpyAsync(d_dets, dets, sizeof(unsigned long long) * 2 * W * n_det, cudaMemcpyDefault, ctx->stream));
    CK(cudaMemcpyAsync(d_co, coeffs, sizeof(double) * n_det, cudaMemcpyDefault, ctx->stream));
    k_default_coeffs<<<(unsigned)std::min<long long>(1024, (ctx->nlab + 255) / 256), 256, 0, ctx->stream>>>(ctx->d_c, ctx->nlab);
    CK(cudaGetLastError());
    CK(cudaMemsetAsync(ctx->d_err, 0, sizeof(int), ctx->stream));
    if (int r = push_sys(ctx)) return r;
    k_hash_clear<<<(unsigned)((cap + 255) / 256), 256, 0, ctx->stream>>>(ctx->d_hash, cap);
    const unsigned nbk = (unsigned)((n_det + 127) / 128);
    if (W == 1) k_hash_build<1><<<nbk, 128, 0, ctx->stream>>>(ctx->d_sys, ctx->d_hash, d_dets, d_co, n_det, ctx->d_err);
    else k_hash_build<2><<<nbk, 128, 0, ctx->stream>>>(ctx->d_sys, ctx->d_hash, d_dets, d_co, n_det, ctx->d_err);
    CK(cudaGetLastError());
    int flag = 0;
    if (int r = check_err_flag(ctx, &flag)) return r;
    if (flag) {
        free_reference(ctx);
        if (flag & 32) return fail(ctx, MRQ_HASH_OVERFLOW, "hash insertion ran past the probe bound");
        return fail(ctx, MRQ_BAD_REFERENCE, "reference determinant with a core hole, a virtual electron, "
                                            "a wrong electron count or a duplicate (flags %d)", flag);
    }
    // start determinant (largest |c|, first on ties), E0, norm, gamma, eps
    k_argmax_abs<<<1, 1024, 0, ctx->stream>>>(d_co, n_det, d_idx);
    const unsigned nd = (unsigned)((n_det + 127) / 128), nw8 = (unsigned)std::min<long long>((n_det + 7) / 8, 8LL * ctx->n_sm);
    if (W == 1) {
        k_ref_diag<1><<<nd, 128, 0, ctx->stream>>>(ctx->d_sys, d_dets, n_det, d_e);
        k_ref_energy<1><<<nw8, 256, 0, ctx->stream>>>(ctx->d_sys, d_dets, d_co, n_det, d_e);
    } else {
        k_ref_diag<2><<<nd, 128, 0, ctx->stream>>>(ctx->d_sys, d_dets, n_det, d_e);
        k_ref_energy<2><<<nw8, 256, 0, ctx->stream>>>(ctx->d_sys, d_dets, d_co, n_det, d_e);
    }
    k_ref_sum<<<MRQ_REF_BLOCKS, 128, 0, ctx->stream>>>(d_e, d_co, n_det, d_part);
    CK(cudaGetLastError());
    if (ctx->na > 0) {
        const dim3 grid(ctx->na * ctx->na, MRQ_RDM_SLICES);
        if (W == 1) k_ref_rdm<1><<<grid, 256, 0, ctx->stream>>>(ctx->d_sys, d_dets, d_co, n_det, d_rdm);
        else k_ref_rdm<2><<<grid, 256, 0, ctx->stream>>>(ctx->d_sys, d_dets, d_co, n_det, d_rdm);
        CK(cudaGetLastError());
    }
    k_setup_finish<<<1, 1024, 0, ctx->stream>>>(ctx->d_sys, d_part, d_rdm, ctx->d_gamma, ctx->d_eps, d_scal);
    CK(cudaGetLastError());
    double scal[8];
    CK(cudaMemcpyAsync(&ctx->start_idx, d_idx, sizeof(long long), cudaMemcpyDeviceToHost, ctx->stream));
    CK(cudaMemcpyAsync(scal, d_scal, sizeof(double) * 4, cudaMemcpyDeviceToHost, ctx->stream));
    ctx->eps.assign(ctx->n, 0.0);
    ctx->gamma.assign((size_t)ctx->na * ctx->na, 0.0);
    CK(cudaMemcpyAsync(ctx->eps.data(), ctx->d_eps, sizeof(double) * ctx->n, cudaMemcpyDeviceToHost, ctx->stream));
    if (ctx->na)
        CK(cudaMemcpyAsync(ctx->gamma.data(), ctx->d_gamma, sizeof(double) * ctx->na * ctx->na, cudaMemcpyDeviceToHost,
                           ctx->stream));
    if (int r_ = sync_stream(ctx)) return r_;
    memset(ctx->start, 0, sizeof ctx->start);
    {
        unsigned long long tmp[4] = {0, 0, 0, 0};
        CK(cudaMemcpyAsync(tmp, d_dets + ctx->start_idx * 2 * W, sizeof(unsigned long long) * 2 * W, cudaMemcpyDeviceToHost,
                           ctx->stream));
        CK(cudaMemcpyAsync(&ctx->start_c, d_co + ctx->start_idx, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
        if (int r_ = sync_stream(ctx)) return r_;
        for (int w = 0; w < W; w++) {
            ctx->start[w] = tmp[w];
            ctx->start[2 + w] = tmp[W + w];
        }
    }
    ctx->e0 = scal[0];
    ctx->norm0 = scal[1];
    ctx->e_core = scal[2];
    ctx->sum_eps_core = scal[3];
    int flag2 = 0;
    if (int r = check_err_flag(ctx, &flag2)) return r;
    if (flag2 & MRQ_ERR_HASH) return fail(ctx, MRQ_HASH_OVERFLOW, "hash probe bound exceeded during setup");
    if (int r = push_sys(ctx)) return r;
    if (int r_ = sync_stream(ctx)) return r_;
    ctx->ref = true;
    return 0;
}

int mrq_set_coeffs(mrq_ctx* ctx, int64_t n_labels, const double* c) {
    if (!ctx) return MRQ_INVALID_ARG;
    ctx->err[0] = 0;
    if (!ctx->ref) return fail(ctx, MRQ_NOT_LOADED, "load the Hamiltonian and the reference first");
    if (n_labels != ctx->nlab || !c)
        return fail(ctx, MRQ_INVALID_ARG, "expected %lld coefficients", (long long)ctx->nlab);
    CK(cudaSetDevice(ctx->device));
    dfree(ctx->d_am_m);     // a new coefficient vector starts a new optimisation
    dfree(ctx->d_am_v);
    dfree(ctx->d_am_vh);
    CK(cudaMemcpyAsync(ctx->d_c, c, sizeof(double) * n_labels, cudaMemcpyDefault, ctx->stream));
    if (int r_ = sync_stream(ctx)) return r_;
    return 0;
}

int mrq_setup_info(mrq_ctx* ctx, double* out5, double* eps, double* gamma) {
    if (!ctx || !out5) return MRQ_INVALID_ARG;
    if (!ctx->ref) return fail(ctx, MRQ_NOT_LOADED, "no reference loaded");
    out5[0] = ctx->e0;
    out5[1] = ctx->norm0;
    out5[2] = ctx->e_core;
    out5[3] = ctx->sum_eps_core;
    out5[4] = (double)ctx->start_idx;
    if (eps) memcpy(eps, ctx->eps.data(), sizeof(double) * ctx->n);
    if (gamma && ctx->na) memcpy(gamma, ctx->gamma.data(), sizeof(double) * ctx->na * ctx->na);
    return 0;
}

int mrq_debug_local(mrq_ctx* ctx, int64_t n, const uint64_t* dets, mrq_local* local, int64_t max_nb,
                    mrq_neighbour* nb) {
    if (!ctx) return MRQ_INVALID_ARG;
    ctx->err[0] = 0;
    if (!ctx->ref) return fail(ctx, MRQ_NOT_LOADED, "no reference loaded");
    if (n <= 0 || !dets || !local || (nb && max_nb <= 0)) return fail(ctx, MRQ_INVALID_ARG, "bad arguments");
    CK(cudaSetDevice(ctx->device));
    DeadlinePause pause_(ctx);
    const int W = ctx->W;
    unsigned long long* d_dets = nullptr;
    mrq_local* d_loc = nullptr;
    mrq_neighbour* d_nb = nullptr;
    CK(cudaMalloc(&d_dets, sizeof(unsigned long long) * 2 * W * n));
    CK(cudaMalloc(&d_loc, sizeof(mrq_local) * n));
    if (nb) CK(cudaMalloc(&d_nb, sizeof(mrq_neighbour) * n * max_nb));
    CK(cudaMemcpyAsync(d_dets, dets, sizeof(unsigned long long) * 2 * W * n, cudaMemcpyDefault, ctx->stream));
    CK(cudaMemsetAsync(ctx->d_err, 0, sizeof(int), ctx->stream));
    if (int r = push_sys(ctx)) return r;
    const int cap = ctx->hsys.cand_cap;
    const int nw = std::min(warps_of(ctx), MRQ_MAXNW);
    const size_t smem = debug_smem_bytes(nw, cap, ctx->hsys.gstride);
    // neighbour offsets of the CAS units, for the records
    const long long stride = nb ? std::max(1, ctx->hsys.unit_off[8]) : 0;
    if (nb) CK(reserve(ctx->d_nbpre, ctx->cap_nbpre, (size_t)(n * stride)));
    long long* pre = nb ? ctx->d_nbpre : nullptr;
    if (W == 1) {
        CK(cudaFuncSetAttribute(k_debug2<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, MRQ_MAX_SMEM));
        k_debug2<1><<<(unsigned)n, 32 * nw, smem, ctx->stream>>>(ctx->d_sys, d_dets, n, d_loc, max_nb, d_nb, pre,
                                                                 (int)stride);
    } else {
        CK(cudaFuncSetAttribute(k_debug2<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, MRQ_MAX_SMEM));
        k_debug2<2><<<(unsigned)n, 32 * nw, smem, ctx->stream>>>(ctx->d_sys, d_dets, n, d_loc, max_nb, d_nb, pre,
                                                                 (int)stride);
    }
    CK(cudaGetLastError());
    if (int r = sync_stream(ctx)) return r;
    CK(cudaMemcpyAsync(local, d_loc, sizeof(mrq_local) * n, cudaMemcpyDeviceToHost, ctx->stream));
    if (nb) CK(cudaMemcpyAsync(nb, d_nb, sizeof(mrq_neighbour) * n * max_nb, cudaMemcpyDeviceToHost, ctx->stream));
    int flag = 0;
    if (int r = check_err_flag(ctx, &flag)) return r;
    cudaFree(d_dets);
    cudaFree(d_loc);
    if (d_nb) cudaFree(d_nb);
    if (flag & MRQ_ERR_HASH) return fail(ctx, MRQ_HASH_OVERFLOW, "hash probe bound exceeded");
    if (flag & MRQ_ERR_CAP) return fail(ctx, MRQ_TOO_LARGE, "candidate list capacity exceeded");
    return 0;
}

int mrq_walkers_init(mrq_ctx* ctx, const mrq_sample_params* p) {
    if (!ctx || !p) return MRQ_INVALID_ARG;
    ctx->err[0] = 0;
    if (!ctx->ref) return fail(ctx, MRQ_NOT_LOADED, "no reference loaded");
    if (p->n_walkers <= 0 || p->n_groups <= 0 || p->n_groups > 64 || p->n_steps < 0 || p->burn_in < 0)
        return fail(ctx, MRQ_INVALID_ARG, "need n_walkers > 0, 1 <= n_groups <= 64, n_steps >= 0, burn_in >= 0");
    if (p->warps_per_walker != 0 && p->warps_per_walker != 1 && p->warps_per_walker != 2 && p->warps_per_walker != 4 &&
        p->warps_per_walker != 8)
        return fail(ctx, MRQ_INVALID_ARG, "warps_per_walker must be 0, 1, 2, 4 or 8");
    if (p->steps_per_check < 0 || p->target_sigma < 0.0)
        return fail(ctx, MRQ_INVALID_ARG, "need steps_per_check >= 0 and target_sigma >= 0");
    if (p->warps_per_walker) ctx->wpb = p->warps_per_walker;
    CK(cudaSetDevice(ctx->device));
    DeadlinePause pause_(ctx);
    ctx->nwalk = 0;                   // (none, should an allocation fail)
    CK(reserve(ctx->d_walk, ctx->cap_walk, (size_t)p->n_walkers));
    if (int r = alloc_accumulators(ctx, p->n_groups)) return r;
    ctx->nwalk = p->n_walkers;
    ctx->G = p->n_groups;
    ctx->burn = p->burn_in;
    ctx->seed = p->seed;
    ctx->tau = p->screen_tau;
    ctx->total_steps = 0;
    ctx->walk_ms = 0.0;
    ctx->launches = 0;
    ctx->launches_total = 0;
    CK(cudaMemsetAsync(ctx->d_accN, 0, sizeof(double) * ctx->nlab * ctx->G, ctx->stream));
    CK(cudaMemsetAsync(ctx->d_accU, 0, sizeof(double) * ctx->nlab * ctx->G, ctx->stream));
    CK(cudaMemsetAsync(ctx->d_accA, 0, sizeof(double) * ctx->nlab * ctx->G, ctx->stream));
    CK(cudaMemsetAsync(ctx->d_accB, 0, sizeof(double) * ctx->nlab * ctx->G, ctx->stream));
    CK(cudaMemsetAsync(ctx->d_accW, 0, sizeof(double) * ctx->G, ctx->stream));
    CK(cudaMemsetAsync(ctx->d_accE, 0, sizeof(double) * ctx->G, ctx->stream));
    CK(cudaMemsetAsync(ctx->d_types, 0, sizeof(unsigned long long) * MRQ_NTYPES, ctx->stream));
    CK(cudaMemsetAsync(ctx->d_err, 0, sizeof(int), ctx->stream));
    if (int r = push_sys(ctx)) return r;
    double c0 = 1.0;
    CK(cudaMemcpyAsync(&c0, ctx->d_c, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    if (int r_ = sync_stream(ctx)) return r_;
    if (!ctx->d_wptr) CK(cudaMalloc(&ctx->d_wptr, sizeof(Walker*)));
    if (!ctx->d_woff) CK(cudaMalloc(&ctx->d_woff, 2 * sizeof(long long)));
    {
        ctx->h_wset_ptr = ctx->d_walk;
        ctx->h_wset_off[0] = 0;
        ctx->h_wset_off[1] = ctx->nwalk;
        CK(cudaMemcpyAsync(ctx->d_wptr, &ctx->h_wset_ptr, sizeof(Walker*), cudaMemcpyHostToDevice, ctx->stream));
        CK(cudaMemcpyAsync(ctx->d_woff, ctx->h_wset_off, 2 * sizeof(long long), cudaMemcpyHostToDevice, ctx->stream));
    }
    k_walkers_init<<<(unsigned)((ctx->nwalk + 255) / 256), 256, 0, ctx->stream>>>(
        ctx->d_walk, ctx->nwalk, ctx->start[0], ctx->start[1], ctx->start[2], ctx->start[3], c0 * ctx->start_c, 0, ctx->G);
    CK(cudaGetLastError());
    return 0;
}

int mrq_walkers_advance(mrq_ctx* ctx, int64_t n_steps) {
    if (!ctx) return MRQ_INVALID_ARG;
    if (!ctx->ref || !ctx->d_walk || ctx->nwalk == 0) return fail(ctx, MRQ_NOT_LOADED, "walkers not initialised");
    if (n_steps <= 0) return 0;
    CK(cudaSetDevice(ctx->device));
    const size_t k = (size_t)ctx->launches * 2;
    while (ctx->evs.size() < k + 2) {
        cudaEvent_t e;
        CK(cudaEventCreate(&e));
        ctx->evs.push_back(e);
    }
    CK(cudaEventRecord(ctx->evs[k], ctx->stream));
    WalkSet ws{ctx->d_sys, ctx->d_wptr, ctx->d_woff, 1, ctx->nwalk};
    WalkNeed need;
    need.add(ctx);
    WalkLaunch L;
    L.wpb = warps_of(ctx);
    if (int r = l2_window(ctx, L.l2win)) return r;
    const int64_t spl = ctx->spl > 0 ? ctx->spl : n_steps;
    for (int64_t done = 0; done < n_steps; done += spl)
        if (int r = launch_walk(ctx, ctx->W, ws, (int)std::min<int64_t>(spl, n_steps - done), need, L))
            return r;
    CK(cudaGetLastError());
    CK(cudaEventRecord(ctx->evs[k + 1], ctx->stream));
    ctx->launches++;
    ctx->total_steps += n_steps * ctx->nwalk;
    return 0;
}

static long long fin_scratch_doubles(const mrq_ctx* ctx, int* nchunk) {
    *nchunk = (int)((ctx->nlab + FIN_CHUNK - 1) / FIN_CHUNK);
    return (long long)(ctx->G + 1) * (*nchunk) * FIN_NV;
}

// finalize with the partial sums in `scratch` (at least fin_scratch_doubles() doubles)
// (the device copy of the system is current since mrq_walkers_init pushed it, so nothing is copied
// in: a copy from pageable host memory would wait for the walk and defeat the deadline)
static int finalize_with(mrq_ctx* ctx, mrq_result* out, double* scratch, int nchunk) {
    k_fin_list<<<nchunk, 1024, 0, ctx->stream>>>(ctx->d_sys, FIN_CHUNK, ctx->d_flist);
    k_fin_labels<<<(ctx->G + 1) * nchunk, 256, 0, ctx->stream>>>(ctx->d_sys, ctx->tau, nchunk, FIN_CHUNK, ctx->d_flist, scratch);
    CK(cudaGetLastError());
    k_fin_reduce<<<1, 1024, 0, ctx->stream>>>(ctx->d_sys, scratch, nchunk, ctx->d_res);
    CK(cudaGetLastError());
    ctx->kernels += 3;
    if (int r = sync_stream(ctx)) return r;
    CK(cudaMemcpyAsync(out, ctx->d_res, sizeof(mrq_result), cudaMemcpyDeviceToHost, ctx->stream));
    int flag = 0;
    if (int r = check_err_flag(ctx, &flag)) return r;
    for (int i = 0; i < ctx->launches; i++) {
        float ms = 0.0f;
        if (cudaEventElapsedTime(&ms, ctx->evs[2 * i], ctx->evs[2 * i + 1]) == cudaSuccess) ctx->walk_ms += ms;
    }
    out->walk_launches = ctx->launches_total += ctx->launches;
    ctx->launches = 0;
    out->seconds = ctx->walk_ms * 1e-3;
    out->total_steps = ctx->total_steps;
    out->status = 0;
    if (flag & MRQ_ERR_HASH) out->status = MRQ_HASH_OVERFLOW;
    else if (flag & MRQ_ERR_CAP) out->status = MRQ_TOO_LARGE;
    else if (flag & (MRQ_ERR_NOMOVE | MRQ_ERR_LABEL)) out->status = MRQ_NO_MOVE;
    if (out->status) return fail(ctx, out->status, "device flagged an error during the walk (flags %d)", flag);
    return 0;
}

int mrq_finalize(mrq_ctx* ctx, mrq_result* out) {
    if (!ctx || !out) return MRQ_INVALID_ARG;
    if (!ctx->ref || !ctx->d_accN) return fail(ctx, MRQ_NOT_LOADED, "walkers not initialised");
    CK(cudaSetDevice(ctx->device));
    int nchunk = 0;
    const long long need = fin_scratch_doubles(ctx, &nchunk);
    CK(reserve(ctx->d_partial, ctx->cap_partial, (size_t)need));
    return finalize_with(ctx, out, ctx->d_partial, nchunk);
}

int mrq_finalize_noalloc(mrq_ctx* ctx, mrq_result* out) {
    if (!ctx || !out) return MRQ_INVALID_ARG;
    ctx->err[0] = 0;
    if (!ctx->ref || !ctx->d_accN) return fail(ctx, MRQ_NOT_LOADED, "walkers not initialised");
    double* scratch = nullptr;
    if (ctx->device >= 0 && ctx->device < MRQ_MAX_DEVICES) {
        std::lock_guard<std::mutex> lock(g_noalloc_mu);
        scratch = g_noalloc_ptr[ctx->device];
    }
    if (scratch == nullptr)
        return fail(ctx, MRQ_CUDA_ERROR, "fixed finalize scratch has no device address on device %d", ctx->device);
    int nchunk = 0;
    const long long need = fin_scratch_doubles(ctx, &nchunk);
    if (need > MRQ_NOALLOC_SCRATCH_DOUBLES)
        return fail(ctx, MRQ_TOO_LARGE,
                    "mrq_finalize_noalloc: %lld labels x %d groups need %lld scratch doubles, more than its fixed "
                    "%d (use mrq_finalize)", (long long)ctx->nlab, ctx->G, need, MRQ_NOALLOC_SCRATCH_DOUBLES);
    CK(cudaSetDevice(ctx->device));
    return finalize_with(ctx, out, scratch, nchunk);
}

int mrq_mrci_gradient(mrq_ctx* ctx, double* grad, double* energy) {
    if (!ctx) return MRQ_INVALID_ARG;
    ctx->err[0] = 0;
    if (!ctx->ref || !ctx->d_accA) return fail(ctx, MRQ_NOT_LOADED, "no walk to take the gradient from");
    CK(cudaSetDevice(ctx->device));
    if (!ctx->d_grad) CK(cudaMalloc(&ctx->d_grad, sizeof(double) * (ctx->nlab + 1)));
    if (int r = push_sys(ctx)) return r;
    k_mrci_grad<<<(unsigned)std::min<long long>(1024, (ctx->nlab + 255) / 256), 256, 0, ctx->stream>>>(
        ctx->d_sys, ctx->d_grad, ctx->d_grad + ctx->nlab);
    CK(cudaGetLastError());
    double e = 0.0;
    if (grad) CK(cudaMemcpyAsync(grad, ctx->d_grad, sizeof(double) * ctx->nlab, cudaMemcpyDefault, ctx->stream));
    CK(cudaMemcpyAsync(&e, ctx->d_grad + ctx->nlab, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    if (int r_ = sync_stream(ctx)) return r_;
    if (energy) *energy = e;
    return 0;
}

int mrq_amsgrad_step(mrq_ctx* ctx, double lr, double beta1, double beta2, double eps) {
    if (!ctx) return MRQ_INVALID_ARG;
    ctx->err[0] = 0;
    if (!ctx->d_grad) return fail(ctx, MRQ_NOT_LOADED, "call mrq_mrci_gradient first");
    if (!(lr > 0.0) || !(beta1 >= 0.0 && beta1 < 1.0) || !(beta2 >= 0.0 && beta2 < 1.0) || !(eps > 0.0))
        return fail(ctx, MRQ_INVALID_ARG, "need lr > 0, 0 <= beta < 1, eps > 0");
    CK(cudaSetDevice(ctx->device));
    if (!ctx->d_am_m || !ctx->d_am_v || !ctx->d_am_vh) {     // (the last one is missing where a call ran out of memory)
        for (double** p : {&ctx->d_am_m, &ctx->d_am_v, &ctx->d_am_vh})
            if (!*p) CK(cudaMalloc(p, sizeof(double) * ctx->nlab));
        CK(cudaMemsetAsync(ctx->d_am_m, 0, sizeof(double) * ctx->nlab, ctx->stream));
        CK(cudaMemsetAsync(ctx->d_am_v, 0, sizeof(double) * ctx->nlab, ctx->stream));
        CK(cudaMemsetAsync(ctx->d_am_vh, 0, sizeof(double) * ctx->nlab, ctx->stream));
    }
    k_amsgrad<<<(unsigned)std::min<long long>(1024, (ctx->nlab + 255) / 256), 256, 0, ctx->stream>>>(
        ctx->d_c, ctx->d_grad, ctx->d_am_m, ctx->d_am_v, ctx->d_am_vh, ctx->nlab, lr, beta1, beta2, eps);
    CK(cudaGetLastError());
    if (int r_ = sync_stream(ctx)) return r_;
    return 0;
}

int mrq_read_coeffs(mrq_ctx* ctx, double* c) {
    if (!ctx || !c) return MRQ_INVALID_ARG;
    if (!ctx->ref) return fail(ctx, MRQ_NOT_LOADED, "no reference loaded");
    CK(cudaSetDevice(ctx->device));
    if (int r = sync_stream(ctx)) return r;
    CK(cudaMemcpyAsync(c, ctx->d_c, sizeof(double) * ctx->nlab, cudaMemcpyDefault, ctx->stream));
    if (int r_ = sync_stream(ctx)) return r_;
    return 0;
}

static int batch_check(mrq_ctx* const* ctxs, int n) {
    if (!ctxs || n <= 0) return MRQ_INVALID_ARG;
    mrq_ctx* lead = ctxs[0];
    if (!lead) return MRQ_INVALID_ARG;
    for (int i = 0; i < n; i++) {
        if (!ctxs[i]) return fail(lead, MRQ_INVALID_ARG, "context %d is null", i);
        if (ctxs[i]->device != lead->device)
            return fail(lead, MRQ_INVALID_ARG, "contexts of one batch must share a device");
        if (!ctxs[i]->ref || !ctxs[i]->d_walk || ctxs[i]->nwalk == 0)
            return fail(lead, MRQ_NOT_LOADED, "context %d has no initialised walkers", i);
        for (int j = 0; j < i; j++)
            if (ctxs[j] == ctxs[i]) return fail(lead, MRQ_INVALID_ARG, "context %d appears twice", i);
    }
    return 0;
}

// the batch's systems of determinant width W whose launches take nw_eff warps per block (the requested
// nw, at most what each system's candidate lists allow): device tables in the lead context, walker
// arrays from `walkers` (the contexts' own, or the tuner's scratch copies)
static int batch_tables(mrq_ctx* const* ctxs, int n, int W, Walker* const* walkers, WalkSet& ws, WalkNeed& need, int nw,
                        int nw_eff) {
    mrq_ctx* ctx = ctxs[0];
    CK(reserve(ctx->d_bsys, ctx->cap_bsys, (size_t)n));
    CK(reserve(ctx->d_bwptr, ctx->cap_bwptr, (size_t)n));
    CK(reserve(ctx->d_boff, ctx->cap_boff, (size_t)n + 1));
    std::vector<SysDev> sys;
    std::vector<Walker*> wp;
    std::vector<long long> off(1, 0);
    need = WalkNeed();
    for (int i = 0; i < n; i++) {
        if (ctxs[i]->W != W || std::min(nw, ctxs[i]->max_nw) != nw_eff) continue;
        sys.push_back(ctxs[i]->hsys);
        wp.push_back(walkers[i]);
        off.push_back(off.back() + ctxs[i]->nwalk);
        need.add(ctxs[i]);
    }
    ws = WalkSet{ctx->d_bsys, ctx->d_bwptr, ctx->d_boff, (int)sys.size(), off.back()};
    if (sys.empty()) return 0;
    const int k = (int)sys.size();
    CK(cudaMemcpy(ctx->d_bsys, sys.data(), sizeof(SysDev) * k, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->d_bwptr, wp.data(), sizeof(Walker*) * k, cudaMemcpyHostToDevice));
    CK(cudaMemcpy(ctx->d_boff, off.data(), sizeof(long long) * (k + 1), cudaMemcpyHostToDevice));
    return 0;
}

// the key of a graph of this launch; the workspace and the launch shapes are prepared
static void graph_key(const mrq_ctx* ctx, const WalkSet& ws, const WalkNeed& need, int wpb, int spl, mrq_ctx::GraphKey& key) {
    memset((void*)&key, 0, sizeof key);
    key.sys = ws.systems;
    key.wptr = ws.walkers;
    key.off = ws.offsets;
    key.nslots = ws.nslots;
    key.k = ws.nsys;
    key.wpb = wpb;
    key.spl = spl;
    key.cap = need.cap;
    key.rows_minb = ctx->rows_minb;
    key.rows_blocks = ctx->rows_blocks;
    key.frows_blocks = ctx->frows_blocks;
    memcpy((void*)&key.work, (const void*)&ctx->work, sizeof(WalkScratch));
}

// n_steps steps of one width's walk set: launches of `spl` steps (the reporting interval), replayed
// from a CUDA graph when the lead context asks for it
static int batch_run(mrq_ctx* const* ctxs, int n, int W, const WalkSet& ws, const WalkNeed& need, int64_t n_steps, int wpb,
                     int64_t spl, int accumulate, bool graph, int slot) {
    mrq_ctx* const ctx = ctxs[0];
    WalkLaunch L;
    L.peers.ctxs = ctxs;
    L.peers.n = n;
    L.wpb = wpb;
    L.accumulate = accumulate;
    if (spl <= 0 || spl > n_steps) spl = n_steps;
    const int64_t nfull = n_steps / spl, rem = n_steps % spl;
    if (graph && nfull > 0) {
        if (int r = work_prepare(ctx, ws.nslots, need, L.peers)) return r;
        if (int r = rows_prepare(ctx, W, std::min(wpb, MRQ_MAXNW), need.cap)) return r;
        mrq_ctx::GraphKey key;
        graph_key(ctx, ws, need, wpb, (int)spl, key);
        cudaGraphExec_t& ex = ctx->gexec[slot];
        if (!ex || memcmp(&ctx->gkey[slot], &key, sizeof key) != 0) {
            if (ex) CK(cudaGraphExecDestroy(ex));
            ex = nullptr;
            CK(cudaStreamBeginCapture(ctx->stream, cudaStreamCaptureModeThreadLocal));
            L.captured = true;
            const long long before = ctx->kernels;
            const int r = launch_walk(ctx, W, ws, (int)spl, need, L);
            ctx->gkernels[slot] = ctx->kernels - before;
            ctx->kernels = before;
            cudaGraph_t g = nullptr;
            const cudaError_t e = cudaStreamEndCapture(ctx->stream, &g);
            if (r || e != cudaSuccess) {
                if (g) cudaGraphDestroy(g);
                return r ? r : fail(ctx, MRQ_CUDA_ERROR, "stream capture: %s", cudaGetErrorString(e));
            }
            const cudaError_t ei = cudaGraphInstantiate(&ex, g, 0);
            cudaGraphDestroy(g);
            if (ei != cudaSuccess) {
                ex = nullptr;
                return fail(ctx, MRQ_CUDA_ERROR, "cudaGraphInstantiate: %s", cudaGetErrorString(ei));
            }
            memcpy(&ctx->gkey[slot], &key, sizeof key);
        }
        for (int64_t i = 0; i < nfull; i++) CK(cudaGraphLaunch(ex, ctx->stream));
        ctx->graph_replays += nfull;
        ctx->kernels += nfull * ctx->gkernels[slot];
        L.captured = false;
    } else {
        for (int64_t i = 0; i < nfull; i++)
            if (int r = launch_walk(ctx, W, ws, (int)spl, need, L)) return r;
    }
    if (rem > 0)
        if (int r = launch_walk(ctx, W, ws, (int)rem, need, L)) return r;
    return 0;
}

int mrq_batch_advance(mrq_ctx* const* ctxs, int n, int64_t n_steps) {
    if (int r = batch_check(ctxs, n)) return r;
    mrq_ctx* lead = ctxs[0];
    if (n_steps <= 0) return 0;
    lead->err[0] = 0;
    cudaError_t e0 = cudaSetDevice(lead->device);
    if (e0 != cudaSuccess) return fail(lead, MRQ_CUDA_ERROR, "cudaSetDevice: %s", cudaGetErrorString(e0));
    mrq_ctx* ctx = lead;   // for CK
    for (int i = 0; i < n; i++) CK(cudaStreamSynchronize(ctxs[i]->stream));
    std::vector<Walker*> own(n);
    for (int i = 0; i < n; i++) own[i] = ctxs[i]->d_walk;
    // one launch sequence per determinant width and warps per block
    for (int slot = 0; slot < mrq_ctx::NSLOT; slot++) {
        const int W = 1 + slot / 4, nw_eff = MRQ_MAXNW >> (slot % 4), nw = lead->wpb > 0 ? lead->wpb : MRQ_MAXNW;
        WalkSet ws;
        WalkNeed need;
        if (int r = batch_tables(ctxs, n, W, own.data(), ws, need, nw, nw_eff)) return r;
        if (ws.nsys == 0) continue;
        const size_t q = (size_t)ctx->launches * 2;
        while (ctx->evs.size() < q + 2) {
            cudaEvent_t ev;
            CK(cudaEventCreate(&ev));
            ctx->evs.push_back(ev);
        }
        CK(cudaEventRecord(ctx->evs[q], ctx->stream));
        if (int r = batch_run(ctxs, n, W, ws, need, n_steps, nw_eff, lead->spl, 1, lead->use_graph != 0, slot))
            return r;
        CK(cudaEventRecord(ctx->evs[q + 1], ctx->stream));
        ctx->launches++;
        if (int r_ = sync_stream(ctx)) return r_;   // the tables are reused by the next launch
    }
    for (int i = 0; i < n; i++) ctxs[i]->total_steps += n_steps * ctxs[i]->nwalk;
    return 0;
}

int mrq_set_launch(mrq_ctx* ctx, int warps_per_walker, int steps_per_launch, int use_graph) {
    if (!ctx) return MRQ_INVALID_ARG;
    if (warps_per_walker != 0 && warps_per_walker != 1 && warps_per_walker != 2 && warps_per_walker != 4 &&
        warps_per_walker != 8)
        return fail(ctx, MRQ_INVALID_ARG, "warps_per_walker must be 0 (automatic), 1, 2, 4 or 8");
    if (steps_per_launch < 0) return fail(ctx, MRQ_INVALID_ARG, "steps_per_launch must be >= 0");
    ctx->wpb = warps_per_walker;
    ctx->spl = steps_per_launch;
    ctx->use_graph = use_graph != 0;
    return 0;
}

int mrq_tune_batch(mrq_ctx* const* ctxs, int n, int64_t trial_steps, mrq_tune_result* out) {
    if (int r = batch_check(ctxs, n)) return r;
    mrq_ctx* ctx = ctxs[0];
    if (trial_steps < 1 || trial_steps > 1024) return fail(ctx, MRQ_INVALID_ARG, "trial_steps must be in [1, 1024]");
    ctx->err[0] = 0;
    CK(cudaSetDevice(ctx->device));
    for (int i = 0; i < n; i++) CK(cudaStreamSynchronize(ctxs[i]->stream));
    // scratch copies of every system's walkers: the trials move those, never the real ones
    long long tot = 0;
    for (int i = 0; i < n; i++) tot += ctxs[i]->nwalk;
    CK(reserve(ctx->d_tune, ctx->cap_tune, (size_t)tot));
    std::vector<Walker*> scratch(n);
    {
        long long o = 0;
        for (int i = 0; i < n; i++) {
            scratch[i] = ctx->d_tune + o;
            o += ctxs[i]->nwalk;
        }
    }
    auto restore = [&]() -> int {
        for (int i = 0; i < n; i++)
            CK(cudaMemcpyAsync(scratch[i], ctxs[i]->d_walk, sizeof(Walker) * ctxs[i]->nwalk, cudaMemcpyDeviceToDevice,
                               ctx->stream));
        return 0;
    };
    const int wpbs[3] = {2, 4, 8};
    std::vector<int64_t> spls;
    for (int64_t v : {(int64_t)1, (int64_t)4, (int64_t)16})
        if (v <= trial_steps) spls.push_back(v);
    mrq_tune_result res{};
    double best = 1e300;
    int reps = 3;
    for (int pass = -1; pass < (int)(3 * spls.size()); pass++) {
        const int wpb = pass < 0 ? 8 : wpbs[pass / (int)spls.size()];
        const int64_t spl = pass < 0 ? 1 : spls[pass % spls.size()];
        double ms_best = 1e300;
        for (int rep = 0; rep < (pass < 0 ? 1 : reps); rep++) {
            if (int r = restore()) return r;
            CK(cudaEventRecord(ctx->ev0, ctx->stream));
            for (int slot = 0; slot < mrq_ctx::NSLOT; slot++) {
                const int W = 1 + slot / 4, nw_eff = MRQ_MAXNW >> (slot % 4);
                WalkSet ws;
                WalkNeed need;
                if (int r = batch_tables(ctxs, n, W, scratch.data(), ws, need, wpb, nw_eff)) return r;
                if (ws.nsys == 0) continue;
                if (int r = batch_run(ctxs, n, W, ws, need, trial_steps, nw_eff, spl, 0, false, slot)) return r;
                if (int r_ = sync_stream(ctx)) return r_;
            }
            CK(cudaEventRecord(ctx->ev1, ctx->stream));
            CK(cudaEventSynchronize(ctx->ev1));
            float ms = 0.0f;
            CK(cudaEventElapsedTime(&ms, ctx->ev0, ctx->ev1));
            ms_best = std::min(ms_best, (double)ms);
            if (ms > 200.0f) reps = 1;     // long trials: one repetition is precise enough
        }
        if (pass < 0) continue;            // warm-up
        if (res.n_tried < MRQ_TUNE_MAX) {
            res.tried_warps_per_walker[res.n_tried] = wpb;
            res.tried_steps_per_launch[res.n_tried] = (int)spl;
            res.tried_ms[res.n_tried] = ms_best;
            res.n_tried++;
        }
        if (ms_best < best) {
            best = ms_best;
            res.warps_per_walker = wpb;
            res.steps_per_launch = (int)spl;
        }
    }
    for (int i = 0; i < n; i++) {
        ctxs[i]->wpb = res.warps_per_walker;
        ctxs[i]->spl = res.steps_per_launch;
    }
    if (out) *out = res;
    return 0;
}

int mrq_sample_batch(mrq_ctx* const* ctxs, int n, const mrq_sample_params* params, mrq_result* out) {
    if (!ctxs || n <= 0 || !params || !out) return MRQ_INVALID_ARG;
    for (int i = 0; i < n; i++)
        if (params[i].n_steps != params[0].n_steps)
            return fail(ctxs[0], MRQ_INVALID_ARG, "all systems of a batch take the same number of steps");
    for (int i = 0; i < n; i++)
        if (int r = mrq_walkers_init(ctxs[i], &params[i])) return r;
    if (int r = mrq_batch_advance(ctxs, n, params[0].n_steps)) return r;
    int rc = 0;
    for (int i = 0; i < n; i++) {
        int r = mrq_finalize(ctxs[i], &out[i]);
        if (r && !rc) rc = r;
    }
    return rc;
}

int mrq_sample(mrq_ctx* ctx, const mrq_sample_params* p, mrq_result* out) {
    if (int r = mrq_walkers_init(ctx, p)) return r;
    if (!(p->target_sigma > 0.0)) {
        if (int r = mrq_walkers_advance(ctx, p->n_steps)) return r;
        return mrq_finalize(ctx, out);
    }
    const int64_t chunk = p->steps_per_check > 0 ? p->steps_per_check : std::max<int64_t>(1, p->n_steps / 16);
    int64_t done = 0;
    bool fresh = false;
    while (done < p->n_steps) {
        const int64_t k = std::min(chunk, p->n_steps - done);
        if (int r = mrq_walkers_advance(ctx, k)) return r;
        done += k;
        fresh = false;
        if (done <= p->burn_in) continue;
        if (int r = mrq_finalize(ctx, out)) return r;
        fresh = true;
        const double sig = p->method == MRQ_SC_MRCI ? out->e_var_sigma : out->e2_sigma;
        if (sig <= p->target_sigma) break;
    }
    return fresh ? 0 : mrq_finalize(ctx, out);
}

int mrq_read_accumulators(mrq_ctx* ctx, double* accN, double* accU, double* accW, double* accE, int64_t* type_steps) {
    if (!ctx) return MRQ_INVALID_ARG;
    if (!ctx->d_accN) return fail(ctx, MRQ_NOT_LOADED, "no accumulators");
    CK(cudaSetDevice(ctx->device));
    if (int r = sync_stream(ctx)) return r;
    const long long L = ctx->nlab * ctx->G;
    if (accN) CK(cudaMemcpyAsync(accN, ctx->d_accN, sizeof(double) * L, cudaMemcpyDeviceToHost, ctx->stream));
    if (accU) CK(cudaMemcpyAsync(accU, ctx->d_accU, sizeof(double) * L, cudaMemcpyDeviceToHost, ctx->stream));
    if (accW) CK(cudaMemcpyAsync(accW, ctx->d_accW, sizeof(double) * ctx->G, cudaMemcpyDeviceToHost, ctx->stream));
    if (accE) CK(cudaMemcpyAsync(accE, ctx->d_accE, sizeof(double) * ctx->G, cudaMemcpyDeviceToHost, ctx->stream));
    if (type_steps)
        CK(cudaMemcpyAsync(type_steps, ctx->d_types, sizeof(int64_t) * MRQ_NTYPES, cudaMemcpyDeviceToHost, ctx->stream));
    if (int r_ = sync_stream(ctx)) return r_;
    return 0;
}

int mrq_load_accumulators(mrq_ctx* ctx, int32_t n_groups, const double* accN, const double* accU, const double* accW,
                          const double* accE, const double* accA, const double* accB, const int64_t* type_steps,
                          int64_t total_steps) {
    if (!ctx) return MRQ_INVALID_ARG;
    ctx->err[0] = 0;
    if (!ctx->ref) return fail(ctx, MRQ_NOT_LOADED, "no reference loaded");
    if (n_groups <= 0 || n_groups > 64 || !accN || !accU || !accW || !accE || !type_steps || total_steps < 0)
        return fail(ctx, MRQ_INVALID_ARG, "need 1 <= n_groups <= 64, the N, U, W, E sums and the type counts");
    CK(cudaSetDevice(ctx->device));
    if (int r = sync_stream(ctx)) return r;
    DeadlinePause pause_(ctx);
    if (int r = alloc_accumulators(ctx, n_groups)) return r;
    const long long L = ctx->nlab * n_groups;
    CK(cudaMemcpyAsync(ctx->d_accN, accN, sizeof(double) * L, cudaMemcpyDefault, ctx->stream));
    CK(cudaMemcpyAsync(ctx->d_accU, accU, sizeof(double) * L, cudaMemcpyDefault, ctx->stream));
    if (accA) CK(cudaMemcpyAsync(ctx->d_accA, accA, sizeof(double) * L, cudaMemcpyDefault, ctx->stream));
    else CK(cudaMemsetAsync(ctx->d_accA, 0, sizeof(double) * L, ctx->stream));
    if (accB) CK(cudaMemcpyAsync(ctx->d_accB, accB, sizeof(double) * L, cudaMemcpyDefault, ctx->stream));
    else CK(cudaMemsetAsync(ctx->d_accB, 0, sizeof(double) * L, ctx->stream));
    CK(cudaMemcpyAsync(ctx->d_accW, accW, sizeof(double) * n_groups, cudaMemcpyDefault, ctx->stream));
    CK(cudaMemcpyAsync(ctx->d_accE, accE, sizeof(double) * n_groups, cudaMemcpyDefault, ctx->stream));
    CK(cudaMemcpyAsync(ctx->d_types, type_steps, sizeof(int64_t) * MRQ_NTYPES, cudaMemcpyDefault, ctx->stream));
    CK(cudaMemsetAsync(ctx->d_err, 0, sizeof(int), ctx->stream));
    ctx->G = n_groups;
    ctx->nwalk = 0;                    // the walkers no longer match the groups: walkers_init first
    ctx->total_steps = total_steps;
    ctx->walk_ms = 0.0;
    ctx->launches = 0;
    if (int r = push_sys(ctx)) return r;
    return sync_stream(ctx);
}

int mrq_read_gradient_sums(mrq_ctx* ctx, double* accA, double* accB) {
    if (!ctx) return MRQ_INVALID_ARG;
    if (!ctx->d_accA) return fail(ctx, MRQ_NOT_LOADED, "no accumulators");
    CK(cudaSetDevice(ctx->device));
    if (int r = sync_stream(ctx)) return r;
    const size_t bytes = sizeof(double) * ctx->nlab * ctx->G;
    if (accA) CK(cudaMemcpyAsync(accA, ctx->d_accA, bytes, cudaMemcpyDeviceToHost, ctx->stream));
    if (accB) CK(cudaMemcpyAsync(accB, ctx->d_accB, bytes, cudaMemcpyDeviceToHost, ctx->stream));
    if (int r_ = sync_stream(ctx)) return r_;
    return 0;
}

int mrq_debug_race_screen(mrq_ctx* ctx, int64_t n, const uint64_t* k53, const double* rate, const double* t_best,
                          uint8_t* pass, double* exact) {
    if (!ctx) return MRQ_INVALID_ARG;
    ctx->err[0] = 0;
    if (n <= 0 || !k53 || !rate || !t_best || !pass || !exact) return fail(ctx, MRQ_INVALID_ARG, "bad arguments");
    for (int64_t i = 0; i < n; i++)
        if (k53[i] >= (1ull << 53)) return fail(ctx, MRQ_INVALID_ARG, "k53[%lld] has more than 53 bits", (long long)i);
    CK(cudaSetDevice(ctx->device));
    unsigned long long* d_k = nullptr;
    double *d_r = nullptr, *d_t = nullptr, *d_e = nullptr;
    unsigned char* d_p = nullptr;
    CK(cudaMalloc(&d_k, sizeof(unsigned long long) * n));
    CK(cudaMalloc(&d_r, sizeof(double) * n));
    CK(cudaMalloc(&d_t, sizeof(double) * n));
    CK(cudaMalloc(&d_e, sizeof(double) * n));
    CK(cudaMalloc(&d_p, n));
    CK(cudaMemcpyAsync(d_k, k53, sizeof(unsigned long long) * n, cudaMemcpyDefault, ctx->stream));
    CK(cudaMemcpyAsync(d_r, rate, sizeof(double) * n, cudaMemcpyDefault, ctx->stream));
    CK(cudaMemcpyAsync(d_t, t_best, sizeof(double) * n, cudaMemcpyDefault, ctx->stream));
    k_race_screen<<<(unsigned)((n + 255) / 256), 256, 0, ctx->stream>>>(d_k, d_r, d_t, n, d_p, d_e);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(pass, d_p, n, cudaMemcpyDefault, ctx->stream));
    CK(cudaMemcpyAsync(exact, d_e, sizeof(double) * n, cudaMemcpyDefault, ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    cudaFree(d_k);
    cudaFree(d_r);
    cudaFree(d_t);
    cudaFree(d_e);
    cudaFree(d_p);
    return 0;
}

int mrq_debug_race(mrq_ctx* ctx, int64_t n, const uint32_t* exc, const double* t, double psi, uint64_t seed, int32_t n_walkers,
                   const uint32_t* walker, const uint32_t* step, int32_t slices, uint32_t* winner) {
    if (!ctx) return MRQ_INVALID_ARG;
    ctx->err[0] = 0;
    if (n <= 0 || !exc || !t || !(psi != 0.0) || !std::isfinite(psi) || n_walkers <= 0 || !walker || !step || slices < 1 || slices > 4096 || !winner)
        return fail(ctx, MRQ_INVALID_ARG, "bad arguments");
    CK(cudaSetDevice(ctx->device));
    if (int r = sync_stream(ctx)) return r;
    const size_t nw = (size_t)n_walkers;
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t o_exc = up(8 * (size_t)n), o_wid = o_exc + up(4 * (size_t)n), o_step = o_wid + up(4 * nw),
                 o_best = o_step + up(4 * nw), o_bound = o_best + up(sizeof(RaceBest) * nw);
    std::vector<RaceBest> best(nw);
    for (RaceBest& b : best) b = RaceBest{0x7F800000u, 0xFFFFFFFFu, 0.0};
    const std::vector<unsigned> bound(nw, 0x7F800000u);
    unsigned char* d = nullptr;
    CK(cudaMalloc(&d, o_bound + 4 * nw));
    const auto run = [&]() -> int {
        CK(cudaMemcpyAsync(d, t, 8 * (size_t)n, cudaMemcpyDefault, ctx->stream));
        CK(cudaMemcpyAsync(d + o_exc, exc, 4 * (size_t)n, cudaMemcpyDefault, ctx->stream));
        CK(cudaMemcpyAsync(d + o_wid, walker, 4 * nw, cudaMemcpyDefault, ctx->stream));
        CK(cudaMemcpyAsync(d + o_step, step, 4 * nw, cudaMemcpyDefault, ctx->stream));
        CK(cudaMemcpyAsync(d + o_best, best.data(), sizeof(RaceBest) * nw, cudaMemcpyHostToDevice, ctx->stream));
        CK(cudaMemcpyAsync(d + o_bound, bound.data(), 4 * nw, cudaMemcpyHostToDevice, ctx->stream));
        const long long warps = (long long)((nw + MRQ_TGW - 1) / MRQ_TGW) * slices;
        if ((warps + 7) / 8 > 0x7FFFFFFFLL) return fail(ctx, MRQ_INVALID_ARG, "too many walkers");
        k_debug_race<<<(unsigned)((warps + 7) / 8), 256, 0, ctx->stream>>>(
            (const unsigned*)(d + o_exc), (const double*)d, n, 1.0 / psi, seed, (const unsigned*)(d + o_wid),
            (const unsigned*)(d + o_step), n_walkers, slices, (RaceBest*)(d + o_best), (unsigned*)(d + o_bound));
        CK(cudaGetLastError());
        CK(cudaMemcpyAsync(best.data(), d + o_best, sizeof(RaceBest) * nw, cudaMemcpyDeviceToHost, ctx->stream));
        CK(cudaStreamSynchronize(ctx->stream));
        for (size_t i = 0; i < nw; i++) winner[i] = best[i].exc;
        return 0;
    };
    const int r = run();
    cudaFree(d);
    return r;
}

int64_t mrq_kernel_launches(const mrq_ctx* ctx) { return ctx ? ctx->kernels : 0; }

int mrq_set_l2_window(mrq_ctx* ctx, double fraction) {
    if (!ctx) return MRQ_INVALID_ARG;
    if (!(fraction >= 0.0 && fraction <= 1.0)) return fail(ctx, MRQ_INVALID_ARG, "fraction must be in [0, 1]");
    ctx->l2_fraction = fraction;
    return 0;
}

int mrq_set_deadline(mrq_ctx* ctx, double seconds) {
    if (!ctx) return MRQ_INVALID_ARG;
    if (!(seconds >= 0.0)) return fail(ctx, MRQ_INVALID_ARG, "deadline must be >= 0 seconds");
    ctx->deadline_s = seconds;
    return 0;
}

int mrq_debug_set_limits(mrq_ctx* ctx, int max_probe, int cand_cap) {
    if (!ctx) return MRQ_INVALID_ARG;
    if (max_probe < 0 || max_probe > 64 || cand_cap < 0) return fail(ctx, MRQ_INVALID_ARG, "need 0 <= max_probe <= 64, cand_cap >= 0");
    ctx->probe_limit = max_probe;
    ctx->cap_limit = cand_cap;
    if (ctx->ham) {
        CK(cudaSetDevice(ctx->device));
        if (int r = push_sys(ctx)) return r;
    }
    return 0;
}

int mrq_read_walkers(mrq_ctx* ctx, uint64_t* dets, double* psi) {
    if (!ctx) return MRQ_INVALID_ARG;
    if (!ctx->d_walk) return fail(ctx, MRQ_NOT_LOADED, "walkers not initialised");
    CK(cudaSetDevice(ctx->device));
    if (int r = sync_stream(ctx)) return r;
    std::vector<Walker> w(ctx->nwalk);
    CK(cudaMemcpyAsync(w.data(), ctx->d_walk, sizeof(Walker) * ctx->nwalk, cudaMemcpyDeviceToHost, ctx->stream));
    if (int r_ = sync_stream(ctx)) return r_;
    const int W = ctx->W;
    for (long long i = 0; i < ctx->nwalk; i++) {
        if (dets)
            for (int k = 0; k < W; k++) {
                dets[i * 2 * W + k] = w[i].d[0][k];
                dets[i * 2 * W + W + k] = w[i].d[1][k];
            }
        if (psi) psi[i] = w[i].psi;
    }
    return 0;
}

int mrq_set_heat_bath_cutoff(mrq_ctx* ctx, double eps) {
    if (!ctx) return MRQ_INVALID_ARG;
    ctx->err[0] = 0;
    if (!ctx->ham) return fail(ctx, MRQ_NOT_LOADED, "load the Hamiltonian first");
    if (!(eps >= 0.0) || !std::isfinite(eps)) return fail(ctx, MRQ_INVALID_ARG, "the cutoff must be finite and >= 0");
    CK(cudaSetDevice(ctx->device));
    if (int r = sync_stream(ctx)) return r;
    DeadlinePause pause_(ctx);
    ctx->hsys.hb_eps = eps;
    ctx->hsys.hb_on = eps > 0.0 ? 1 : 0;
    if (int r = push_sys(ctx)) return r;
    k_build_tab<<<2432, 256, 0, ctx->stream>>>(ctx->d_sys, ctx->d_tab);
    CK(cudaGetLastError());
    return sync_stream(ctx);
}

int mrq_read_hamiltonian(mrq_ctx* ctx, double* h1, double* eri) {
    if (!ctx) return MRQ_INVALID_ARG;
    ctx->err[0] = 0;
    if (!ctx->ham) return fail(ctx, MRQ_NOT_LOADED, "no Hamiltonian loaded");
    CK(cudaSetDevice(ctx->device));
    if (int r = sync_stream(ctx)) return r;
    if (h1) CK(cudaMemcpyAsync(h1, ctx->d_h1, sizeof(double) * ctx->n * ctx->n, cudaMemcpyDefault, ctx->stream));
    if (eri) CK(cudaMemcpyAsync(eri, ctx->d_eri, sizeof(double) * ctx->neri, cudaMemcpyDefault, ctx->stream));
    return sync_stream(ctx);
}

}  // extern "C"

int mrq_internal_ham(mrq_ctx* ctx, MrqHamView* out) {
    if (!ctx->ham) return fail(ctx, MRQ_NOT_LOADED, "load the Hamiltonian first");
    ctx->err[0] = 0;
    *out = MrqHamView{ctx->device, ctx->stream, ctx->n, ctx->nc, ctx->na, ctx->nv, ctx->nalpha, ctx->nbeta, ctx->W,
                      ctx->d_h1, ctx->d_eri, ctx->neri, ctx->e_nuc};
    return 0;
}

int mrq_internal_fail(mrq_ctx* ctx, int code, const char* fmt, ...) {
    if (ctx) {
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(ctx->err, sizeof ctx->err, fmt, ap);
        va_end(ap);
    }
    return code;
}

int mrq_internal_work_limit(mrq_ctx* ctx, long long bytes) {
    ctx->work_limit = std::max(0LL, bytes);
    if ((long long)ctx->work_cap <= ctx->work_limit) return 0;
    CK(cudaSetDevice(ctx->device));
    if (int r = sync_stream(ctx)) return r;
    free_work(ctx);
    return 0;
}

long long mrq_internal_work_floor(int n_core, int n_act, int n_virt, int n_alpha, int n_beta, long long n_ref) {
    const int n = n_core + n_act + n_virt;
    if (n_core < 0 || n_act < 0 || n_virt < 0 || n <= 0 || n > MRQ_MAXN || n_core > 64 || n_act > 32 || n_alpha < n_core ||
        n_beta < n_core || n_alpha > n_core + n_act || n_beta > n_core + n_act)
        return 0;
    mrq_ctx c;                        // (host side only)
    SysDev& s = c.hsys;
    s.n = n;
    s.nc = n_core;
    s.na = n_act;
    s.nv = n_virt;
    s.nalpha = n_alpha;
    s.nbeta = n_beta;
    s.nca = n_core + n_act;
    s.nav = n_act + n_virt;
    if (walk_plan(&c, s)) return 0;
    c.nref = n_ref;
    WalkNeed need;
    need.add(&c);
    return (long long)work_size(256, need, 0, 0).bytes;
}

int mrq_internal_sync(mrq_ctx* ctx) { return sync_stream(ctx); }

