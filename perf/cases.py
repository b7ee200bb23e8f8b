"""What this library is used for, as timed cases.

A user loads a Hamiltonian and a reference once, then walks: `Context.sample` from a fresh start,
`walkers_advance` + `finalize` in blocks (convergence checks, blocking analysis), `sample_batch`
over several systems, and the SC-MRCI(s) loop of walk, gradient and AMSGrad step.  Each case is one
such call on a seeded synthetic system; sizes are those of the named workloads, the batched and
served mixes of `synthetic`, and shapes between them.
"""
import itertools
import math

import numpy as np
import torch

import paper_1909_06935_gb300 as P
import synthetic as S

_SYS = ("nc", "na", "nv", "ea", "eb")          # core, active, virtual orbitals; active alpha, beta electrons


def _case(name, kind, nc, na, nv, ea, eb, walkers, steps, burn=0, strings=0, frozen=False, systems=1):
    return dict(name=name, kind=kind, nc=nc, na=na, nv=nv, ea=ea, eb=eb, walkers=walkers, steps=steps, burn=burn,
                strings=strings, frozen=frozen, systems=systems)


def listed():
    return [
        # the smallest system (12 orbitals, CAS(4e,4o)) sampled from a fresh start: launches count
        _case("sample_12o", "sample", 2, 4, 6, 2, 2, 128, 24, burn=4),
        # the served mix: small requests of 12-18 orbitals advanced together, 256 walkers each
        _case("batch_served", "batch", 2, 4, 10, 2, 2, 256, 16, burn=4, systems=8),
        # the batched mix: systems of different widths and active spaces in one call
        _case("batch_mixed", "batch", 4, 8, 60, 4, 4, 96, 2, systems=6),
        # the paper's own implementation correlates no core: frozen-core coefficients, CAS(8e,8o)
        _case("frozen_34o", "sample", 4, 8, 22, 4, 4, 512, 6, burn=1, frozen=True),
        # open shell, odd counts, two words per spin, a ragged number of walkers
        _case("open_67o", "sample", 3, 7, 57, 4, 3, 333, 3),
        # one SC-MRCI(s) iteration: walk, energy gradient, AMSGrad update
        _case("mrci_30o", "mrci", 4, 6, 20, 3, 3, 512, 16, burn=4),
        # a short fresh run on the 56-orbital CAS(10e,10o) workload
        _case("sample_56o", "sample", 6, 10, 40, 5, 5, 512, 8, burn=2),
        # the headline: one block of the running walk (step + finalize) of 4,096 walkers
        _case("block_56o", "block", 6, 10, 40, 5, 5, 4096, 1),
        # the largest named system: 104 orbitals, 10^6-determinant selected-CI reference
        _case("block_104o", "block", 10, 14, 80, 7, 7, 1024, 1, strings=1000),
        # set-up of a system from host arrays: integrals, reference, coefficients
        _case("load_56o", "load", 6, 10, 40, 5, 5, 0, 0),
    ]


def _neighbours(c):
    """Singles and doubles of a CAS determinant (all of them stay in the CAS or the first-order space)."""
    oa, ob = c["nc"] + c["ea"], c["nc"] + c["eb"]
    n = c["nc"] + c["na"] + c["nv"]
    va, vb = n - oa, n - ob
    return oa * va + ob * vb + math.comb(oa, 2) * math.comb(va, 2) + math.comb(ob, 2) * math.comb(vb, 2) + oa * va * ob * vb


def draw(rng):
    """One more case: any of the kinds, sizes log-uniform, work bounded by the largest listed case's."""
    while True:
        kind = rng.choice(["sample", "sample", "block", "block", "mrci", "batch", "load"])
        na = rng.randint(4, 10)
        ea = rng.randint(max(1, na // 2 - 1), na // 2 + 1)
        eb = ea if na > 8 or rng.random() < 0.6 else max(1, ea - 1)
        nv = int(round(math.exp(rng.uniform(math.log(6), math.log(80)))))
        walkers = 0 if kind == "load" else int(round(math.exp(rng.uniform(math.log(32), math.log(4096)))))
        steps = 0 if kind == "load" else 1 if kind == "block" else rng.randint(1, 16)
        burn = rng.randint(0, steps // 2) if kind in ("sample", "batch", "mrci") else 0
        systems = rng.randint(2, 8) if kind == "batch" else 1
        if kind == "batch":
            na, nv = min(na, 8), min(nv, 60)
            ea = eb = min(ea, na // 2)
        c = _case("", kind, rng.randint(1, 10), na, nv, ea, eb, walkers, steps, burn=burn, systems=systems,
                  frozen=kind == "sample" and rng.random() < 0.3)
        del c["name"]
        if walkers * max(steps, 1) * systems * _neighbours(c) <= 4096 * 350_000:
            return c


# --------------------------------------------------------------------------- inputs

def _packed(L):
    """8-fold packed (pq|rs) of the Cholesky factors, formed on the GPU."""
    n = L.shape[1]
    dev = torch.as_tensor(L, device="cuda")
    r, q = torch.tril_indices(n, n, device="cuda")
    Lp = dev[:, r, q]
    M = Lp.T @ Lp
    i, j = torch.tril_indices(M.shape[0], M.shape[0], device="cuda")
    eri = M[i, j].contiguous()
    torch.cuda.synchronize()          # the context reads it on a stream of its own
    return eri


def _reference_device(c, h1, eri, strings):
    """A context whose reference is built on the device (selected CI over strings; every string: CAS-CI)."""
    ctx = P.Context()
    ne = c["nc"] + c["ea"]
    ctx.load_hamiltonian(c["nc"], c["na"], c["nv"], ne, ne, h1, eri)
    ref = ctx.sci_reference(strings, n_seed_strings=min(256, strings))
    return ctx, ref


def _system(c, seed):
    """A loaded context and its label coefficients for case c."""
    n = c["nc"] + c["na"] + c["nv"]
    sigma = 0.06 if n <= 20 else 0.05
    full = math.comb(c["na"], c["ea"])
    if c["ea"] == c["eb"] and (c["strings"] or full * full > 400):
        h1, L = S.make_integrals(c["nc"], c["na"], c["nv"], 3 * n, seed, chol_sigma=sigma)
        ctx, _ = _reference_device(c, h1, _packed(L), c["strings"] or full)
        co = S.psi_s_coeffs(S.n_labels(c["nc"], c["nv"]), seed + 17)
    else:
        s = S.make_system(c["nc"], c["na"], c["nv"], c["nc"] + c["ea"], c["nc"] + c["eb"], 3 * n, seed, chol_sigma=sigma)
        ctx, co = P.Context.from_system(s), s.c
    if c["frozen"]:
        co = P.frozen_core_coeffs(co, c["nc"], c["nv"])
    ctx.set_coeffs(co)
    return ctx, co


def _batch_members(c, seed):
    """The systems of a batch: sizes spread around the case's, as the served and batched mixes do."""
    rng = np.random.Generator(np.random.PCG64(c["na"] * 1000 + c["nv"]))
    out = []
    for k in range(c["systems"]):
        na = c["na"] if c["na"] <= 4 else int(rng.choice([max(4, c["na"] - 2), c["na"]]))
        ea = min(c["ea"], na // 2)
        nv = max(2, int(round(c["nv"] * rng.uniform(0.6, 1.2))))
        out.append((dict(c, na=na, ea=ea, eb=ea, nv=nv, nc=max(1, c["nc"] - k % 2)),
                    max(32, c["walkers"] * (1 + k % 3) // 2), seed + 101 * k))
    return out


def prepare(case, seed):
    c = case
    if c["kind"] == "load":
        ne = c["nc"] + c["ea"]
        n = c["nc"] + c["na"] + c["nv"]
        if c["ea"] != c["eb"]:
            s = S.make_system(c["nc"], c["na"], c["nv"], ne, c["nc"] + c["eb"], 3 * n, seed, chol_sigma=0.05)
            return dict(c=c, ctx=P.Context(), ea=ne, eb=c["nc"] + c["eb"], h1=s.h1, eri=s.eri, dets=s.dets, co=s.coeffs, cl=s.c)
        h1, L = S.make_integrals(c["nc"], c["na"], c["nv"], 3 * n, seed, chol_sigma=0.05)
        ctx, ref = _reference_device(c, h1, _packed(L), math.comb(c["na"], c["ea"]))
        h1, eri = ctx.read_hamiltonian()
        core = np.uint64((1 << c["nc"]) - 1)
        words = core | (ref["strings"].astype(np.uint64) << np.uint64(c["nc"]))
        m, W = len(words), (n + 63) // 64
        dets = np.zeros((m * m, 2 * W), np.uint64)
        dets[:, 0] = np.repeat(words, m)
        dets[:, W] = np.tile(words, m)
        return dict(c=c, ctx=ctx, ea=ne, eb=ne, h1=h1, eri=eri, dets=dets, co=np.ascontiguousarray(ref["coeffs"]).ravel(),
                    cl=S.psi_s_coeffs(S.n_labels(c["nc"], c["nv"]), seed + 17))
    if c["kind"] == "batch":
        ctxs, ps = [], []
        for cc, walkers, sd in _batch_members(c, seed):
            ctx, _ = _system(cc, sd)
            ctxs.append(ctx)
            ps.append(ctx.params(walkers, c["steps"], burn_in=c["burn"], seed=sd, n_groups=16))
        return dict(c=c, ctxs=ctxs, ps=ps)
    ctx, co = _system(c, seed)
    st = dict(c=c, ctx=ctx, p=ctx.params(c["walkers"], c["steps"], burn_in=c["burn"], seed=seed, n_groups=16))
    if c["kind"] == "block":
        # a walk that has left its start determinant
        ctx.walkers_init(st["p"])
        ctx.walkers_advance(3)
        ctx.finalize()
    if c["kind"] == "mrci":
        st["co"] = co
    return st


# --------------------------------------------------------------------------- one pass

def _numbers(res):
    return {k: np.asarray(v) for k, v in res.items() if k not in ("seconds", "walk_launches", "reserved")}


def run(state):
    c = state["c"]
    if c["kind"] == "load":
        ctx = state["ctx"]
        ctx.load_hamiltonian(c["nc"], c["na"], c["nv"], state["ea"], state["eb"], state["h1"], state["eri"])
        ctx.load_reference(state["dets"], state["co"])
        ctx.set_coeffs(state["cl"])
        return _numbers(ctx.setup_info())
    if c["kind"] == "batch":
        res = [_numbers(r) for r in P.sample_batch(state["ctxs"], state["ps"])]
        return {k: np.stack([r[k] for r in res]) for k in res[0]}
    ctx = state["ctx"]
    if c["kind"] == "block":
        ctx.walkers_advance(c["steps"])
        res = ctx.finalize()
        dets, psi = ctx.walkers(c["walkers"])
        return dict(res=_numbers(res), dets=dets.view(np.int64), psi=psi)
    if c["kind"] == "mrci":
        ctx.set_coeffs(state["co"])
        res = ctx.sample(state["p"])
        grad, energy = ctx.mrci_gradient()
        ctx.amsgrad_step(0.01)
        return dict(res=_numbers(res), grad=grad, energy=np.asarray(energy), coeffs=ctx.coeffs())
    return _numbers(ctx.sample(state["p"]))


def work(case):
    """Bytes: the packed integrals, the reference (occupations and coefficient) and the label
    coefficients once, and every walker's record (determinant, amplitude, step data) in and out.
    Flops: per neighbour of a walker the product of its element, overlap and coefficient, and the
    sums of t and |t| (4); the overlaps themselves are shared between walkers in a way that depends
    on the walk, so none are counted."""
    c = case
    members = [(cc, w) for cc, w, _ in _batch_members(c, 0)] if c["kind"] == "batch" else [(c, c["walkers"])]
    by = fl = 0.0
    for cc, w in members:
        n = cc["nc"] + cc["na"] + cc["nv"]
        npair = n * (n + 1) // 2
        nref = c["strings"] ** 2 or math.comb(cc["na"], cc["ea"]) * math.comb(cc["na"], cc["eb"])
        by += 4.0 * npair * (npair + 1) + 16.0 * nref + 8.0 * S.n_labels(cc["nc"], cc["nv"]) + 192.0 * w * c["steps"]
        fl += 4.0 * w * c["steps"] * _neighbours(cc)
        if c["kind"] == "load":   # E0: every reference determinant against its active singles and doubles
            va, vb = cc["na"] - cc["ea"], cc["na"] - cc["eb"]
            fl += 2.0 * nref * (cc["ea"] * va + cc["eb"] * vb + math.comb(cc["ea"], 2) * math.comb(va, 2)
                                + math.comb(cc["eb"], 2) * math.comb(vb, 2) + cc["ea"] * va * cc["eb"] * vb)
    return {"bytes": by, "flops": fl}


# --------------------------------------------------------------------------- 64-bit values

def exact(case, seed):
    c = case
    if c["kind"] == "load":
        return _exact_setup(c, prepare(c, seed))
    n = c["nc"] + c["na"] + c["nv"]
    if c["kind"] != "sample" or n > 12 or c["na"] > 4 or c["walkers"] * c["steps"] > 4000 or c["ea"] != c["eb"]:
        return None               # thousands of neighbours per step and walker: far over 20 seconds in numpy
    s = S.make_system(c["nc"], c["na"], c["nv"], c["nc"] + c["ea"], c["nc"] + c["eb"], 3 * n, seed, chol_sigma=0.06)
    cl = s.c.copy()
    if c["frozen"]:
        cl[1 + 2 * c["nv"] + math.comb(2 * c["nv"], 2):] = 0.0
    return _exact_walk(s, cl, c, seed)


def _square(eri, n):
    """(pq|rs) as an n^4 array."""
    npair = n * (n + 1) // 2
    M = np.zeros((npair, npair))
    i, j = np.tril_indices(npair)
    M[i, j] = M[j, i] = eri
    p = np.arange(n)
    P2 = np.maximum(p[:, None], p) * (np.maximum(p[:, None], p) + 1) // 2 + np.minimum(p[:, None], p)
    return M[P2[:, :, None, None], P2[None, None]]


def _dyall(h1, g, nc, na, gamma):
    """Core Fock operator, core energy and the generalised-Fock diagonal."""
    hc = h1 + 2.0 * np.einsum("pqii->pq", g[:, :, :nc, :nc]) - np.einsum("piiq->pq", g[:, :nc, :nc, :])
    ecore = float(np.trace(h1[:nc, :nc]) + np.trace(hc[:nc, :nc]))
    a = slice(nc, nc + na)
    eps = np.diag(hc) + np.einsum("pptu,tu->p", g[:, :, a, a], gamma) - 0.5 * np.einsum("ptup,tu->p", g[:, a, a, :], gamma)
    return hc, ecore, eps


def _exact_setup(c, st):
    n, nc, na = c["nc"] + c["na"] + c["nv"], c["nc"], c["na"]
    dets, co, W = st["dets"], st["co"], (n + 63) // 64
    g = _square(st["eri"], n)
    act = (1 << na) - 1
    a = ((dets[:, 0] >> np.uint64(nc)) & np.uint64(act)).astype(np.int64)
    b = ((dets[:, W] >> np.uint64(nc)) & np.uint64(act)).astype(np.int64)
    sa, sb = np.unique(a), np.unique(b)
    C = np.zeros((len(sa), len(sb)))
    C[np.searchsorted(sa, a), np.searchsorted(sb, b)] = co

    def excited(strs, X):          # E_tu X along the first index, for every (t, u)
        out = np.zeros((na * na,) + X.shape)
        for t, u in itertools.product(range(na), repeat=2):
            for i, s in enumerate(strs.tolist()):
                if s >> u & 1 and (t == u or not s >> t & 1):
                    lo, hi = min(t, u), max(t, u)
                    sign = -1.0 if bin(s >> (lo + 1) & ((1 << max(0, hi - lo - 1)) - 1)).count("1") & 1 else 1.0
                    out[t * na + u, np.searchsorted(strs, s ^ (1 << u) | (1 << t))] += sign * X[i]
        return out

    D = (excited(sa, C) + excited(sb, np.ascontiguousarray(C.T)).transpose(0, 2, 1)).reshape(na * na, -1)
    norm = float(co @ co)
    gamma = (D @ C.ravel() / norm).reshape(na, na)
    hc, ecore, eps = _dyall(st["h1"], g, nc, na, gamma)
    ga = g[nc:nc + na, nc:nc + na, nc:nc + na, nc:nc + na]
    k = hc[nc:nc + na, nc:nc + na] - 0.5 * np.einsum("tvvu->tu", ga)
    DD = (D @ D.T).reshape(na, na, na, na)                 # <E_ut phi | E_vw phi>
    e0 = ecore + float((k * gamma).sum() + 0.5 * np.einsum("tuvw,utvw->", ga, DD) / norm)
    return dict(e0=np.asarray(e0), norm0=np.asarray(norm), e_core=np.asarray(ecore), sum_eps_core=eps[:nc].sum(), start=None,
                eps=eps, gamma=gamma)


def _philox(exc, step, walker, seed):
    """First two words of Philox4x32-10 (Salmon et al., SC'11) with counter (exc, step, walker, 0)."""
    u32 = np.uint64(0xFFFFFFFF)
    z = np.zeros_like(exc, dtype=np.uint64)
    c0, c1, c2, c3 = exc.astype(np.uint64), z + np.uint64(step), z + np.uint64(walker), z
    k0, k1 = np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)
    for _ in range(10):
        p0, p1 = c0 * np.uint64(0xD2511F53), c2 * np.uint64(0xCD9E8D57)
        c0, c1, c2, c3 = (p1 >> np.uint64(32)) ^ c1 ^ k0, p1 & u32, (p0 >> np.uint64(32)) ^ c3 ^ k1, p0 & u32
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & u32, (k1 + np.uint64(0xBB67AE85)) & u32
    return c0, c1


def _exact_walk(s, cl, c, seed):
    """The walk in numpy: every element by Slater-Condon on occupation sets, every overlap as a sum
    over the whole reference, the first-reaction race with Philox clocks, the averages of Eq. 4-16."""
    n, nc, na, nv = s.n_orb, s.n_core, s.n_act, s.n_virt
    h1, g = s.h1, _square(s.eri, n)
    so = [(x // n, x % n) for x in range(2 * n)]           # spin orbital -> (spin, orbital); alpha first
    det = lambda w: int(w[0]) | int(w[1]) << n             # noqa: E731
    ref = {det(d): float(x) for d, x in zip(s.dets, s.coeffs)}
    bits = lambda d: [x for x in range(2 * n) if d >> x & 1]   # noqa: E731

    def between(d, x, y):
        x, y = min(x, y), max(x, y)
        return bin(d >> (x + 1) & ((1 << max(0, y - x - 1)) - 1)).count("1")

    def two(p, q, r, t):                                   # <pq||rt> over spin orbitals
        (sp, p), (sq, q), (sr, r), (st, t) = so[p], so[q], so[r], so[t]
        return (g[p, r, q, t] if sp == sr and sq == st else 0.0) - (g[p, t, q, r] if sp == st and sq == sr else 0.0)

    def diag(d, hop):
        o = bits(d)
        return sum(hop[so[x][1], so[x][1]] for x in o) + sum(two(x, y, x, y) for x, y in itertools.combinations(o, 2))

    def elem(d, rem, add, hop, occ):                       # <d'|H|d>, d' = d with rem -> add
        if len(rem) == 1:
            (x,), (y,) = rem, add
            if so[x][0] != so[y][0]:
                return 0.0
            v = hop[so[y][1], so[x][1]] + sum(two(y, j, x, j) for j in occ)
            return -v if between(d, x, y) & 1 else v
        (x, y), (a, b) = rem, add
        sign = between(d, x, a) + between(d ^ 1 << x ^ 1 << a, y, b)
        v = two(a, b, x, y)
        return -v if sign & 1 else v

    def split(d):                                          # core holes and virtual electrons
        H = [sg * nc + i for sg in (0, 1) for i in range(nc) if not d >> (sg * n + i) & 1]
        V = [sg * nv + i for sg in (0, 1) for i in range(nv) if d >> (sg * n + nc + na + i) & 1]
        return H, V

    def rank(xs, m):
        return 0 if not xs else 1 + xs[0] if len(xs) == 1 else 1 + m + xs[1] * (xs[1] - 1) // 2 + xs[0]

    nP = 1 + 2 * nv + math.comb(2 * nv, 2)
    label = lambda H, V: rank(H, 2 * nc) * nP + rank(V, 2 * nv)   # noqa: E731
    gamma = np.zeros((na, na))
    for d, x in ref.items():
        for t, u, sg in itertools.product(range(na), range(na), (0, 1)):
            a, b = sg * n + nc + t, sg * n + nc + u
            if d >> b & 1 and (t == u or not d >> a & 1):
                gamma[t, u] += x * ref.get(d ^ 1 << b | 1 << a, 0.0) * (-1.0) ** between(d, a, b)
    norm = sum(x * x for x in ref.values())
    gamma /= norm
    hc, ecore, eps = _dyall(h1, g, nc, na, gamma)
    acts = {sg * n + nc + t for sg in (0, 1) for t in range(na)}
    overlaps = {}

    def overlap(m):
        if m not in overlaps:
            o, v = bits(m), 0.0
            for k, x in ref.items():
                r, a = m & ~k, k & ~m
                if bin(r).count("1") <= 2 and (r or a):
                    v += x * elem(m, tuple(bits(r)), tuple(bits(a)), h1, o)
            overlaps[m] = v
        return overlaps[m]

    def psi(m, H, V):
        return cl[0] * ref.get(m, 0.0) if not H and not V else cl[label(H, V)] * overlap(m)

    memo = {}

    def local(d):
        if d in memo:
            return memo[d]
        occ = bits(d)
        emp = [x for x in range(2 * n) if not d >> x & 1]
        H, V = split(d)
        l, pn = label(H, V), psi(d, H, V)
        ms, ex, ts, ps = [], [], [], []
        num = 0.0
        pairs = [((x,), (a,)) for x in occ for a in emp if so[x][0] == so[a][0]]
        pairs += [((x, y), (a, b)) for x, y in itertools.combinations(occ, 2) for a, b in itertools.combinations(emp, 2)
                  if so[x][0] + so[y][0] == so[a][0] + so[b][0]]
        for rem, add in pairs:
            m = d
            for x in rem + add:
                m ^= 1 << x
            Hm, Vm = split(m)
            if len(Hm) > 2 or len(Vm) > 2:
                continue
            pm = psi(m, Hm, Vm)
            hm = elem(d, rem, add, h1, occ)
            ms.append(m)
            ex.append(rem[0] | rem[-1] << 8 | add[0] << 16 | add[-1] << 24)
            ts.append(hm * pm)
            ps.append(pm)
            if l and set(rem) <= acts and set(add) <= acts:
                num += (elem(d, rem, add, hc, [j for j in occ if j in acts]) if len(rem) == 1 else hm) * pm
        t = np.array(ts)
        rate = np.abs(t / pn)
        active = [x for x in occ if x in acts]
        hd = (ecore + sum(hc[so[x][1], so[x][1]] for x in active) + sum(two(x, y, x, y) for x, y in itertools.combinations(active, 2))
              + sum(eps[nc + na + x % nv] for x in V) - sum(eps[x % nc] for x in H))
        memo[d] = (ms, np.array(ex, np.uint64), rate, ps, 1.0 / rate.sum(), diag(d, h1) + t.sum() / pn,
                   hd + num / pn if l else 0.0, l, 3 * len(H) + len(V), pn)
        return memo[d]

    G, L = 16, len(cl)
    N, U, Wg, E = np.zeros((G, L)), np.zeros((G, L)), np.zeros(G), np.zeros(G)
    types = np.zeros(9, np.int64)
    start = det(s.dets[int(np.argmax(np.abs(s.coeffs)))])
    for w in range(c["walkers"]):
        d = start
        for step in range(c["steps"]):
            ms, ex, rate, _, wt, el, num, l, ty, _ = local(d)
            if step >= c["burn"]:
                q = w % G
                Wg[q] += wt
                E[q] += wt * el
                N[q, l] += wt / cl[l] ** 2
                U[q, l] += wt * num / cl[l] ** 2
                types[ty] += 1
            x, y = _philox(ex, step, w, seed)
            k53 = (x << np.uint64(32) | y) >> np.uint64(11)
            with np.errstate(divide="ignore"):
                clock = -np.log((k53.astype(np.float64) + 1.0) * 2.0 ** -53) / rate
            clock[rate == 0.0] = np.inf
            d = ms[int(np.lexsort((ex, clock))[0])]
    e0 = sum(x * (x * diag(k, h1) + sum(ref[j] * elem(k, tuple(bits(k & ~j)), tuple(bits(j & ~k)), h1, bits(k))
                                        for j in ref if j != k and bin(k & ~j).count("1") <= 2)) for k, x in ref.items()) / norm
    ltype = np.array([3 * (0 if r == 0 else 1 if r <= 2 * nc else 2) + (0 if p == 0 else 1 if p <= 2 * nv else 2)
                      for r in range(L // nP) for p in range(nP)])

    def estimates(keep):
        Nk, Uk = N[keep].sum(0), U[keep].sum(0)
        seen = (Nk > 0) & (ltype > 0)
        ratio = Nk / Nk[0]
        use = seen & (ratio >= 1e-10)
        e2 = np.zeros(L)
        e2[use] = ratio[use] / (e0 - Uk[use] / Nk[use])
        by = lambda x: np.bincount(ltype, x, 9)            # noqa: E731
        tn, te = by(np.where(use, ratio, 0.0)), by(e2)
        return dict(e2=te.sum(), e_var=E[keep].sum() / Wg[keep].sum(), a0sq=cl[0] ** 2 * Nk[0] / Wg[keep].sum(), tn=tn, te=te,
                    scr=by(np.where(seen & ~use, 1.0, 0.0)), scrn=float(ratio[seen & ~use].sum()), vis=float(seen.sum()))

    every = np.arange(G)
    f = estimates(every)
    jack = [estimates(every != q) for q in range(G)]

    def sigma(key):
        v = np.array([j[key] for j in jack])
        return np.sqrt((G - 1) / G * ((v - v.mean(0)) ** 2).sum(0))

    return dict(e0=e0, e2=f["e2"], e2_sigma=sigma("e2"), e_var=f["e_var"], e_var_sigma=sigma("e_var"), a0sq=f["a0sq"],
                a0sq_sigma=sigma("a0sq"), e_mrci_q=f["e_var"] + (1 - f["a0sq"]) * (f["e_var"] - e0),
                type_norm=f["tn"], type_norm_sigma=sigma("tn"), type_e2=f["te"], type_e2_sigma=sigma("te"), type_screened=f["scr"],
                screened_norm=np.asarray(f["scrn"]), n_labels_visited=np.asarray(f["vis"]), type_steps=types, walker_steps=int(types.sum()),
                total_steps=c["walkers"] * c["steps"], status=0)
