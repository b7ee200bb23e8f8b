"""The sums that the walk's own kernels form, determinant by determinant.

`debug_local` evaluates a determinant with lists of its own, so its records pin the formulas but not the kernels
of a walk step (shared rows, groups of first-order neighbours, task groups).  Here the walk itself gives them: with
one walker per group and a burn-in of all steps but the last, the accumulators hold each walker's last step,
W = 1/S, E = E_L/S, N_l = 1/(S c_l^2) and U_l = num/(S c_l^2) of the determinant it stood on.  They are compared
with the oracle, or, at 56 and 104 orbitals, for every walker with debug_local, whose values the parity tests hold
against the oracle there.

Tolerance: S is a sum of non-negative terms, E_L and the numerator cancel down from sums of size |H_nn| + S; both
sides add at most 4e6 FP64 terms whose overlaps are sums of a few hundred, in different orders: 1e-10 of that size,
the repository's tolerance for these quantities.
"""
import numpy as np
import pytest

import oracle as O
import synthetic as S

pytestmark = pytest.mark.gpu

G = 64
RTOL = 1e-10


def _last_steps(ctx, n, steps, seed):
    """Determinants on which n <= 64 walkers stood at their last of `steps` steps, and that step's S, E_L, numerator."""
    ctx.walkers_init(ctx.params(n, steps, burn_in=steps - 1, seed=seed, n_groups=G))
    if steps > 1:
        ctx.walkers_advance(steps - 1)
    dets, _ = ctx.walkers(n)
    ctx.walkers_advance(1)
    acc = ctx.accumulators(G)
    c = ctx.coeffs()
    rate = 1.0 / acc["W"][:n]
    label = np.array([np.flatnonzero(acc["N"][g])[0] for g in range(n)])
    assert all(np.count_nonzero(acc["N"][g]) == 1 for g in range(n))
    norm = acc["N"][np.arange(n), label] * c[label] ** 2 * rate             # 1 for each
    return dets, label, rate, acc["E"][:n] * rate, acc["U"][np.arange(n), label] * c[label] ** 2 * rate, norm


def _compare(got, want):
    dets, label, rate, e_local, num, norm = got
    for i, r in enumerate(want):
        size = abs(r["Hnn"]) + abs(r["HDnn"]) + r["S"]
        assert label[i] == r["label"], i
        assert abs(norm[i] - 1.0) <= 1e-14, i                               # three products and a quotient
        assert abs(rate[i] - r["S"]) <= RTOL * r["S"], (i, rate[i], r["S"])
        assert abs(e_local[i] - r["EL"]) <= RTOL * size, (i, e_local[i], r["EL"])
        assert abs(num[i] - r["num"]) <= RTOL * size, (i, num[i], r["num"])


def _debug(ctx, dets):
    loc, _ = ctx.debug_local(dets)
    return [dict(S=x["S"], EL=x["e_local"], num=x["num"], Hnn=x["h_nn"], HDnn=x["hd_nn"], label=x["label"]) for x in loc]


# rows and first-order groups just below, at and above 1,024 entries (n_virt^2 for two virtual electrons of
# opposite spin, of which a first-order determinant may hold one), open shells, two words per spin, one orbital
# of a kind
SYSTEMS = [(1, 2, 31, 2, 2), (1, 2, 32, 2, 2), (2, 2, 33, 3, 3), (1, 3, 32, 2, 3), (2, 4, 6, 4, 4), (4, 2, 1, 5, 5), (1, 1, 1, 1, 2),
           (62, 3, 5, 64, 63)]


@pytest.mark.parametrize("nc,na,nv,a,b", SYSTEMS)
def test_last_steps_match_the_oracle(nc, na, nv, a, b):
    import paper_1909_06935_gb300 as P
    s = S.make_system(nc, na, nv, a, b, rank=12, seed=700 + nc + nv, chol_sigma=0.1)
    orc = O.Oracle.from_system(s)
    n = 12 if nc > 10 else 48
    with P.Context.from_system(s) as ctx:
        for steps in (1, 3, 6):
            got = _last_steps(ctx, n, steps, 5 + steps)
            want = {d.tobytes(): orc.local(d) for d in np.unique(got[0], axis=0)}
            _compare(got, [want[d.tobytes()] for d in got[0]])


@pytest.mark.parametrize("name", ["cas10_56o", "sci_104o_cas14"])
def test_last_steps_match_the_evaluated_determinants_at_full_size(name):
    import paper_1909_06935_gb300 as P
    with P.Context.from_system(S.workload(name)) as ctx:
        kinds = set()
        for steps in (1, 4, 9):
            got = _last_steps(ctx, G, steps, 40 + steps)
            once, back = np.unique(got[0], axis=0, return_inverse=True)
            loc = _debug(ctx, once)
            _compare(got, [loc[k] for k in back.ravel()])
            kinds |= {bool(x) for x in got[1]}
        assert kinds == {False, True}                                       # CAS and first-order determinants


@pytest.mark.parametrize("walkers", [4127, 4128, 4129])
def test_full_task_groups_match_the_oracle_walk(walkers):
    """From 4,096 walkers on a task group holds 32: at the start all walkers stand on one determinant, and the last
    group has 31, 32 and 1 of them."""
    import paper_1909_06935_gb300 as P
    s = S.make_system(2, 3, 4, 4, 4, rank=12, seed=77, chol_sigma=0.1)
    steps = 4
    ref = O.Oracle.from_system(s).sample(walkers, steps, 1, 6, 8, trajectory=True)
    with P.Context.from_system(s) as ctx:
        ctx.sample(ctx.params(walkers, steps, burn_in=1, seed=6, n_groups=8))
        assert np.array_equal(ctx.walkers(walkers)[0], ref["trajectory"][:, -1, :])
        acc = ctx.accumulators(8)
    assert np.array_equal(acc["type_steps"], ref["type_steps"])
    for key in ("N", "U", "W", "E"):
        x, y = np.asarray(acc[key]), np.asarray(ref[key])
        assert np.all(np.abs(x - y) <= 1e-14 + RTOL * np.maximum(np.abs(x), np.abs(y))), key
