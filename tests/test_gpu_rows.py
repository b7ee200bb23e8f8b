"""The walk's rows and neighbour groups at the edges of their cuts, against the oracle's walk.

The overlaps outside the CAS are computed in rows (one active remnant, all core holes and virtual
electrons of a class), cut into tasks of 1,024 entries; first-order determinants take theirs in groups
cut at 1,024 neighbours; the walkers of one determinant are raced in groups of at most 32.  The systems
put rows and groups just below, at and above those lengths, with odd orbital counts, one core or one
virtual orbital, an open shell, and an active block across a word boundary.  Trajectories are bit-exact
and accumulators within the repository's 1e-10 (each is a sum of at most a few thousand FP64 terms).
"""
import numpy as np
import pytest

import oracle as O
import synthetic as S

pytestmark = pytest.mark.gpu

# n_core, n_act, n_virt, n_alpha, n_beta, walkers: a remnant with one alpha electron less has
# n_core (n_virt^2 + n_virt (n_virt - 1) / 2) entries in its row of one hole and two virtual electrons
SYSTEMS = [
    (1, 2, 26, 2, 2, 33),      # 1,001 entries: one task, one walker more than a task group holds
    (1, 3, 27, 2, 3, 5),       # 1,080: two tasks, open shell
    (3, 2, 21, 4, 4, 64),      # 1,953: the cut falls inside the second spin group
    (2, 3, 37, 4, 3, 40),      # 4,070: four tasks
    (1, 1, 1, 1, 2, 3),        # one orbital of each kind
    (4, 2, 1, 5, 5, 7),        # one virtual orbital
    (62, 3, 5, 64, 63, 6),     # two words, active block across the boundary
]


@pytest.mark.parametrize("nc,na,nv,a,b,walkers", SYSTEMS)
def test_cut_rows_and_groups_match_the_oracle_walk(nc, na, nv, a, b, walkers):
    import paper_1909_06935_gb300 as P
    s = S.make_system(nc, na, nv, a, b, rank=12, seed=900 + nc + nv, chol_sigma=0.08)
    steps, G = 6, 4
    orc = O.Oracle.from_system(s)
    ref = orc.sample(walkers, steps, 1, 77, G, trajectory=True)
    with P.Context.from_system(s) as ctx:
        ctx.sample(ctx.params(walkers, steps, burn_in=1, seed=77, n_groups=G))
        dets, _ = ctx.walkers(walkers)
        acc = ctx.accumulators(G)
    assert np.array_equal(dets, ref["trajectory"][:, -1, :])
    assert np.array_equal(acc["type_steps"], ref["type_steps"])
    for key in ("N", "U", "W", "E"):
        x, y = np.asarray(acc[key]), np.asarray(ref[key])
        assert np.all(np.abs(x - y) <= 1e-14 + 1e-10 * np.maximum(np.abs(x), np.abs(y))), key
