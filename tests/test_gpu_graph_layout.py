"""A captured batch graph is replayed for the layout that it was captured for, and for no other.

A graph's kernels hold the walk's workspace by value: where its row buffers lie and how large they are.
Both follow the batch's systems, also where the sizes that the launch shapes follow - longest candidate
list, operator, slices, row references, groups - are another member's and stay.  Batches whose members
change, and contexts that are loaded anew, therefore walk as without a graph, bit for bit.
"""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

STEPS, G = 6, 4


def _walk(ctxs, walkers, seeds, graph):
    import paper_1909_06935_gb300 as P
    for c, nw, seed in zip(ctxs, walkers, seeds):
        c.set_launch(0, 3, graph)
        c.walkers_init(c.params(nw, STEPS, burn_in=1, seed=seed, n_groups=G))
    P.batch_advance(ctxs, STEPS)
    return [(c.walkers(nw)[0], c.accumulators(G)) for c, nw in zip(ctxs, walkers)]


def _same(a, b):
    for (da, aa), (db, ab) in zip(a, b):
        assert np.array_equal(da, db)
        for key in ("N", "U", "W", "E", "type_steps"):
            assert np.array_equal(aa[key], ab[key]), key


def test_partner_with_longer_rows_does_not_replay_the_other_partners_graph():
    import paper_1909_06935_gb300 as P
    # the lead has the longest list, operator, slices, references and groups; its neighbours are 13,008 per
    # CAS determinant, the partners' 3,192 and 27,558
    lead = P.Context.from_system(S.make_system(2, 8, 12, 6, 6, rank=20, seed=301, chol_sigma=0.06))
    small = P.Context.from_system(S.make_system(2, 4, 10, 4, 4, rank=16, seed=302, chol_sigma=0.08))
    large = P.Context.from_system(S.make_system(5, 3, 20, 7, 6, rank=16, seed=303, chol_sigma=0.08))
    walkers, seeds = [96, 64], [5, 6]
    ref_large = _walk([lead, large], walkers, seeds, False)        # the workspace has the larger size from here on
    ref_small = _walk([lead, small], walkers, seeds, False)
    for _ in range(2):
        _same(_walk([lead, small], walkers, seeds, True), ref_small)
        _same(_walk([lead, large], walkers, seeds, True), ref_large)
    for c in (lead, small, large):
        c.close()


def test_lead_loaded_with_fewer_electrons_captures_anew():
    import paper_1909_06935_gb300 as P
    # the same orbitals with 3 + 3 and 1 + 1 active electrons: lists, operator, references and groups of
    # one size, 360 and 198 neighbours
    systems = [S.make_system(1, 4, 3, 1 + e, 1 + e, rank=10, seed=311, chol_sigma=0.08) for e in (3, 1)]
    ref = []
    for s in systems:
        with P.Context.from_system(s) as c:
            ref.append(_walk([c], [300], [9], False))
    with P.Context() as c:
        for k in (0, 1, 0, 1):
            s = systems[k]
            c.load_hamiltonian(s.n_core, s.n_act, s.n_virt, s.n_alpha, s.n_beta, s.h1, s.eri, s.e_nuc)
            c.load_reference(s.dets, s.coeffs)
            c.set_coeffs(s.c)
            for _ in range(2):
                _same(_walk([c], [300], [9], True), ref[k])
