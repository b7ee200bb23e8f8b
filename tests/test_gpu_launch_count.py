"""mrq_kernel_launches counts the kernels of walks and finalizes, replayed graphs included."""
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu


def test_kernels_are_counted_where_they_are_launched():
    import paper_1909_06935_gb300 as P
    with P.Context.from_system(S.workload("tiny_12o_cas4")) as c:
        c.walkers_init(c.params(64, 6, seed=1, n_groups=4))
        n0 = c.kernel_launches
        c.walkers_advance(2)               # a launch: 1; a step of one segment and one wave of each kind: 5 + 3 + 5 + 1
        assert c.kernel_launches - n0 == 1 + 2 * 14
        c.finalize()
        assert c.kernel_launches - n0 == 1 + 2 * 14 + 3
        counts = []
        for graph in (False, True, True):
            c.set_launch(0, 3, graph)
            n1 = c.kernel_launches
            P.batch_advance([c], 7)        # two launches of three steps and one of one
            counts.append(c.kernel_launches - n1)
        assert counts == [3 + 7 * 14] * 3
