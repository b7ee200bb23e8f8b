"""A context that has run out of memory says so, and can be used again.

Walkers that no device holds are asked for (the allocation is refused; nothing runs); the context then has no
walkers, whatever it had before, and starts ordinary ones as a fresh context would.
"""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

MRQ_OOM, MRQ_NOT_LOADED = -4, -2


@pytest.mark.parametrize("huge", [1 << 34, 1 << 60])
def test_walkers_that_do_not_fit_leave_a_usable_context(huge):
    import paper_1909_06935_gb300 as P
    s = S.workload("tiny_12o_cas4")
    with P.Context.from_system(s) as ctx:
        p = ctx.params(64, 6, burn_in=1, seed=3, n_groups=4)
        want = ctx.sample(p)
        dets = ctx.walkers(64)[0]
        with pytest.raises(P.MRQError) as e:
            ctx.walkers_init(ctx.params(huge, 1, n_groups=4))
        assert e.value.code == MRQ_OOM
        with pytest.raises(P.MRQError) as e:
            ctx.walkers_advance(1)
        assert e.value.code == MRQ_NOT_LOADED
        got = ctx.sample(p)
        assert np.array_equal(ctx.walkers(64)[0], dets)
        for key in ("e2", "e2_sigma", "e_var", "a0sq", "walker_steps"):
            assert got[key] == want[key], key
