"""The walk's workspace follows the determinants of a step, leaves memory to others, and changes no result.

A context's workspace takes at most an eighth of the free memory, so that many contexts walk on a nearly full
device; it grows when a step has had more determinants than its waves hold; and the walk is the same, bit for bit,
however many waves and segments it takes.
"""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

GIB = 1 << 30
G = 4


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _walk(ctx, walkers, steps, seed, block=None):
    ctx.walkers_init(ctx.params(walkers, steps, burn_in=1, seed=seed, n_groups=G))
    for _ in range(steps // (block or steps)):
        ctx.walkers_advance(block or steps)
        ctx.finalize()
    return ctx.walkers(walkers)[0], ctx.accumulators(G)


def _same(a, b):
    assert np.array_equal(a[0], b[0])
    for key in ("N", "U", "W", "E", "type_steps"):
        assert np.array_equal(a[1][key], b[1][key]), key


def test_contexts_on_a_nearly_full_device_all_walk():
    import torch
    import paper_1909_06935_gb300 as P
    s = S.make_system(8, 4, 48, 10, 10, rank=16, seed=401, chol_sigma=0.05)     # 2.9 MB of rows per determinant
    with P.Context.from_system(s) as c:
        want = _walk(c, 4096, 3, 8)
    torch.cuda.empty_cache()
    hold = torch.empty(max(0, _free() - 12 * GIB), dtype=torch.uint8, device="cuda")
    ctxs = []
    try:
        for k in range(8):
            c = P.Context.from_system(s)
            ctxs.append(c)
            c.walkers_init(c.params(4096, 3, burn_in=1, seed=8, n_groups=G))
            before = _free()
            c.walkers_advance(3)
            assert _free() >= before - before // 8 - (64 << 20), k      # (64 MiB: launch bookkeeping of the driver)
            c.finalize()
            _same((c.walkers(4096)[0], c.accumulators(G)), want)
        for c in ctxs:                                                  # and once more on what they have
            _same(_walk(c, 4096, 3, 8), want)
        # together they walk in the first one's workspace, and the others give theirs back
        for c in ctxs:
            c.walkers_init(c.params(4096, 3, burn_in=1, seed=8, n_groups=G))
        before = _free()
        P.batch_advance(ctxs, 3)
        assert _free() > before
        for c in ctxs:
            _same((c.walkers(4096)[0], c.accumulators(G)), want)
    finally:
        for c in ctxs:
            c.close()
        del hold
        torch.cuda.empty_cache()


def test_a_grown_workspace_changes_no_result():
    import paper_1909_06935_gb300 as P
    # 25 MB of rows per determinant, 400 reference determinants of about equal weight for 512 walkers to spread
    # over; the first wave holds a third of the walkers
    s = S.make_system(20, 6, 60, 23, 23, rank=12, seed=402, chol_sigma=0.07)
    rng = np.random.default_rng(4)
    s.coeffs = np.ascontiguousarray(rng.uniform(0.5, 1.0, len(s.coeffs)) * rng.choice([-1.0, 1.0], len(s.coeffs)))
    with P.Context.from_system(s) as c:
        want = _walk(c, 512, 12, 9)
    with P.Context.from_system(s) as c:
        c.walkers_init(c.params(512, 12, burn_in=1, seed=9, n_groups=G))
        free = [_free()]
        for _ in range(4):
            c.walkers_advance(3)
            c.finalize()
            free.append(_free())
        dets = np.unique(c.walkers(512)[0], axis=0)
        assert free[0] > free[1] > free[4], (free, len(dets))          # made, then grown
        _same((c.walkers(512)[0], c.accumulators(G)), want)
