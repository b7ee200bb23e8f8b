"""The winner of the move race is that of the exact FP64 clocks, whatever the sizes of the rates.

The walk's race (screen, FP32 clocks, tasks that meet in one record per walker) against -ln(u)/Gamma in numpy:
amplitudes and elements whose rates, clocks or both lie outside FP32's range, as well as ordinary ones.  numpy's
and the device's logarithms differ by at most an ulp each, so a winner's clock may exceed the smallest by
4 roundings.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _draws(exc, step, walker, seed):
    """u of Philox4x32-10 (Salmon et al., SC'11) with counter (exc, step, walker, 0): (k + 1) 2^-53 of its top 53 bits."""
    lo = np.uint64(0xFFFFFFFF)
    z = np.zeros(len(exc), np.uint64)
    c0, c1, c2, c3 = exc.astype(np.uint64), z + np.uint64(step), z + np.uint64(walker), z
    k0, k1 = np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)
    for _ in range(10):
        p0, p1 = c0 * np.uint64(0xD2511F53), c2 * np.uint64(0xCD9E8D57)
        c0, c1, c2, c3 = (p1 >> np.uint64(32)) ^ c1 ^ k0, p1 & lo, (p0 >> np.uint64(32)) ^ c3 ^ k1, p0 & lo
        k0, k1 = (k0 + np.uint64(0x9E3779B9)) & lo, (k1 + np.uint64(0xBB67AE85)) & lo
    k = (c0 << np.uint64(32) | c1) >> np.uint64(11)
    return (k.astype(np.float64) + 1.0) * 2.0 ** -53


def _clocks(exc, t, psi, step, walker, seed):
    with np.errstate(divide="ignore"):
        return np.where(t != 0.0, -np.log(_draws(exc, step, walker, seed)) / np.abs(t * (1.0 / psi)), np.inf)


def _check(exc, t, psi, seed, walkers, steps, slices):
    import paper_1909_06935_gb300 as P
    with P.Context() as ctx:
        won = ctx.race(exc, t, psi, seed, walkers, steps, slices)
    at = {int(e): i for i, e in enumerate(exc)}
    for i, (w, s) in enumerate(zip(walkers, steps)):
        c = _clocks(exc, t, psi, int(s), int(w), seed)
        got = c[at[int(won[i])]]
        assert got <= c.min() * (1.0 + 4 * 2.0 ** -52), (i, got, c.min())


def _neighbours(n, rng):
    return rng.permutation(1 << 24)[:n].astype(np.uint32) * np.uint32(7) + np.uint32(3)


# amplitude of the walkers' determinant; scale of t
SCALES = [(0.3, 1.0), (1e-12, 1e-9), (1e-36, 1e-3), (1e-45, 1.0), (1e-50, 1e-6), (1e-80, 1e-5), (1e-300, 1e-2),
          (1e30, 1e-9), (1e12, 1e-40), (1e40, 1e-2), (1e-20, 1e15)]


@pytest.mark.parametrize("psi,scale", SCALES)
@pytest.mark.parametrize("n,slices", [(1, 1), (63, 1), (64, 3), (65, 2), (3000, 7)])
def test_winner_is_that_of_the_exact_clocks(psi, scale, n, slices):
    rng = np.random.default_rng(n + 17 * slices)
    t = scale * rng.standard_normal(n) * np.exp(rng.uniform(-6.0, 0.0, n))
    if n > 1:
        t[rng.integers(0, n, n // 5)] = 0.0
    if not t.any():
        t[0] = scale
    walkers = np.concatenate([np.arange(33), [2 ** 32 - 1]]).astype(np.uint32)
    steps = (np.arange(len(walkers)) % 5).astype(np.uint32)
    _check(_neighbours(n, rng), t, psi, 0x123456789ABCDEF + n, walkers, steps, slices)


def test_rates_of_very_different_sizes_meet_in_one_race():
    rng = np.random.default_rng(3)
    t = 10.0 ** rng.uniform(-80.0, 40.0, 2000)
    walkers = np.arange(40, dtype=np.uint32)
    for psi in (1.0, 1e-30, 1e30):
        _check(_neighbours(2000, rng), t, psi, 99, walkers, np.zeros(40, np.uint32), 5)
