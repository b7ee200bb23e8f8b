"""Candidates whose clocks agree to 5e-5 meet in one walker's record from 4,096 warp tasks at once.

FP32 clocks leave the order of all of them open, so every comparison takes both candidates' exact clocks, from the
record's excitation and t: these have to belong together whenever they are read.  The winner is that of the exact
clocks (numpy, 4 roundings), whatever the number of tasks.
"""
import numpy as np
import pytest

from tests.test_gpu_race_winner import _check, _draws, _neighbours

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [1, 2, 3, 4])
@pytest.mark.parametrize("n,slices", [(4096 * 64, 4096), (4096 * 64 - 31, 1024), (640, 10)])
def test_near_ties_from_many_tasks(seed, n, slices):
    rng = np.random.default_rng(seed)
    exc, psi, walker, step = _neighbours(n, rng), 0.25, 11 * seed, 3
    clock = 0.125 * (1.0 + rng.uniform(0.0, 5e-5, n))
    t = psi * -np.log(_draws(exc, step, walker, seed)) / clock
    _check(exc, t, psi, seed, np.array([walker], np.uint32), np.array([step], np.uint32), slices)
