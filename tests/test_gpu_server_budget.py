"""A server's requests and its walk workspace stay within the budget together, whatever is admitted and when.

The device's free memory is read after every round: the requests' own buffers and the workspace that their batch
walks in never exceed the budget by more than the allocator's granularity (32 MiB a request), also where requests
arrive while the first one's workspace fills what the budget had left; and each result is that of the request
alone, bit for bit, however few determinants and walkers the workspace holds.
"""
import numpy as np
import pytest

import synthetic as S

pytestmark = pytest.mark.gpu

MIB = 1 << 20
KEYS = ("e2", "e2_sigma", "e_var", "a0sq")


def _free():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _system(k):
    return S.make_system(8, 6, 48, 11, 11, rank=16, seed=410 + k, chol_sigma=0.05)


def _alone(s, walkers, steps, seed):
    import paper_1909_06935_gb300 as P
    with P.Context.from_system(s) as c:
        return c.sample(c.params(walkers, steps, burn_in=1, seed=seed, n_groups=8))


def test_requests_and_workspace_stay_within_the_budget_across_admissions():
    import paper_1909_06935_gb300 as P
    systems = [_system(k) for k in range(4)]
    steps, walkers = 8, 2048
    alone = [_alone(s, walkers, steps, 30 + k) for k, s in enumerate(systems)]
    base = _free()
    budget = 1600 * MIB
    srv = P.Server(max_active=8, hbm_budget_bytes=budget, steps_per_round=1)
    tickets, used = [], []
    for rnd in range(20):
        if rnd in (0, 2, 3, 5):                       # arrivals while the first one's workspace holds the rest
            k = len(tickets)
            tickets.append(srv.submit(systems[k], walkers, steps, burn_in=1, seed=30 + k, n_groups=8))
        srv.step()
        used.append(base - _free())
        assert used[-1] <= budget + 32 * MIB * len(tickets), (rnd, [u // MIB for u in used])
    assert used[0] > budget // 2                      # the workspace did take what was left
    for t, ref in zip(tickets, alone):
        st = srv.poll(t)
        assert st["state"] == "done", st
        assert np.array_equal(st["result"]["type_steps"], ref["type_steps"])
        for key in KEYS:
            assert st["result"][key] == ref[key], key
    assert srv.info()["bytes"] == 0
    srv.close()


def test_cancelled_leader_gives_its_workspace_back_before_the_next_walk():
    import paper_1909_06935_gb300 as P
    systems = [_system(k) for k in range(2)]
    want = _alone(systems[1], 1024, 4, 5)
    base = _free()
    budget = 1600 * MIB
    srv = P.Server(max_active=8, hbm_budget_bytes=budget, steps_per_round=1)
    a = srv.submit(systems[0], 1024, 100, seed=4, n_groups=8)
    b = srv.submit(systems[1], 1024, 4, burn_in=1, seed=5, n_groups=8)
    srv.step()
    srv.cancel(a)
    for _ in range(3):
        srv.step()
        assert base - _free() <= budget + 64 * MIB
    st = srv.poll(b)
    assert st["state"] == "done" and srv.poll(a)["state"] == "cancelled"
    for key in KEYS:
        assert st["result"][key] == want[key], key
    srv.close()


@pytest.mark.parametrize("steps_per_round", [1, 3])
def test_least_workspace_gives_the_same_walk(steps_per_round):
    """One determinant per wave, 256 walkers per segment, rows forgotten between waves, several steps a launch."""
    import paper_1909_06935_gb300 as P
    systems = [S.workload("tiny_12o_cas4"), S.make_system(3, 4, 12, 6, 5, rank=16, seed=431, chol_sigma=0.08),
               S.make_system(62, 3, 5, 64, 63, rank=10, seed=432, chol_sigma=0.06)]
    for k, s in enumerate(systems):
        walkers, steps = 700, 6
        want = _alone(s, walkers, steps, 50 + k)
        probe = P.Server(max_active=1, hbm_budget_bytes=1 << 40, steps_per_round=1)
        probe.submit(s, walkers, 9, seed=1, n_groups=8)
        probe.step()
        one = probe.info()["bytes"]                   # the request and its least workspace
        probe.close()
        srv = P.Server(max_active=1, hbm_budget_bytes=one, steps_per_round=steps_per_round)
        t = srv.submit(s, walkers, steps, burn_in=1, seed=50 + k, n_groups=8)
        for _ in range(steps):
            srv.step()
        st = srv.poll(t)
        assert st["state"] == "done", st
        assert np.array_equal(st["result"]["type_steps"], want["type_steps"])
        for key in KEYS:
            assert st["result"][key] == want[key], (k, key)
        srv.close()
