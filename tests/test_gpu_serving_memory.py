"""What served gradients take beside their footprint (stored sweeps, tables) is
decided by the request and the server's budget alone, counted while it is held,
and given back."""
import time

import numpy as np
import pytest

import oracle
from paper_2502_10685_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def l1(obs):
    return sum(abs(a) for a, _ in obs)


@pytest.fixture(scope="module")
def stab():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    from paper_2502_10685_gb300 import stab as S
    return S


def most_in_use(srv, ids):
    """The largest bytes_in_use seen until all the requests are done."""
    most = 0
    deadline = time.time() + 120
    while time.time() < deadline:
        st = srv.stats()
        most = max(most, st["bytes_in_use"])
        if st["completed"] == len(ids):
            return most
    pytest.fail("requests not done")


def test_nothing_reserved_for_sweeps_that_are_too_large(stab):
    """69 blocks of wire runs at n = 11: their vectors are more than a context
    keeps, the pair sweep runs, and only the request's footprint is taken."""
    c, obs = W.layered_ansatz(11, 3000, seed=61), W.obs_chain(11)
    srv = stab.Server()
    i = srv.submit(c, "grad", obs)
    most = most_in_use(srv, [i])
    assert srv.wait(i, timeout_s=120)["status"] == 0
    srv.close()
    assert most == stab.Server.footprint(c, "grad", obs)


# n = 8, 1,500 gates: 47 blocks, so at least 94 and at most 146 vectors of 512 KiB
# of stored sweeps (47 to 77 MB) beside a footprint below 10 MB
SWEEPS_FIT, SWEEPS_DO_NOT = 90 << 20, 40 << 20


@pytest.mark.parametrize("budget", [SWEEPS_FIT, SWEEPS_DO_NOT])
def test_gradient_alone_equals_in_mix_bit_for_bit(stab, budget):
    """Six gradients at once, under a budget that holds several footprints but
    the stored sweeps of one request alone (or of none): each result is that of
    the request served alone, on both sides of the rule."""
    obs = W.obs_chain(8)
    reqs = [W.layered_ansatz(8, 1500, seed=70 + k) for k in range(6)]
    fp = max(stab.Server.footprint(c, "grad", obs) for c in reqs)
    assert 3 * fp < SWEEPS_DO_NOT < 94 << 19 and fp + (146 << 19) < SWEEPS_FIT < 188 << 19
    srv = stab.Server(hbm_budget=budget)
    ids = [srv.submit(c, "grad", obs) for c in reqs]
    most = most_in_use(srv, ids)
    mix = [srv.wait(i, timeout_s=120) for i in ids]
    srv.close()
    if budget == SWEEPS_FIT:
        assert most >= 94 << 19            # a gradient was admitted with its sweeps
    for c, r in zip(reqs, mix):
        one = stab.Server(hbm_budget=budget)
        a = one.wait(one.submit(c, "grad", obs), timeout_s=120)
        one.close()
        assert a["status"] == 0 and r["status"] == 0
        assert a["expect"] == r["expect"]
        np.testing.assert_array_equal(a["grads"], r["grads"])
        rot = [i for i, g in enumerate(c.gates) if int(g["op"]) in W.ROTATIONS]
        want = oracle.psr_grad_gate(8, c.gates, c.thetas, obs, rot[len(rot) // 2])
        assert abs(r["grads"][int(c.gates[rot[len(rot) // 2]]["param"])] - want) <= 1e-12 * l1(obs)
