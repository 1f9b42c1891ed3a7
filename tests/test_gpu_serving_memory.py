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
