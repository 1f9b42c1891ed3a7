"""Streamed gradients against the oracle's parameter shift where other tests do
not reach: the pair sweep (no memory for stored sweeps), and slots shared by
several gates at sizes whose full parameter shift takes too long."""
import numpy as np
import pytest

import oracle
from paper_2502_10685_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def stab():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    from paper_2502_10685_gb300 import stab as S
    return S


def runs_everywhere(n, m, seed):
    """Clifford runs at both ends and between two layered circuits, long ones (a
    gather each) next to two-qubit runs."""
    rng = np.random.default_rng(seed)
    cliff = [W.random_circuit(n, 50, seed=seed + k, clifford_only=True).gates for k in range(3)]
    ring = W.gates_from_list([("CX", q, (q + 1) % n) for q in range(n)])
    pairs = W.gates_from_list([("CZ", q, q + 1) for q in range(n - 1)] + [("X", 0), ("X", 0)])
    base = W.layered_ansatz(n, m, seed=seed + 9)
    second = base.gates.copy()
    rot = np.isin(second["op"], W.ROTATIONS)
    second["param"][rot] += base.n_params
    gates = np.concatenate([ring, pairs, ring, cliff[0], base.gates, ring, cliff[1], pairs, ring,
                            second, cliff[2], ring, pairs])
    return W.Circuit(n, gates, rng.uniform(0, 2 * np.pi, 2 * base.n_params))


def slot_derivative(c, obs, slot):
    """Sum of the parameter shifts of the gates that read the slot."""
    at = [i for i, g in enumerate(c.gates)
          if int(g["op"]) in W.ROTATIONS and int(g["param"]) == slot]
    return sum(oracle.psr_grad_gate(c.n, c.gates, c.thetas, obs, i) for i in at)


@pytest.mark.parametrize("memory", [0, 4 << 30])
@pytest.mark.parametrize("n,family,m", [(5, "runs", 60), (6, "runs", 60), (7, "runs", 70),
                                        (7, "random", 160), (8, "runs", 60), (8, "random", 140),
                                        (9, "runs", 40), (9, "random", 90)])
def test_both_forms_match_parameter_shift(stab, n, family, m, memory):
    c = runs_everywhere(n, m, 160 + n) if family == "runs" else \
        W.random_circuit(n, m, seed=170 + n, shared_params=7)
    obs = W.obs_chain(n) + W.random_observable(n, 3, seed=161)
    tol = 1e-12 * sum(abs(a) for a, _ in obs)
    s = stab.Stab(n, kernel="streamed" if n < 7 else "auto")
    s.set_grad_memory(memory)
    s.load_circuit(c.gates, c.thetas)
    for _ in range(2):                    # the second call replays the captured launches
        e, g = s.grad(obs)
        assert abs(e - oracle.expect(n, c.gates, c.thetas, obs)) <= tol
        for slot in (0, c.n_params // 2, c.n_params - 1):
            assert abs(g[slot] - slot_derivative(c, obs, slot)) <= tol, slot
    s.close()


@pytest.mark.parametrize("rotations", range(33, 38))
def test_groups_that_fill_the_default_shared_memory(stab, rotations):
    """A tile group of the pair sweep keeps a row per rotation in shared memory:
    35 rotations of one group take exactly 48 KiB, where the kernel's static
    shared memory no longer fits beside them."""
    n = 7
    row = W.gates_from_list([("RX", q, k) for k, q in enumerate(range(1, n))])
    row2 = W.gates_from_list([("RY", q, n + k) for k, q in enumerate(range(1, n))])
    cx = W.gates_from_list([("CX", 0, 1)])
    run = W.gates_from_list([(("RX", "RY", "RZ")[k % 3], 0, 2 * n + k) for k in range(rotations)])
    gates = np.concatenate([row, cx, row2, cx, run])
    c = W.Circuit(n, gates, np.random.default_rng(rotations).uniform(0, 6, 2 * n + rotations))
    obs = W.obs_chain(n)
    tol = 1e-12 * sum(abs(a) for a, _ in obs)
    s = stab.Stab(n)
    s.set_grad_memory(0)
    s.load_circuit(c.gates, c.thetas)
    e, g = s.grad(obs)
    s.close()
    assert abs(e - oracle.expect(n, c.gates, c.thetas, obs)) <= tol
    assert np.abs(g - oracle.psr_grad(n, c.gates, c.thetas, obs)).max() <= tol
