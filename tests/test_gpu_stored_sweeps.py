"""Streamed gradients from stored sweeps: every shape a plan can take around its
blocks of wire passes (Clifford runs at the ends, several in a row, long runs,
shared slots, one or two tile shapes), against the CPU oracle."""
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


def wrapped(n, m, seed):
    """Clifford-only stretches before, between and after layered circuits, long
    enough to become one gather, directly followed by two-qubit runs."""
    rng = np.random.default_rng(seed)
    cliff = [W.random_circuit(n, 60, seed=seed + k, clifford_only=True).gates for k in range(3)]
    ring = W.gates_from_list([("CX", q, (q + 1) % n) for q in range(n)])
    rows = W.gates_from_list([("H", q) for q in range(n)])
    base = W.layered_ansatz(n, m, seed=seed + 9)
    second = base.gates.copy()
    rot = np.isin(second["op"], W.ROTATIONS)
    second["param"][rot] += base.n_params
    gates = np.concatenate([cliff[0], ring, base.gates, ring, rows, cliff[1], ring, second, ring,
                            cliff[2], rows])
    return W.Circuit(n, gates, rng.uniform(0, 2 * np.pi, 2 * base.n_params))


CASES = [(2, "layered", 40, "streamed"), (3, "random", 120, "streamed"),
         (4, "wrapped", 50, "streamed"), (5, "random", 160, "streamed"),
         (5, "paper", 3, "streamed"), (6, "layered", 151, "streamed"),
         (6, "wrapped", 60, "streamed"), (7, "layered", 300, "auto"), (7, "wrapped", 80, "auto"),
         (8, "random", 140, "auto"), (8, "sparse", 400, "auto"), (9, "layered", 130, "auto"),
         (10, "layered", 90, "auto")]


@pytest.mark.parametrize("n,family,size,kernel", CASES)
def test_gradient_matches_parameter_shift(stab, n, family, size, kernel):
    if family == "layered":
        c = W.layered_ansatz(n, size, seed=800 + n)
    elif family == "random":
        c = W.random_circuit(n, size, seed=801 + n, shared_params=9)
    elif family == "sparse":
        c = W.clifford_plus_rotations(n, size, 12, seed=802 + n)
    elif family == "paper":
        c = W.paper_shaped_ansatz(n, size, 15, seed=803 + n)      # 45 rotations a run
    else:
        c = wrapped(n, size, seed=804 + n)
    obs = W.obs_chain(n) + W.random_observable(n, 3, seed=805)
    tol = 1e-12 * sum(abs(a) for a, _ in obs)
    s = stab.Stab(n, kernel=kernel)
    s.load_circuit(c.gates, c.thetas)
    th2 = np.random.default_rng(806).uniform(-9, 9, c.n_params)
    rot = [i for i, gt in enumerate(c.gates) if int(gt["op"]) in W.ROTATIONS]
    picks = {rot[0], rot[-1]} | ({rot[len(rot) // 2], rot[len(rot) // 3]} if n < 9 else set())
    for k, th in enumerate((c.thetas, th2, th2)):     # the third call replays the captured graph
        if k == 1:
            s.set_params(th)
        e, g = s.grad(obs)
        if k == 1:
            first = (e, g.copy())
            continue
        if k == 2:
            assert e == first[0] and np.array_equal(g, first[1])
        assert abs(e - oracle.expect(n, c.gates, th, obs)) <= tol
        if family == "random" and n < 8:
            assert np.abs(g - oracle.psr_grad(n, c.gates, th, obs)).max() <= tol
            continue
        if family == "random":
            continue
        for gi in picks:
            want = oracle.psr_grad_gate(n, c.gates, th, obs, gi)
            assert abs(g[int(c.gates[gi]["param"])] - want) <= tol, gi
    s.close()
