"""Long plans at n <= 4 through their segments' unitaries: generators, <O>, the
density matrix and the gradient against the CPU oracle at the sizes where the
segments, the tree and the wire runs can go wrong."""
import numpy as np
import pytest

import layout
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


def bitrev(n):
    return [int(format(i, "0%db" % n)[::-1], 2) for i in range(2 ** n)]


def h_heavy(n, layers, run, seed):
    """Layers of `run` gates per wire, two thirds of them H, S or X, then a CZ / CX ring:
    every parity of H gates before, in and after a run, and runs longer than a warp."""
    rng = np.random.default_rng(seed)
    items, slots = [], 0
    for _ in range(layers):
        for q in range(n):
            for _ in range(int(rng.integers(1, run + 1))):
                op = str(rng.choice(["H", "H", "S", "X", "RX", "RZ"]))
                if op in ("RX", "RZ"):
                    items.append((op, q, slots))
                    slots += 1
                else:
                    items.append((op, q))
        for q in range(n):
            items.append((str(rng.choice(["CX", "CZ"])), q, (q + 1) % n))
    return W.Circuit(n, W.gates_from_list(items), rng.uniform(0, 2 * np.pi, slots))


CASES = [
    ("layered", 4, 270), ("layered", 4, 1777), ("layered", 3, 999), ("layered", 2, 2001),
    ("random", 4, 900), ("random", 3, 2500), ("random", 2, 1500),
    ("h_heavy", 4, 30), ("h_heavy", 3, 41), ("h_heavy", 2, 70), ("h_long", 4, 24), ("h_long", 2, 45),
]


@pytest.mark.parametrize("family,n,size", CASES)
def test_segments_match_oracle(stab, family, n, size):
    if family == "layered":
        c = W.layered_ansatz(n, size, seed=900 + size)
    elif family == "random":
        c = W.random_circuit(n, size, seed=901 + size, shared_params=7)
    else:
        c = h_heavy(n, size, 6 if family == "h_heavy" else 90, seed=902 + size)
    obs = W.random_observable(n, 6, seed=903) + [(0.5, "I" * n), (0.25, "Y" * n)]
    s = stab.Stab(n)
    s.load_circuit(c.gates, c.thetas)
    assert s.split_info()[0] > 0
    th2 = np.random.default_rng(904).uniform(-7, 7, c.n_params)
    tol = 1e-12 * sum(abs(a) for a, _ in obs)
    perm = bitrev(n)
    for k, th in enumerate((c.thetas, th2)):
        if k:
            s.set_params(th)
        e0, g = s.grad(obs)
        rho = s.density_matrix()
        s.run_generators()
        gens = layout.lib_to_paper(n, s.generators())
        e1 = s.expect(obs)
        want = oracle.expect(n, c.gates, th, obs)
        assert abs(e0 - want) <= tol and abs(e1 - want) <= tol
        assert np.abs(gens - oracle.generators(n, c.gates, th)).max() <= 1e-12
        assert np.abs(rho[np.ix_(perm, perm)] - oracle.density_matrix(n, c.gates, th)).max() \
            <= 1e-12
        if family == "random":      # shared slots: each gradient sums over its gates
            assert np.abs(g - oracle.psr_grad(n, c.gates, th, obs)).max() <= tol
        else:
            rot = [i for i, gt in enumerate(c.gates) if int(gt["op"]) in W.ROTATIONS]
            for gi in {rot[0], rot[-1]} | {rot[(len(rot) * j) // 9] for j in range(1, 9)}:
                want = oracle.psr_grad_gate(n, c.gates, th, obs, gi)
                assert abs(g[int(c.gates[gi]["param"])] - want) <= tol, gi
    s.close()


@pytest.mark.parametrize("n,m", [(2, 700), (3, 1500), (4, 5000)])
def test_long_clifford_circuits_stay_bit_exact(stab, n, m):
    c = W.random_circuit(n, m, seed=910 + n, clifford_only=True)
    s = stab.Stab(n)
    s.apply_circuit(c.gates, c.thetas)
    assert s.split_info()[0] > 0
    np.testing.assert_array_equal(layout.lib_to_paper(n, s.generators()),
                                  oracle.generators(n, c.gates, c.thetas))
    obs = W.obs_chain(n)
    assert s.expect(obs) == oracle.expect(n, c.gates, c.thetas, obs)
    s.close()


@pytest.mark.parametrize("n,m", [(1, 1023), (1, 1024), (1, 5000), (2, 40000)])
def test_runs_of_thousands_of_gates(stab, n, m):
    # one wire run of m gates per qubit, composed by a CTA
    c = W.random_circuit(1, m, seed=920 + m)
    gates = np.concatenate([c.gates] * n)
    for q in range(n):
        gates["q0"][q * m:(q + 1) * m] = q
    obs = [(1.0, "Z" * n), (0.5, "X" + "I" * (n - 1)), (-0.25, "Y" * n)]
    s = stab.Stab(n)
    s.apply_circuit(gates, c.thetas)
    tol = 1e-10 if m >= 40000 else 1e-12
    assert np.abs(layout.lib_to_paper(n, s.generators())
                  - oracle.generators(n, gates, c.thetas)).max() <= tol
    assert abs(s.expect(obs) - oracle.expect(n, gates, c.thetas, obs)) <= 1.75 * tol
    s.close()


@pytest.mark.parametrize("n", [2, 3])
@pytest.mark.parametrize("layers", [1, 2, 3, 4, 5, 12, 21, 22])
def test_short_plans(stab, n, layers):
    """From 8 passes on plans of two and three qubits run through the unitaries,
    below through the coefficients; all read-outs, and Clifford circuits exactly."""
    for c, exact in ((h_heavy(n, layers, 4, seed=940 + 10 * n + layers), False),
                     (W.random_circuit(n, 6 * layers, seed=950 + layers, clifford_only=True), True)):
        obs = W.obs_chain(n) + [(0.25, "Y" * n)]
        tol = 0.0 if exact else 1e-12 * sum(abs(a) for a, _ in obs)
        s = stab.Stab(n)
        s.apply_circuit(c.gates, c.thetas)
        gens = layout.lib_to_paper(n, s.generators())
        assert np.abs(gens - oracle.generators(n, c.gates, c.thetas)).max() <= tol
        assert abs(s.expect(obs) - oracle.expect(n, c.gates, c.thetas, obs)) <= tol
        perm = bitrev(n)
        rho = s.density_matrix()[np.ix_(perm, perm)]
        assert np.abs(rho - oracle.density_matrix(n, c.gates, c.thetas)).max() <= max(tol, 1e-15)
        e, g = s.grad(obs)
        assert abs(e - oracle.expect(n, c.gates, c.thetas, obs)) <= tol
        if c.n_params:
            want = oracle.psr_grad(n, c.gates, c.thetas, obs)
            assert np.abs(g - want).max() <= 1e-12 * sum(abs(a) for a, _ in obs)
        s.close()
