"""Clifford runs as gathers (streamed plans): source index and sign against the
gates applied one at a time, on the host."""
import numpy as np
import pytest

from paper_2502_10685_gb300 import _lib, workloads as W


@pytest.mark.parametrize("n", [1, 2, 3, 5, 8, 12])
@pytest.mark.parametrize("m", [0, 1, 2, 9, 200])
def test_gather_equals_gate_by_gate(n, m):
    L = _lib.load()
    c = W.random_circuit(n, m, seed=31 * n + m, clifford_only=True)
    g = np.ascontiguousarray(c.gates)
    assert L.stab_selftest_pull(n, g.ctypes.data if m else None, m) == 0


@pytest.mark.parametrize("op", ["H", "S", "SDG", "X", "Y", "Z", "CX", "CZ"])
def test_gather_of_single_gates_and_rings(op):
    L = _lib.load()
    two = op in ("CX", "CZ")
    for n in (2, 4):
        for a in range(n):
            g = np.ascontiguousarray(W.gates_from_list([(op, a, (a + 1) % n) if two else (op, a)]))
            assert L.stab_selftest_pull(n, g.ctypes.data, 1) == 0
        ring = W.gates_from_list([(op, a, (a + 1) % n) if two else (op, a) for a in range(n)])
        g = np.ascontiguousarray(ring)
        assert L.stab_selftest_pull(n, g.ctypes.data, n) == 0


def test_rotations_are_refused():
    L = _lib.load()
    g = np.ascontiguousarray(W.gates_from_list([("RX", 0, 0)]))
    assert L.stab_selftest_pull(2, g.ctypes.data, 1) == -2
