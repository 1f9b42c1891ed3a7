"""Term lists of known content across the sizes where the sparse path changes
form: one CTA's shared memory (4,096 terms), one round of tiles and several, a
capacity that is just enough or one short.

H on wire 0 and CX from it to wires 1 .. k-1 turn generator 0 into X ... X; R_z
on each of those wires doubles the list (every term spawns its partner), R_z on
each once more keeps it (every term has its partner).  The coefficient of the
string with Y on the wires of a mask is the product of cos or sin of the summed
angles.
"""
import math

import numpy as np
import pytest

from paper_2502_10685_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required")
    from paper_2502_10685_gb300 import stab
    return stab


def _circuit(k, seed):
    rng = np.random.default_rng(seed)
    th = rng.uniform(0.0, 2.0 * math.pi, 2 * k)
    g = np.zeros(3 * k, dtype=W.GATE_DTYPE)
    g["param"] = -1
    g[0] = (W.OPS["H"], 0, 0, 0, -1)
    for q in range(1, k):
        g[q] = (W.OPS["CX"], 0, q, 0, -1)
    for j in range(2 * k):
        g[k + j] = (W.OPS["RZ"], j % k, 0, 0, j)
    return g, th


@pytest.mark.parametrize("n,k", [(1, 1), (5, 5), (12, 11), (13, 12), (13, 13), (24, 14),
                                 (32, 16), (20, 20)])
def test_doubling_then_paired(S, n, k):
    gates, th = _circuit(k, 100 * n + k)
    order = 1 << k
    sp = S.Sparse(n, max_terms=order)
    sp.load_circuit(gates, th)
    terms, info = sp.generator(0)
    assert info["order_max"] == info["order_final"] == len(terms) == order
    assert np.all(terms["x"] == order - 1)
    want = np.ones(1)
    for q in range(k - 1, -1, -1):
        a = th[q] + th[k + q]
        want = np.concatenate([want * math.cos(a), want * math.sin(a)]) if q == k - 1 else \
            np.stack([want * math.cos(a), want * math.sin(a)], axis=-1).ravel()
    # wire q is bit q: the last factor taken above is wire 0
    got = np.zeros(order)
    got[terms["z"].astype(np.int64)] = terms["coeff"]
    # 2k rotations of a unit vector, a few roundings each
    assert np.max(np.abs(got - want)) <= 2 * k * 8 * 2.0 ** -52
    # <Z_0>: backward it passes the R_z and the CX and becomes X_0, not x-free
    value, _ = sp.expect([(1.0, "Z" + "I" * (n - 1))])
    assert value == 0.0
    sp.close()
    if k > 1:
        sp = S.Sparse(n, max_terms=order - 1)
        sp.load_circuit(gates, th)
        with pytest.raises(S.StabError) as e:
            sp.generator(0)
        assert e.value.code == -2
        sp.close()
