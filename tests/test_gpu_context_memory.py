"""What a context holds of a gradient's stored sweeps goes back when a circuit is
loaded that needs much less, or when the caller says so."""
import ctypes

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


def test_stored_sweeps_go_back_at_the_load_of_a_small_circuit(stab):
    """n = 10: 30 blocks of wire runs keep at least 60 vectors of 8 MiB, the small
    circuit's two at most ten."""
    import torch
    from paper_2502_10685_gb300 import _lib
    L, live = _lib.load(), {}

    def _alloc(nbytes, st, user):
        p = int(torch.cuda.caching_allocator_alloc(int(nbytes), 0))
        live[p] = int(nbytes)
        return p

    def _free(ptr, nbytes, st, user):
        assert live.pop(int(ptr)) == int(nbytes)
        torch.cuda.caching_allocator_delete(int(ptr))

    hooks = _lib.ALLOC_FN(_alloc), _lib.FREE_FN(_free)
    o = stab.stab_default_opts()
    o.device = 0
    o.alloc, o.free = hooks
    h = ctypes.c_void_p()
    assert L.stab_create(10, ctypes.byref(o), ctypes.byref(h)) == 0
    obs = W.obs_chain(10)
    terms = stab.terms_from_observable(10, obs)
    held = []
    for c in (W.layered_ansatz(10, 1200, seed=150), W.layered_ansatz(10, 50, seed=151)):
        g, e, out = np.ascontiguousarray(c.gates), ctypes.c_double(), np.zeros(c.n_params)
        assert L.stab_load_circuit(h, g.ctypes.data, c.m, c.thetas.ctypes.data, c.n_params) == 0
        held.append(sum(live.values()))
        assert L.stab_grad(h, terms.ctypes.data, len(terms), ctypes.byref(e), out.ctypes.data) == 0
        held.append(sum(live.values()))
        tol = 1e-12 * sum(abs(a) for a, _ in obs)
        assert abs(e.value - oracle.expect(10, c.gates, c.thetas, obs)) <= tol
        rot = [i for i, gt in enumerate(c.gates) if int(gt["op"]) in W.ROTATIONS]
        want = oracle.psr_grad_gate(10, c.gates, c.thetas, obs, rot[-1])
        assert abs(out[int(c.gates[rot[-1]]["param"])] - want) <= tol
    assert held[1] >= 60 * 8 << 20          # the first gradient's sweeps
    assert held[2] <= held[1] - (60 * 8 << 20) and held[3] < held[1] // 2
    assert L.stab_destroy(h) == 0 and not live


def test_the_caller_may_limit_the_memory(stab):
    """With no memory for the sweeps' vectors a gradient carries a fixed number of
    them; with a limit just below what it needs as well; with enough, and as
    before, it keeps them."""
    import torch
    from paper_2502_10685_gb300._lib import StabError
    c, obs = W.layered_ansatz(9, 360, seed=152), W.obs_chain(9)
    e_want = oracle.expect(9, c.gates, c.thetas, obs)
    tol = 1e-12 * sum(abs(a) for a, _ in obs)
    s = stab.Stab(9)
    s.load_circuit(c.gates, c.thetas)
    e0, g0 = s.grad(obs)
    kept = torch.cuda.memory_allocated()
    values = []
    # 10 blocks: 25 vectors of 2 MiB
    for limit in (0, (25 * 2 << 20) - 1, 25 * 2 << 20):
        s.set_grad_memory(limit)
        e, g = s.grad(obs)
        values.append((e, g))
        assert abs(e - e_want) <= tol and np.abs(g - g0).max() <= tol
    assert values[0][0] == values[1][0] and np.array_equal(values[0][1], values[1][1])
    assert values[2][0] == e0 and np.array_equal(values[2][1], g0)
    s.set_grad_memory(0)
    assert torch.cuda.memory_allocated() < kept
    with pytest.raises(StabError):
        s.set_grad_memory(-1)
    s.close()
