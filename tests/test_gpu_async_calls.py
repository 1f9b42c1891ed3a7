"""The asynchronous calls only queue: the first generators, <O> and gradient
after a load return while work queued before them on the caller's stream is
still running."""
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


@pytest.mark.parametrize("n,m", [(7, 300), (8, 200), (9, 110)])
def test_first_calls_after_a_load_do_not_wait(stab, n, m):
    import torch
    obs = W.obs_chain(n)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        # the second context: kernels are loaded by then, and memory is at hand
        for c in (W.layered_ansatz(n, m, seed=140), W.layered_ansatz(n, m, seed=141)):
            s = stab.Stab(n)
            s.load_circuit(c.gates, np.zeros(c.n_params))
            s.set_observable(obs)
            th = torch.tensor(c.thetas, device="cuda")
            e = torch.zeros(2, dtype=torch.float64, device="cuda")
            g = torch.zeros(c.n_params, dtype=torch.float64, device="cuda")
            gens = torch.zeros(n, 4 ** n, dtype=torch.float64, device="cuda")
            torch.cuda.synchronize()
            before = torch.cuda.Event()
            torch.cuda._sleep(1_000_000_000)        # half a second
            before.record(st)
            s.set_params(th)
            s.run_generators()
            s.generators(out=gens)
            s.expect_async(e[:1])
            s.grad_async(e[1:], g)
            queued = not before.query()
            torch.cuda.synchronize()
            got = e.cpu().numpy(), g.cpu().numpy(), gens.cpu().numpy()
            s.close()
    assert queued
    tol = 1e-12 * sum(abs(a) for a, _ in obs)
    assert np.abs(got[0] - oracle.expect(n, c.gates, c.thetas, obs)).max() <= tol
    rot = [i for i, gt in enumerate(c.gates) if int(gt["op"]) in W.ROTATIONS]
    for gi in (rot[0], rot[-1]):
        want = oracle.psr_grad_gate(n, c.gates, c.thetas, obs, gi)
        assert abs(got[1][int(c.gates[gi]["param"])] - want) <= tol
    want = oracle.forward(n, c.gates, c.thetas, oracle.generator(n, n - 1))
    assert np.abs(layout.lib_to_paper(n, got[2][n - 1]) - want).max() <= 1e-12


@pytest.mark.parametrize("n,m", [(7, 2000), (9, 600)])
def test_a_second_run_waits_for_the_copy_of_the_first(stab, n, m):
    """Generators copied to device memory are those of the run before the copy,
    also where the copy is still queued when the generators run again."""
    import torch
    c = W.layered_ansatz(n, m, seed=180 + n)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        s = stab.Stab(n)
        s.load_circuit(c.gates, c.thetas)
        out = torch.zeros(6, n, 4 ** n, dtype=torch.float64, device="cuda")
        s.run_generators()
        s.generators(out=out[0])
        for k in range(1, 6):
            s.run_generators()
            torch.cuda._sleep(300_000 * k)
            s.generators(out=out[k])
        s.run_generators()
        torch.cuda.synchronize()
        s.close()
    assert all(torch.equal(out[0], out[k]) for k in range(1, 6))
    got = out[0].cpu().numpy()
    want = oracle.forward(n, c.gates, c.thetas, oracle.generator(n, 0))
    assert np.abs(layout.lib_to_paper(n, got[0]) - want).max() <= 1e-12
