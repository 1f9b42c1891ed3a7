"""What served gradients take beside their footprint (stored sweeps, tables) is
decided by the request and the server's budget alone, counted while it is held,
and given back."""
import threading
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


def test_nothing_reserved_for_tables_that_are_not_used(stab):
    """<O> at n = 9 runs as launches, without the chains' tables."""
    c, obs = W.layered_ansatz(9, 2000, seed=62), W.obs_chain(9)
    srv = stab.Server()
    i = srv.submit(c, "expect", obs)
    most = most_in_use(srv, [i])
    assert srv.wait(i, timeout_s=120)["status"] == 0
    srv.close()
    assert most == stab.Server.footprint(c, "expect", obs)


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


class HookedServer:
    """A server on allocator hooks: ``refuse(nbytes, live)`` says which
    allocations fail (live: the sizes of the blocks handed out)."""

    def __init__(self, stab, refuse=lambda nbytes, live: False, **fields):
        import ctypes

        import torch
        from paper_2502_10685_gb300 import _lib
        self.stab, self.lib, self.live, self.most = stab, _lib.load(), {}, 0
        self.allocs = 0
        self.lock = threading.Lock()

        def _alloc(nbytes, st, user):
            with self.lock:
                if refuse(int(nbytes), self.live.values()):
                    return None
                p = int(torch.cuda.caching_allocator_alloc(int(nbytes), 0))
                self.live[p] = int(nbytes)
                self.allocs += 1
                self.most = max(self.most, sum(self.live.values()))
                return p

        def _free(ptr, nbytes, st, user):
            with self.lock:
                assert self.live.pop(int(ptr)) == int(nbytes)
            torch.cuda.caching_allocator_delete(int(ptr))

        self.hooks = (_lib.ALLOC_FN(_alloc), _lib.FREE_FN(_free))
        o = _lib.StabServerOpts()
        o.alloc, o.free = self.hooks
        for k, v in fields.items():
            setattr(o, k, v)
        self.h = ctypes.c_void_p()
        assert self.lib.stab_server_create(ctypes.byref(o), ctypes.byref(self.h)) == 0

    def stats(self):
        return self.stab.Server.stats(self)

    def submit(self, c, kind, obs):
        import ctypes
        keep, i = [], ctypes.c_int64()
        r = self.stab.Server._request(c, kind, obs, keep)
        assert self.lib.stab_server_submit(self.h, ctypes.byref(r), ctypes.byref(i)) == 0
        return i.value

    def wait(self, i, n_params):
        import ctypes
        from paper_2502_10685_gb300 import _lib
        res, grads = _lib.StabResult(), np.zeros(n_params)
        assert self.lib.stab_server_wait(self.h, i, 120.0, ctypes.byref(res),
                                         grads.ctypes.data) == 0
        return res.status, res.expect, grads

    def close(self):
        assert self.lib.stab_server_destroy(self.h) == 0
        assert not self.live


@pytest.mark.parametrize("blocks_at_once", [1, 0])
def test_no_memory_for_the_sweeps_beside_others(stab, blocks_at_once):
    """The device has room for the stored sweeps of one request at a time (or of
    none): requests wait for it, all are served, and every result is that of the
    request alone on the same device."""
    obs = W.obs_chain(8)
    reqs = [W.layered_ansatz(8, 1500, seed=90 + k) for k in range(5)]
    assert stab.Server.footprint(reqs[0], "grad", obs) < 40 << 20 < 94 << 19

    def refuse(nbytes, live):
        return nbytes > 40 << 20 and sum(b > 40 << 20 for b in live) >= blocks_at_once

    srv = HookedServer(stab, refuse)
    ids = [srv.submit(c, "grad", obs) for c in reqs]
    mix = [srv.wait(i, c.n_params) for i, c in zip(ids, reqs)]
    srv.close()
    for c, (status, e, g) in zip(reqs, mix):
        one = HookedServer(stab, refuse)
        status1, e1, g1 = one.wait(one.submit(c, "grad", obs), c.n_params)
        one.close()
        assert status == 0 and status1 == 0
        assert e == e1
        np.testing.assert_array_equal(g, g1)


@pytest.mark.parametrize("kind", ["expect", "grad"])
@pytest.mark.parametrize("n,m", [(7, 5000), (8, 2500)])
def test_tables_are_counted(stab, n, m, kind):
    """Random circuits have a table per Clifford run: what a request has
    allocated at any time (beside a megabyte of a context's and the server's own
    small buffers) is covered by what it was admitted with."""
    c, obs = W.random_circuit(n, m, seed=95 + n), W.obs_chain(n)
    srv = HookedServer(stab)
    i = srv.submit(c, kind, obs)
    most = most_in_use(srv, [i])
    status, e, g = srv.wait(i, c.n_params)
    srv.close()
    assert status == 0
    assert abs(e - oracle.expect(n, c.gates, c.thetas, obs)) <= 1e-12 * l1(obs)
    assert srv.most <= most + (1 << 20)


def test_no_budget_for_the_tables(stab):
    """A budget of the footprint alone: the same request runs without tables."""
    c, obs = W.random_circuit(8, 2500, seed=97), W.obs_chain(8)
    want = oracle.expect(8, c.gates, c.thetas, obs)
    for kind in ("expect", "grad"):
        fp = stab.Server.footprint(c, kind, obs)
        srv = HookedServer(stab, hbm_budget=fp)
        i = srv.submit(c, kind, obs)
        most = most_in_use(srv, [i])
        status, e, g = srv.wait(i, c.n_params)
        srv.close()
        assert status == 0 and most == fp and srv.most <= fp + (1 << 20)
        assert abs(e - want) <= 1e-12 * l1(obs)


def test_idle_contexts_memory_stays_inside_the_budget(stab):
    """Contexts keep up to 64 MiB of stored sweeps between requests; a request
    that needs that room in the budget gets it first.  (Four requests at once
    leave four contexts with 50 MiB each, then one of n = 9 needs 210.)"""
    obs = W.obs_chain(8)
    reqs = [W.layered_ansatz(8, 1500, seed=110 + k) for k in range(4)]
    big = W.layered_ansatz(9, 1800, seed=120)
    budget = 370 << 20
    srv = HookedServer(stab, hbm_budget=budget, max_active=4)
    ids = [srv.submit(c, "grad", obs) for c in reqs]
    small = [srv.wait(i, c.n_params) for i, c in zip(ids, reqs)]
    status, e, g = srv.wait(srv.submit(big, "grad", W.obs_chain(9)), big.n_params)
    again = srv.wait(srv.submit(reqs[0], "grad", obs), reqs[0].n_params)
    srv.close()
    assert status == 0 and all(r[0] == 0 for r in small + [again])
    assert srv.most <= budget + (1 << 20)
    assert abs(e - oracle.expect(9, big.gates, big.thetas, W.obs_chain(9))) <= \
        1e-12 * l1(W.obs_chain(9))
    assert again[1] == small[0][1]
    np.testing.assert_array_equal(again[2], small[0][2])


@pytest.mark.parametrize("n,m,iter_max_n", [(8, 250, 8), (6, 3000, 6), (4, 60200, 4)])
def test_iter_max_n_takes_long_requests(stab, n, m, iter_max_n):
    """A caller's iter_max_n holds for requests of any length: a long gradient runs
    in the iteration engine (many slices of both phases), which takes one block
    of memory a request, also for the second of two equal ones (a pooled context
    would have its buffers by then)."""
    c, obs = W.layered_ansatz(n, m, seed=130 + n), W.obs_chain(n)
    srv = HookedServer(stab, iter_max_n=iter_max_n, iter_chunks=8)
    assert srv.wait(srv.submit(c, "grad", obs), c.n_params)[0] == 0
    before = srv.allocs
    status, e, g = srv.wait(srv.submit(c, "grad", obs), c.n_params)
    assert srv.allocs - before == 1
    srv.close()
    tol = (1e-10 if m > 20000 else 1e-12) * l1(obs)
    assert status == 0
    assert abs(e - oracle.expect(n, c.gates, c.thetas, obs)) <= tol
    rot = [i for i, gt in enumerate(c.gates) if int(gt["op"]) in W.ROTATIONS]
    for gi in (rot[0], rot[len(rot) // 2], rot[-1]):
        want = oracle.psr_grad_gate(n, c.gates, c.thetas, obs, gi)
        assert abs(g[int(c.gates[gi]["param"])] - want) <= tol


def test_idle_contexts_hand_large_tables_back(stab):
    """100,000 random gates at n = 8 have more than 64 MiB of tables: an idle context
    keeps none of them."""
    c, obs = W.random_circuit(8, 100000, seed=200), W.obs_chain(8)
    srv = HookedServer(stab)
    status, e, g = srv.wait(srv.submit(c, "expect", obs), c.n_params)
    most, after = srv.most, sum(srv.live.values())
    srv.close()
    assert status == 0
    s = stab.Stab(8)
    s.load_circuit(c.gates, c.thetas)
    assert abs(e - s.expect(obs)) <= 1e-10 * l1(obs)
    s.close()
    assert most > 80 << 20 and after < most - (60 << 20)
