"""Long items of a batch (chains on many SMs): creation leaves nothing behind
that the first run would have to wait for."""
import ctypes
import math

import numpy as np
import pytest

import layout
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


class HookedBatch:
    """A batch of items on caller-given allocator hooks: ``on_alloc(nbytes, stream)``
    runs before every allocation and refuses it by returning False."""

    def __init__(self, stab, items, on_alloc):
        import torch
        from paper_2502_10685_gb300 import _lib
        self.lib, self.keep, self.items, self.live = _lib.load(), [], items, {}
        arr = (_lib.StabBatchItem * len(items))()
        for a, it in zip(arr, items):
            c = it.circuit
            g = np.ascontiguousarray(c.gates)
            th = np.ascontiguousarray(c.thetas if c.n_params else np.zeros(1))
            self.keep += [g, th]
            a.n, a.m, a.n_params = c.n, c.m, c.n_params
            a.kind = stab.ITEM_KINDS[it.kind]
            a.gates, a.thetas = (g.ctypes.data if c.m else None), th.ctypes.data
            if it.kind == "expect":
                t = stab.terms_from_observable(c.n, it.observable)
                self.keep.append(t)
                a.obs, a.n_terms = t.ctypes.data, len(t)

        def _alloc(nbytes, st, user):
            if on_alloc(int(nbytes), int(st or 0)) is False:
                return None
            p = int(torch.cuda.caching_allocator_alloc(int(nbytes), 0))
            self.live[p] = int(nbytes)
            return p

        def _free(ptr, nbytes, st, user):
            assert self.live.pop(int(ptr)) == int(nbytes)
            torch.cuda.caching_allocator_delete(int(ptr))

        self.hooks = (_lib.ALLOC_FN(_alloc), _lib.FREE_FN(_free))
        o = stab.stab_default_opts()
        o.device = 0
        o.alloc, o.free = self.hooks
        self.h = ctypes.c_void_p()
        self.rc = self.lib.stab_batch_create(arr, len(items), ctypes.byref(o),
                                             ctypes.byref(self.h))

    def run(self):
        assert self.lib.stab_apply_batch(self.h) == 0

    def expectations(self):
        out = np.empty(len(self.items))
        assert self.lib.stab_batch_expectations(self.h, out.ctypes.data) == 0
        return out

    def close(self):
        assert self.lib.stab_batch_destroy(self.h) == 0
        assert not self.live


def test_terms_are_there_before_the_first_run(stab):
    """The terms of a long <O> item are uploaded on its context's own stream,
    here behind a tenth of a second of other work on that stream (queued when
    the terms are allocated): when creation returns, every stream that memory
    was taken on is idle, so the first run reads the terms."""
    import torch
    items = [W.BatchItem(W.layered_ansatz(8, 1301, seed=5), "expect", W.obs_chain(8)),
             W.BatchItem(W.random_circuit(7, 2500, seed=6), "expect", W.obs_chain(7))]
    streams = {}
    first = []

    def on_alloc(nbytes, st):
        if not first:
            first.append(st)              # the batch's stream
        if st not in streams:
            streams[st] = torch.cuda.ExternalStream(st)
            if st != first[0]:
                with torch.cuda.stream(streams[st]):
                    torch.cuda._sleep(200_000_000)

    b = HookedBatch(stab, items, on_alloc)
    assert b.rc == 0
    assert len(streams) > 1
    assert all(s.query() for s in streams.values())
    b.run()
    ex = b.expectations()
    b.close()
    for e, it in zip(ex, items):
        c = it.circuit
        want = oracle.expect(c.n, c.gates, c.thetas, it.observable)
        assert abs(e - want) <= 1e-12 * l1(it.observable)


def test_identity_circuits_among_long_items(stab):
    """An n = 8 circuit that does nothing (no gates, or pairs that cancel) counts
    as long and has no chain step: its values come out all the same, alone and
    beside a chain."""
    empty = W.Circuit(8, np.zeros(0, dtype=W.GATE_DTYPE), np.zeros(0))
    pairs = W.Circuit(8, W.gates_from_list([("X", 3), ("X", 3)]), np.zeros(0))
    obs = [(0.75, "ZIIIIIIZ"), (0.5, "IIIIIIII"), (2.0, "XIIIIIII")]
    still = [W.BatchItem(empty, "generators"), W.BatchItem(pairs, "expect", obs)]
    deep = W.BatchItem(W.layered_ansatz(8, 1301, seed=5), "expect", W.obs_chain(8))
    for items in (still[:1], still[1:], still, still + [deep]):
        b = stab.Batch(items)
        for _ in range(2):
            b.run()
            ex = b.expectations()
            for k, it in enumerate(items):
                c = it.circuit
                if it.kind == "generators":
                    assert math.isnan(ex[k])
                    want = oracle.generators(8, c.gates, c.thetas)
                    assert np.array_equal(layout.lib_to_paper(8, b.generators(k)), want)
                else:
                    want = oracle.expect(8, c.gates, c.thetas, it.observable)
                    assert abs(ex[k] - want) <= 1e-12 * l1(it.observable)
        b.close()


def test_no_room_for_the_long_items_contexts(stab):
    """An allocation that fails while the long items are set up (their terms, or
    the last one of all) does not refuse the batch: they run as other items."""
    items = [W.BatchItem(W.layered_ansatz(6, 3001, seed=5), "expect", W.obs_chain(6)),
             W.BatchItem(W.layered_ansatz(6, 2000, seed=8), "generators")]
    items += [W.BatchItem(W.layered_ansatz(3, 60 + k, seed=20 + k), "expect", W.obs_chain(3))
              for k in range(5)]
    calls = []
    b = HookedBatch(stab, items, lambda nbytes, st: calls.append(st))
    assert b.rc == 0
    b.close()
    terms = next(k for k, st in enumerate(calls) if st != calls[0])
    for refuse in (terms, len(calls) - 1):
        at = []

        def on_alloc(nbytes, st):
            at.append(st)
            return len(at) - 1 != refuse

        b = HookedBatch(stab, items, on_alloc)
        assert b.rc == 0 and len(at) > len(calls) // 2
        b.run()
        ex = b.expectations()
        b.close()
        for e, it in zip(ex, items):
            if it.kind == "expect":
                c = it.circuit
                want = oracle.expect(c.n, c.gates, c.thetas, it.observable)
                assert abs(e - want) <= 1e-12 * l1(it.observable)
