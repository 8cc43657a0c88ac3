"""Buffers that only make a call faster -- the tiles of a run-major join, bit
planes, a batch's list of long runs -- give way when the device memory for them
cannot be had: the call then runs in the form that does without."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1111_7171_gb300 import passjoin as pj
from paper_1111_7171_gb300 import synth

pytestmark = pytest.mark.gpu

COUNTS = ("lookups", "candidates", "accepted", "hits")


class Memory:
    """An allocator that refuses to hold more than `limit` bytes at once, and
    once each of the sizes in `refused`."""

    def __init__(self, monkeypatch):
        self.limit, self.refused = 1 << 60, []
        self.live, self.now, self.peak, self.refusals = {}, 0, 0, 0
        self.alloc, self.free = pj.ALLOC_FN(self._alloc), pj.FREE_FN(self._free)
        monkeypatch.setattr(pj, "_torch_alloc", self.alloc)
        monkeypatch.setattr(pj, "_torch_free", self.free)

    def _alloc(self, ctx, nbytes, stream):
        if self.now + nbytes > self.limit or nbytes in self.refused:
            self.refusals += 1
            if nbytes in self.refused:
                self.refused.remove(nbytes)
            return None
        p = torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device(), stream or 0)
        self.live[p] = nbytes
        self.now += nbytes
        self.peak = max(self.peak, self.now)
        return p

    def _free(self, ctx, p, stream):
        self.now -= self.live.pop(p)
        torch.cuda.caching_allocator_delete(p)


@pytest.mark.parametrize("knobs", [{}, {"PJ_ACCEPT_INITIAL": "16"}, {"PJ_GROUP_BUDGET": "30000"}])
def test_tiles_give_way(knobs, monkeypatch):
    strings = synth.generate("short", 4, n=6001)
    b, o = synth.pack(strings)
    want = oracle.self_join(b, o, 4, banded=True)
    mem = Memory(monkeypatch)
    monkeypatch.setenv("PJ_VERIFY_PAIRS", "0")
    for k, x in knobs.items():
        monkeypatch.setenv(k, x)
    idx = pj.pj_build_index(strings, 4)

    def join(tiles_from, limit=1 << 60):
        monkeypatch.setenv("PJ_TILES_MIN_HITS", str(tiles_from))
        mem.limit, mem.peak, mem.refusals = limit, mem.now, 0
        r = pj.pj_self_join(idx, 4)
        mem.limit = 1 << 60
        assert np.array_equal(r.pairs, want)
        return {k: r.stats[k] for k in COUNTS}, mem.peak, mem.refusals

    held = mem.now
    counts, queued, _ = join(1 << 40)
    tiled_counts, tiled, _ = join(1)
    assert tiled_counts == counts and tiled > queued
    for k in range(8):  # from what the queued form needs to somewhat short of the tiles' need, which varies a little
        got, _, refusals = join(1, queued + (tiled - queued) * k // 8)
        assert got == counts and refusals > 0, k
    assert mem.now == held
    idx.free()


def test_planes_and_run_lists_give_way(monkeypatch):
    strings = synth.generate("short", 4, n=5003)
    queries = [s for s in strings[::61]] + [b"", b"abcdefgh" * 6]
    b, o = synth.pack(strings)
    qb, qo = synth.pack(queries)
    taus = np.full(len(queries), 4, dtype=np.uint8)
    want, want_q = oracle.self_join(b, o, 4, banded=True), oracle.join(qb, qo, b, o, 4)
    mem = Memory(monkeypatch)

    def without(size, call):  # the first allocation of that size in the call is refused
        mem.refused, mem.refusals = [size], 0
        out = call()
        assert mem.refusals == 1, size
        return out

    planes, run_parts = 32 * len(queries), 32 << 18  # a string's planes, or a part of a run, are 32 bytes
    idx = without(32 * len(strings), lambda: pj.pj_build_index(strings, 4))
    assert np.array_equal(pj.pj_self_join(idx, 4).pairs, want)
    assert np.array_equal(pj.pj_query(idx, queries, 4).pairs, want_q)
    idx.free()
    idx = pj.pj_build_index(strings, 4)
    for size in (planes, run_parts):
        assert np.array_equal(without(size, lambda: pj.pj_query(idx, queries, 4)).pairs, want_q)
        assert np.array_equal(without(size, lambda: pj.pj_query_multi(idx, queries, taus)).pairs, want_q)
    for size in (planes, 32 << 12):
        plan = without(size, lambda: pj.Plan(idx, max_queries=len(queries), max_bytes=1 << 16))
        assert np.array_equal(plan.query(queries, taus).pairs, want_q)
        plan.free()
    idx.free()
    assert mem.now == 0
