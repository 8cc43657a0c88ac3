"""Plans of many queries: room for the parts of long posting runs grows with
the batch (without it most runs are walked unevenly, by the warps that found
them), and batches of more than 2^18 groups are answered by the probe passes
where the strings are short."""
import numpy as np
import pytest

pytest.importorskip("torch")

from paper_1111_7171_gb300 import passjoin as pj
from paper_1111_7171_gb300 import synth
from test_gpu_tight_memory import Memory

pytestmark = pytest.mark.gpu

PART_BYTES = 32


def test_plan_has_room_for_four_parts_a_group():
    idx = pj.pj_build_index(synth.generate("short", 4, n=20_000), 4)
    groups = 5 * 9  # of a query at tau 4: tau + 1 segments of 2 tau + 1 lengths
    small, large = (pj.Plan(idx, max_queries=n, max_bytes=1 << 20, accepted_capacity=1 << 16, pairs_capacity=1 << 16)
                    for n in (64, 5_000))
    more = large.info()["device_bytes"] - small.info()["device_bytes"]
    assert more >= PART_BYTES * (4 * groups * 5_000 - 4096)
    small.free()
    large.free()
    idx.free()


@pytest.mark.parametrize("hits_capacity", [0, 1])
def test_large_batches_take_the_probe_passes(hits_capacity):
    strings = synth.generate("short", 4, n=20_000) + [b"", b"ab", b"abcd"]
    idx = pj.pj_build_index(strings, 4)
    queries = [s[1:] + s[:1] for s in strings[:16_000]]
    taus = (np.arange(len(queries)) % 5).astype(np.uint8)  # 19 groups on average, 304,000 in all
    plan = pj.Plan(idx, max_queries=16_384, max_bytes=1 << 20, hits_capacity=hits_capacity)
    got = plan.query(queries, taus)
    passes = plan.info()["graph_kernels"]
    q = len(queries) // 4
    lookups = hits = 0
    for k in range(4):  # in quarters, eager: the query kernel
        want = pj.pj_query_multi(idx, queries[k * q:(k + 1) * q], taus[k * q:(k + 1) * q])
        lookups, hits = lookups + want.stats["lookups"], hits + want.stats["hits"]
        part = got.pairs[(got.pairs["a"] >= k * q) & (got.pairs["a"] < (k + 1) * q)].copy()
        part["a"] -= k * q
        assert np.array_equal(part, want.pairs)
        assert np.array_equal(plan.query(queries[k * q:(k + 1) * q], taus[k * q:(k + 1) * q]).pairs, want.pairs)
        assert plan.info()["graph_kernels"] < passes
    assert (got.stats["lookups"], got.stats["hits"]) == (lookups, hits)
    again = plan.query(queries, taus)
    assert np.array_equal(again.pairs, got.pairs) and plan.info()["graph_kernels"] == passes
    plan.free()
    idx.free()


@pytest.mark.parametrize("refused", [4 * 45 * 16_384, 8 * 45 * 16_384, 32 * 2 * 45 * 16_384, 32 << 20])
def test_large_plans_without_memory(refused, monkeypatch):
    """Group counts, masks, hits (32 bytes, two a group) or the parts' room
    refused once: the plan does without, or with less room."""
    strings = synth.generate("short", 4, n=20_000)
    mem = Memory(monkeypatch)
    idx = pj.pj_build_index(strings, 4)
    queries, taus = strings[:16_000], (np.arange(16_000) % 5).astype(np.uint8)
    want = pj.pj_query_multi(idx, queries, taus).pairs
    mem.refused, mem.refusals = [refused], 0
    plan = pj.Plan(idx, max_queries=16_384, max_bytes=1 << 20)
    assert mem.refusals == 1
    assert np.array_equal(plan.query(queries, taus).pairs, want)
    plan.free()
    idx.free()
    assert mem.now == 0
