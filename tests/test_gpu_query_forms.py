"""Forms of the query kernel that other tests do not reach: batches of mixed
thresholds whose largest needs more than a warp's 32 lanes a window, and lists
of long runs with room for some of them only."""
import numpy as np
import pytest

import oracle
from paper_1111_7171_gb300 import passjoin as pj
from paper_1111_7171_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tau_max", [31, 32])
def test_mixed_thresholds_wider_than_a_warp(tau_max):
    strings = synth.generate("medium", 8, n=150) + synth.generate("long", 32, n=60) + [b"", b"abc" * 9, b"x" * 33]
    queries = strings[::3] + [s[5:] + b"tail" for s in strings[1::7]]
    taus = np.array([(0, 3, 8, 16, 30, 31, tau_max)[k % 7] for k in range(len(queries))], dtype=np.uint8)
    b, o = synth.pack(strings)
    idx = pj.pj_build_index(strings, tau_max)
    plan = pj.Plan(idx, max_queries=len(queries), max_bytes=1 << 20)
    for got in (pj.pj_query_multi(idx, queries, taus).pairs, plan.query(queries, taus).pairs):
        for t in np.unique(taus).tolist():
            sel = np.flatnonzero(taus == t)
            qb, qo = synth.pack([queries[k] for k in sel.tolist()])
            g = got[np.isin(got["a"], sel)].copy()
            g["a"] = np.searchsorted(sel, g["a"])
            assert np.array_equal(g, oracle.join(qb, qo, b, o, int(t))), t
    plan.free()
    idx.free()


def test_room_for_some_of_the_long_runs():
    """A plan of one query has room for 4,096 parts of 256 postings; the 13
    window positions of this query find runs of 150,000 (587 parts) each in two
    kinds of strings, and some warps' parts fit where others' do not."""
    kinds = [b"a" * 15, b"aaaabaaaabaaaab"]
    n = 300_000
    idx = pj.pj_build_index([kinds[k & 1] for k in range(n)], 4)
    plan = pj.Plan(idx, max_queries=1, max_bytes=64)
    kb, ko = synth.pack(kinds)
    for query in (b"a" * 15, b"aaaabaaaaaaaaab", b"b" + b"a" * 14):
        qb, qo = synth.pack([query])
        ed = {int(b): int(e) for _, b, e in oracle.join(qb, qo, kb, ko, 4).tolist()}
        got = plan.query([query], [4]).pairs
        ids = np.flatnonzero(np.isin(np.arange(n) & 1, list(ed)))
        assert len(ids) and np.array_equal(got["b"], ids)
        assert np.array_equal(got["ed"], np.array([ed[k & 1] for k in ids.tolist()]))
        assert np.array_equal(pj.pj_query(idx, [query], 4).pairs, got)
    plan.free()
    idx.free()
