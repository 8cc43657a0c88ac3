"""Signatures and bit planes made by a warp per string (small sets, batches
and plans, long strings): too many set bits would drop similar pairs."""
import numpy as np
import pytest

import oracle
from paper_1111_7171_gb300 import passjoin as pj
from paper_1111_7171_gb300 import synth

pytestmark = pytest.mark.gpu


def edge_set(seed):
    """Lengths around a warp's 32 characters and the planes' 28, alphabets of
    one character (counts past their limit of 4) to all bytes, near copies."""
    rng = np.random.default_rng(seed)
    out = []
    for n in (0, 1, 5, 27, 28, 29, 31, 32, 33, 63, 64, 65, 129, 700):
        for alphabet in (1, 2, 5, 40, 256):
            base = rng.integers(0, alphabet, size=n) + (0 if alphabet == 256 else 60)
            out.append(bytes(base.astype(np.uint8)))
            for _ in range(3):
                b = base.copy()
                for _ in range(int(rng.integers(0, 4))):
                    if len(b):
                        b[int(rng.integers(0, len(b)))] = int(rng.integers(0, 256))
                out.append(bytes(b.astype(np.uint8)))
    return [out[k] for k in rng.permutation(len(out))]


@pytest.mark.parametrize("tau", [1, 3, 6])
@pytest.mark.parametrize("pairs", ["0", "1"])
def test_signatures_match_oracle(tau, pairs, monkeypatch):
    monkeypatch.setenv("PJ_VERIFY_PAIRS", pairs)
    strings, queries = edge_set(7), edge_set(7)[::3] + edge_set(8)
    b, o = synth.pack(strings)
    qb, qo = synth.pack(queries)
    want = oracle.join(qb, qo, b, o, tau)
    idx = pj.pj_build_index(strings, tau)
    assert np.array_equal(pj.pj_self_join(idx, tau).pairs, oracle.self_join(b, o, tau))
    assert np.array_equal(pj.pj_query(idx, queries, tau).pairs, want)
    plan = pj.Plan(idx, max_queries=len(queries), max_bytes=1 << 20)
    assert np.array_equal(plan.query(queries, np.full(len(queries), tau, dtype=np.uint8)).pairs, want)
    plan.free()
    idx.free()
