"""Run-major extension verification (hits grouped by posting run, tiles of
postings x hits, bit-plane sides) against the oracle and the queued form, at
the sizes where tiles and planes can go wrong."""
import numpy as np
import pytest

import oracle
from paper_1111_7171_gb300 import passjoin as pj
from paper_1111_7171_gb300 import synth

pytestmark = pytest.mark.gpu


def edge_set(tau, seed):
    """Runs of 1, 31..33, 127..129 and 700 equal strings (a tile is 128
    postings by 256 hits), lengths around the planes' 28 and the shortest
    partitioned one, empty strings, and bytes of every value."""
    rng = np.random.default_rng(seed)
    out = [b"", b"", b"a", b"ab"]
    for copies in (1, 31, 32, 33, 127, 128, 129, 700):
        base = bytes(rng.integers(97, 101, size=int(rng.integers(tau + 1, 12))).tolist())
        out += [base] * copies
    for n in (tau, tau + 1, 27, 28, 29, 30, 40, 70):
        for _ in range(12):
            base = bytearray(rng.integers(97, 100, size=n).tolist())
            out.append(bytes(base))
            for _ in range(3):  # near copies with an odd byte
                b = bytearray(base)
                if b:
                    b[int(rng.integers(0, len(b)))] = int(rng.integers(0, 256))
                out.append(bytes(b) + bytes(rng.integers(97, 100, size=int(rng.integers(0, 2))).tolist()))
    return [out[k] for k in rng.permutation(len(out))]


@pytest.mark.parametrize("tau", [0, 1, 2, 3, 4, 5, 9])
@pytest.mark.parametrize("knobs", [{}, {"PJ_LAUNCH_CANDS": "5000", "PJ_ACCEPT_INITIAL": "16", "PJ_ACCEPT_RESERVE": "0",
                                        "PJ_GROUP_BUDGET": "3000"}])
def test_tiles_match_oracle(tau, knobs, monkeypatch):
    strings = edge_set(tau, 40 + tau)
    monkeypatch.setenv("PJ_VERIFY_PAIRS", "0")
    monkeypatch.setenv("PJ_TILES_MIN_HITS", str(1 << 40))
    idx = pj.pj_build_index(strings, tau)
    queued = pj.pj_self_join(idx, tau)
    monkeypatch.setenv("PJ_TILES_MIN_HITS", "1")
    for k, x in knobs.items():
        monkeypatch.setenv(k, x)
    tiled = pj.pj_self_join(idx, tau)
    b, o = synth.pack(strings)
    assert np.array_equal(tiled.pairs, oracle.self_join(b, o, tau))
    for key in ("lookups", "candidates", "accepted", "hits", "dp_cells", "filtered"):
        assert tiled.stats[key] == queued.stats[key], key
    queries = strings[::7] + edge_set(tau, 90 + tau)[::3]
    qb, qo = synth.pack(queries)
    assert np.array_equal(pj.pj_query(idx, queries, tau).pairs, oracle.join(qb, qo, b, o, tau))
    idx.free()


@pytest.mark.parametrize("scheme", ["even", "center"])
def test_tiles_on_names(scheme, monkeypatch):
    strings = synth.generate("short", 4, n=6001)
    monkeypatch.setenv("PJ_TILES_MIN_HITS", "1")
    idx = pj.pj_build_index(strings, 4, partition=scheme)
    b, o = synth.pack(strings)
    assert np.array_equal(pj.pj_self_join(idx, 4).pairs, oracle.self_join(b, o, 4, banded=True))
    idx.free()
