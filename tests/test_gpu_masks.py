"""Position masks of long strings' self joins against the oracle and against
the same join without them (an index under a device budget builds none)."""
import numpy as np
import pytest

import oracle
from paper_1111_7171_gb300 import passjoin as pj
from paper_1111_7171_gb300 import synth

pytestmark = pytest.mark.gpu


def edge_set(tau, seed):
    """Lengths around multiples of 32 (mask words) and of tau + 1 (segment
    lengths), strings too short to partition or with segments of at most four
    bytes, one long string, near copies, and few characters (repeats)."""
    rng = np.random.default_rng(seed)
    parts = tau + 1
    lens = [0, 3, tau, parts, 2 * parts, 4 * parts + 1, 5 * parts - 1, 5 * parts, 5 * parts + 1, 5 * parts + tau, 2001]
    lens += [k * parts + d for k in range(12, 30) for d in (-1, 0, 1, tau // 2)]
    lens += [32 * k + d for k in range(9, 20) for d in (-1, 0, 1)]
    out = []
    for n in lens:
        alphabet = int(rng.integers(2, 40))
        base = rng.integers(0, alphabet, size=n) + 60
        out.append(bytes(base.astype(np.uint8)))
        for _ in range(2):
            b = list(base)
            for _ in range(int(rng.integers(0, tau + 1))):
                at = int(rng.integers(0, len(b) + 1))
                if rng.random() < 0.5 and at < len(b):
                    del b[at]
                else:
                    b.insert(at, int(rng.integers(60, 60 + alphabet)))
            out.append(bytes(np.array(b, dtype=np.uint8)))
    return [out[k] for k in rng.permutation(len(out))]


@pytest.mark.parametrize("form", [{}, {"PJ_FUSED": "1"}, {"PJ_FUSED": "2"}, {"PJ_VERIFY_PAIRS": "0"},
                                  {"PJ_PROBE_INTERLEAVE": "1"}, {"PJ_GROUP_BUDGET": "20000"}])
@pytest.mark.parametrize("tau,scheme", [(20, "even"), (32, "even"), (27, "center")])
def test_masks_match_oracle(tau, scheme, form, monkeypatch):
    strings = edge_set(tau, tau)
    for k, x in form.items():
        monkeypatch.setenv(k, x)
    b, o = synth.pack(strings)
    want = oracle.self_join(b, o, tau, banded=True)
    got = []
    for budget in (0, 4 << 30):
        idx = pj.pj_build_index(strings, tau, partition=scheme, device_budget=budget)
        got.append(pj.pj_self_join(idx, tau))
        assert np.array_equal(got[-1].pairs, want)
        idx.free()
    for key in ("lookups", "candidates", "accepted", "hits"):
        assert got[0].stats[key] == got[1].stats[key], key
