"""Small batches: the kernels that a batch of one query launches, and the bit
planes of queries, which small batches get with their signatures from one
kernel and large ones from a kernel of their own."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_1111_7171_gb300 import passjoin as pj
from paper_1111_7171_gb300 import synth

pytestmark = pytest.mark.gpu


def test_launches_of_one_query():
    """Lengths, signature and planes, the query and its long runs, heads, scan
    and emission of one pair (one match is not sorted)."""
    idx = pj.pj_build_index(synth.generate("short", 2, n=500) + [b"quite another one"], 1)
    q = torch.tensor(list(b"quite another one"), dtype=torch.uint8, device="cuda")
    off = torch.tensor([0, len(q)], dtype=torch.int64, device="cuda")
    out = torch.empty(48, dtype=torch.int32, device="cuda")
    assert pj.pj_query_noalloc(idx, (q, off), 0, out, 16) == 1
    before = pj.pj_kernel_launches()
    assert pj.pj_query_noalloc(idx, (q, off), 0, out, 16) == 1
    assert pj.pj_kernel_launches() - before <= 7
    idx.free()


@pytest.mark.parametrize("tau", [1, 3, 4])
def test_planes_of_small_and_large_batches(tau):
    rng = np.random.default_rng(tau)
    S = [bytes(rng.choice(list(b"abc\xff"), size=n).tolist()) for n in rng.integers(14, 32, size=300)]
    # every other one a character longer, every third with a foreign character
    Q = [(b"a" if k & 1 else b"") + s[:-1] + (b"z" if k % 3 == 0 else s[-1:]) for k, s in enumerate(S)]
    b, o = synth.pack(S)
    want = oracle.join(*synth.pack(Q), b, o, tau)
    idx = pj.pj_build_index(S, tau)
    small = pj.pj_query(idx, Q, tau).pairs
    assert len(want) and np.array_equal(small, want)
    times = 40_000 // len(Q)  # more strings than the one kernel takes
    large = pj.pj_query(idx, Q * times, tau).pairs
    assert len(large) == times * len(want)
    for k in (0, times // 2, times - 1):
        part = large[k * len(want):(k + 1) * len(want)].copy()
        part["a"] -= k * len(Q)
        assert np.array_equal(part, want)
    idx.free()
