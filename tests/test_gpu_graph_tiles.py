"""A self join that verifies its candidates by tiles is not recorded: the
recorded form, which has no tiles, would replay it slower."""
import numpy as np
import pytest

import oracle
from paper_1111_7171_gb300 import passjoin as pj
from paper_1111_7171_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles_from,replay", [("1", 0), (str(1 << 40), 1)])
def test_tiled_joins_stay_eager(tiles_from, replay, monkeypatch):
    monkeypatch.setenv("PJ_VERIFY_PAIRS", "0")
    monkeypatch.setenv("PJ_TILES_MIN_HITS", tiles_from)
    strings = synth.generate("short", 3, n=3000) + [b"", b"ab"]
    b, o = synth.pack(strings)
    want = oracle.self_join(b, o, 3)
    idx = pj.pj_build_index(strings, 3, graph_joins=True)
    for run in range(3):
        r = pj.pj_self_join(idx, 3)
        assert np.array_equal(r.pairs, want)
        assert r.stats["graph_replay"] == (replay if run else 0)
    idx.free()
