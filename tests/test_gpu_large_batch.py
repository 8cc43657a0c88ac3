"""Plans of many queries: room for the parts of long posting runs grows with
the batch (without it most runs are walked unevenly, by the warps that found
them)."""
import pytest

from paper_1111_7171_gb300 import passjoin as pj
from paper_1111_7171_gb300 import synth

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
