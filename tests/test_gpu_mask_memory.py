"""The device memory that position masks take (long strings, high thresholds),
against the same index under a device budget, which has none."""
import pytest

from paper_1111_7171_gb300 import passjoin as pj
from paper_1111_7171_gb300 import synth

pytestmark = pytest.mark.gpu

TAU = 32


def indexes():
    strings = synth.generate("long", TAU, n=400)
    # 12 bytes for every 32 characters and part of them
    masks = 12 * ((sum(map(len, strings)) >> 5) + len(strings) + 1)
    return strings, masks, [pj.pj_build_index(strings, TAU, lazy_partitions=True, device_budget=b) for b in (0, 4 << 30)]


def test_masks_are_counted():
    _, masks, (idx, without) = indexes()
    for i in (idx, without):
        pj.pj_self_join(i, TAU)
    assert idx.device_bytes - without.device_bytes == masks
    idx.free()
    without.free()
