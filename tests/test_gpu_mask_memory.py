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


def test_masks_wait_for_a_self_join():
    """Only self joins read masks: building, queries and R x S joins make none."""
    strings, masks, (idx, without) = indexes()
    for i in (idx, without):
        assert len(pj.pj_query(i, strings[:3], TAU).pairs) >= 3  # builds the threshold
    assert idx.device_bytes == without.device_bytes
    first = [pj.pj_self_join(i, TAU).pairs for i in (idx, without)]
    assert len(first[0]) and (first[0] == first[1]).all()
    assert idx.device_bytes - without.device_bytes == masks
    idx.free()
    without.free()
