"""The destination-grouped scatter at the sizes where its spans and tiles change: chunks of fewer edges than eight a sub-group of lanes, of
more than a span of 128 a warp, and between, whose last span is short; every split of a row over lanes; pools that evict (blocks beside the row
transfers) and pools that hold every vertex.  Rows against the oracle in 64 bits, its accounting exact."""
from dataclasses import replace

import pytest

import taurus_gen as tg
from test_gpu_parity import _full_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,chunk,width,bounded", [
    (3_000, 100, 256, True), (30_000, 2_100, 256, True), (60_000, 20_000, 256, False), (120_000, 61_003, 128, False), (9_000, 7, 64, True),
    (30_000, 4_100, 12, False), (30_000, 1_100, 12, True), (90_000, 45_001, 20, False), (60_000, 3_000, 48, True), (60_000, 3_000, 48, False),
    (50_000, 30_011, 100, False), (100_000, 9_000, 100, True), (40_000, 4_000, 300, True), (12_000, 3_000, 520, False),
])
def test_spans(V, chunk, width, bounded):
    w = replace(tg.scaled(tg.WORKLOADS["large"], V, chunk=chunk), dims=(16, width), fanout=(0,), pool_slots=V * 15 // 16 if bounded else V, hub_count=7)
    lib, _ = _full_check(w, flags=8 if bounded else 8 + 16)   # project-first; the push form of a pool that holds every vertex
    groups, messages = lib["stats"][0]["scatter_groups"], lib["stats"][0]["total_messages"]
    assert 0 < groups <= messages
