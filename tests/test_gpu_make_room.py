"""Bounded pools at the sizes where the one-launch make-room step and the row transfers can go wrong: row widths of one
float4 up to the widest (entries in flight per block 256 down to 28), pools around one tile of the victim select (2 048
slots), few and many victims per chunk.  The oracle's accounting is exact, its rows are in 64 bits."""
from dataclasses import replace

import pytest

import taurus_gen as tg
from test_gpu_parity import _full_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,chunk,pool,width,policy", [
    (5_000, 64, 2_047, 4, 0), (5_000, 64, 2_048, 100, 1), (5_000, 100, 2_049, 256, 2), (12_000, 128, 4_097, 36, 3),
    (4_000, 100, 2_100, 1_024, 0), (60_000, 512, 20_000, 12, 0),
])
def test_make_room_and_transfer_sizes(V, chunk, pool, width, policy):
    w = replace(tg.scaled(tg.WORKLOADS["large"], V, chunk=chunk), dims=(16, width), fanout=(0,), pool_slots=pool, hub_count=7)
    lib, _ = _full_check(w, flags=8, evict_policy=policy)   # project-first: accumulator rows as wide as the output
    assert lib["stats"][0]["evictions"] > 0 and lib["stats"][0]["reloads"] == lib["stats"][0]["evictions"]


@pytest.mark.parametrize("V,chunk,pool,width,mb", [(40_000, 2_600, 34_000, 1_024, 128), (140_000, 9_000, 125_000, 256, 128),
                                                   (130_000, 8_600, 116_000, 1_024, 512)])
def test_pushes_that_touch_many_rows(V, chunk, pool, width, mb):
    """The wider splits of the row transfers (sixteen and thirty-two blocks instead of eight), which the victim select and the projection
    leave room for."""
    w = replace(tg.scaled(tg.WORKLOADS["large"], V, chunk=chunk), dims=(16, width), fanout=(0,), pool_slots=pool, hub_count=7)
    g = tg.make_graph(w)
    assert 4 * width * min(V, chunk + max(int(g.row_ptr[min(V, s + chunk)] - g.row_ptr[s]) for s in range(0, V, chunk))) > mb * 1e6
    lib, _ = _full_check(w, g, flags=8)
    assert lib["stats"][0]["evictions"] > 0 and lib["stats"][0]["reloads"] == lib["stats"][0]["evictions"]
