"""The gather of a resident pool at every size of the batches its warps take: one vertex, up to four at once, two batches a warp, and
full batches handed out from the counter; rows whose last lanes are idle and rows that end inside a 32-byte sector."""
from dataclasses import replace

import pytest

import taurus_gen as tg
from test_gpu_parity import _full_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [2_900, 7_400, 14_300, 40_000, 90_000])   # one chunk completes all of them; about 3 000 to 3 600 warps
@pytest.mark.parametrize("mode,dims", [(tg.SAGE_MEAN, (40, 36)), (tg.GCN_SYM, (70, 132)), (tg.GIN_SUM, (20, 100))])
def test_batches(V, mode, dims):
    w = tg.scaled(tg.WORKLOADS["mid"], V, chunk=V)
    w = replace(w, E=6 * V, dims=dims, fanout=(0,), pool_slots=V, hub_count=0, mode=mode)
    g = tg.make_graph(w)
    assert V < 14_000 or g.in_degree.max() > 256   # segments of long in-lists among the items
    _full_check(w, g, dense_output=True)
