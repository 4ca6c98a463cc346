"""Attention over in-lists by eight lanes, a warp or a block per vertex, at the sizes where a lane's held scores run out (four or eight of them) and
where the next width takes over; several vertices of different lengths side by side, empty in-lists, every head count that has vectors of
scores, sampled and exact.  Rows against the oracle in 64 bits."""
from dataclasses import replace

import numpy as np
import pytest

import taurus_gen as tg
from helpers import csr_from_edges
from test_gpu_parity import _full_check

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("heads,fanout", [(1, 0), (2, 0), (4, 0), (8, 0), (2, 7), (8, 20)])
def test_widths(heads, fanout):
    V = 6_000
    rng = np.random.default_rng(10 * heads + fanout)
    edges = []
    for dst, n in enumerate((0, 1, 7, 8, 9, 31, 32, 33, 63, 64, 65, 127, 129, 255, 256, 257, 511, 1_023, 1_025, 2_047, 2_049, 4_095, 4_096, 4_097, 5_999, 0, 3)):
        edges += [(int(u), dst) for u in rng.choice(V, n, replace=False)]
    edges += [(int(u), int(v)) for u, v in zip(rng.integers(0, V, 9_000), rng.integers(40, V, 9_000))]
    row_ptr, col = csr_from_edges(V, edges)
    g = tg.Graph(V, len(edges), row_ptr, col, np.bincount(col, minlength=V).astype(np.int32))
    w = replace(tg.WORKLOADS["tiny"], V=V, E=g.E, dims=(24, 8 * heads), chunk=1_500, pool_slots=V, hub_count=0, fanout=(fanout,), mode=tg.GAT, gat_heads=heads)
    _full_check(w, g, dense_output=True)
