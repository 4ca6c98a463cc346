"""Rows that the push behind the one that evicted them takes back: out of the staging buffer where the rows of both pushes fit it side by
side, else from the host store.  Row widths of one float4 up to the widest, pushes with and without room for both, pushes that are not
grid cells.  The oracle's accounting is exact, its rows are in 64 bits."""
from dataclasses import replace

import numpy as np
import pytest

import taurus_gen as tg
from gpu_harness import run_library, run_oracle
from helpers import csr_from_edges
from test_gpu_parity import FP32_TOL, _compare_layers, _full_check

pytestmark = pytest.mark.gpu


def _workload(V, chunk, pool, width):
    return replace(tg.scaled(tg.WORKLOADS["large"], V, chunk=chunk), dims=(16, width), fanout=(0,), pool_slots=pool, hub_count=7)


@pytest.mark.parametrize("V,chunk,pool,width", [
    (20_000, 64, 5_500, 256), (20_000, 150, 6_000, 4), (12_000, 200, 4_200, 100), (12_000, 700, 8_500, 36), (9_000, 64, 2_500, 1_024),
    (20_000, 1_500, 13_000, 64),
])
def test_rows_back_in_the_next_push(V, chunk, pool, width):
    lib, _ = _full_check(_workload(V, chunk, pool, width), flags=8)   # project-first: accumulator rows as wide as the output
    assert lib["stats"][0]["evictions"] > 0 and lib["stats"][0]["reloads"] == lib["stats"][0]["evictions"]


@pytest.mark.parametrize("sizes", [(64, 37, 1, 64, 27), (100, 28), (128, 64, 5, 59)])
def test_pushes_off_the_grid(sizes):
    w = _workload(16_000, 128, 4_800, 48)
    g, model = tg.make_graph(w), tg.make_model(w)
    x0 = tg.features(w.seed, 0, 0, g.V, w.dims[0])
    plan, s = [], 0
    while s < g.V:
        plan.append((s, min(g.V, s + sizes[len(plan) % len(sizes)])))
        s = plan[-1][1]
    lib = run_library(w, g, model, x0, flags=8, chunk_plan=plan)
    _compare_layers(lib, run_oracle(w, g, model, x0), FP32_TOL)
    st = lib["stats"][0]
    assert st["completed"] == g.V and st["evictions"] > 0 and st["reloads"] == st["evictions"]
    ids = np.concatenate([x[1] if isinstance(x, tuple) else x for x in lib["completed"][0]])
    assert ids.size == g.V and np.unique(ids).size == g.V


def test_no_room_for_two_pushes():
    """Sources of 18 random edges in two stretches, of 6 elsewhere: pushes of the one kind evict more than half of what the staging buffer
    holds, so the next one finds no row of theirs there; pushes of the other kind leave room."""
    V, chunk, pool = 16_000, 100, 2_000
    rng = np.random.default_rng(5)
    edges = [(u, int(v)) for u in range(V) for v in rng.integers(0, V, 18 if u // 4_000 % 2 == 0 else 6)]
    row_ptr, col = csr_from_edges(V, edges)
    g = tg.Graph(V, len(edges), row_ptr, col, np.bincount(col, minlength=V).astype(np.int32))
    w = replace(_workload(V, chunk, pool, 128), E=g.E, hub_count=0)
    lib, orc = _full_check(w, g, flags=8)
    moved = orc["sims"][0].per_chunk["ev"]   # rows taken back by each push; in steady state as many leave
    both = moved[1:-1] + moved[2:]
    assert (both > pool).any() and ((both < pool) & (moved[2:] > 100)).any()
    assert lib["stats"][0]["reloads"] == lib["stats"][0]["evictions"]
