"""Pools that hold every vertex (the pull form of a layer) at the sizes where it can go wrong: every split of a row over lanes
and both sides of its limits, in-lists longer than one segment (summed in pieces), sampled layers, hubs that own no slot,
pushes that are not cells of the chunk grid, one to sixteen attention heads, and one chunk that holds the whole graph.
Rows against the oracle in 64 bits, accounting exact."""
from dataclasses import replace

import numpy as np
import pytest

import taurus_gen as tg
from gpu_harness import run_library
from test_gpu_parity import _full_check

pytestmark = pytest.mark.gpu


def _workload(V, chunk, dims, **kw):
    w = tg.scaled(tg.WORKLOADS["mid"], V, chunk=chunk)
    return replace(w, dims=dims, fanout=kw.pop("fanout", (0,) * (len(dims) - 1)), pool_slots=V, **kw)


@pytest.mark.parametrize("mode", [tg.SAGE_MEAN, tg.GCN_SYM, tg.GIN_SUM])
@pytest.mark.parametrize("width", [1, 4, 16, 17, 32, 33, 48, 49, 64, 65, 100, 128, 132, 256, 260, 512, 516, 1024])
def test_row_widths(width, mode):
    w = _workload(3_000, 512, (width, max(1, width // 2)), mode=mode)           # the projected rows, half as wide
    g = tg.make_graph(w)
    assert g.in_degree.max() > 384                                              # in-lists of more than two segments
    _full_check(w, g)
    if 4 * (width // 2 + 3) <= 3 * width:
        _full_check(replace(w, dims=(width // 2, width)), g, dense_output=True)   # input rows summed, then transformed


@pytest.mark.parametrize("heads,width", [(1, 8), (2, 24), (3, 36), (4, 128), (5, 60), (8, 256), (16, 64), (16, 512)])
def test_attention_heads(heads, width):
    w = _workload(2_500, 400, (20, width), mode=tg.GAT, gat_heads=heads)
    _full_check(w, dense_output=True)


@pytest.mark.parametrize("plan", ["grid", "ragged", "one"])
@pytest.mark.parametrize("fanout", [0, 1, 10, 64])
@pytest.mark.parametrize("hubs", [0, 25])
def test_push_plans_sampling_and_hubs(plan, fanout, hubs):
    V = 4_001
    w = _workload(V, V if plan == "one" else 600, (24, 40, 7), fanout=(fanout, 0), hub_count=hubs)
    if plan == "ragged":   # the push form of the same pushes is the reference: the simulation knows grid chunks only
        g, model = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
        x0 = tg.features(w.seed, 0, 0, V, w.dims[0])
        chunks = [(s, min(s + 457, V)) for s in range(0, V, 457)]
        a = run_library(w, g, model, x0, chunk_plan=chunks)
        b = run_library(w, g, model, x0, chunk_plan=chunks, flags=4)   # CSR-order kernels
        for l in range(w.L):
            assert {k: v for k, v in a["stats"][l].items()} == {k: v for k, v in b["stats"][l].items()}
            assert all((a["chunk_log"][l][k] == b["chunk_log"][l][k]).all() for k in a["chunk_log"][l])
            assert all(sorted(x) == sorted(y) for x, y in zip(a["completed"][l], b["completed"][l]))
            assert np.linalg.norm(a["outs"][l] - b["outs"][l]) <= 1e-5 * np.linalg.norm(b["outs"][l])
        return
    lib, orc = _full_check(w)
    # one group per destination and chunk that its kept in-edges come from
    assert lib["stats"][0]["scatter_groups"] <= lib["stats"][0]["total_messages"] == int(np.asarray(orc["msets"][0].m).sum())
