"""The pull form of resident pools where one in-list or one row is out of the ordinary: in-lists long enough for every width of the
attention sweeps, and rows that hold infinities or NaN."""
from dataclasses import replace

import numpy as np
import pytest

import taurus_gen as tg
from gpu_harness import run_library, run_oracle
from helpers import csr_from_edges
from test_gpu_parity import _full_check

pytestmark = pytest.mark.gpu


def _graph(V, edges):
    row_ptr, col = csr_from_edges(V, edges)
    return tg.Graph(V, len(edges), row_ptr, col, np.bincount(col, minlength=V).astype(np.int32))


@pytest.mark.parametrize("heads,fanout", [(1, 0), (3, 0), (16, 0), (4, 10)])
def test_attention_of_long_in_lists(heads, fanout):
    """In-lists at and around the limits of the sweeps: 256 / 257 entries (a warp, a block of eight), 4 096 / 4 097 (eight warps,
    thirty-two), 9 000."""
    V = 9_500
    rng = np.random.default_rng(heads)
    edges = [(int(u), int(v)) for u, v in zip(rng.integers(0, V, 30_000), rng.integers(100, V, 30_000))]
    for dst, n in ((3, 255), (7, 256), (11, 257), (40, 4_095), (41, 4_096), (42, 4_097), (60, 9_000)):
        edges += [(int(u), dst) for u in rng.choice(V, n, replace=False)]
    g = _graph(V, edges)
    assert [int(g.in_degree[d]) for d in (7, 11, 41, 42, 60)] == [256, 257, 4_096, 4_097, 9_000]
    w = replace(tg.WORKLOADS["tiny"], V=V, E=g.E, dims=(24, 16 * heads), chunk=2_000, pool_slots=V, hub_count=0, fanout=(fanout,), mode=tg.GAT,
                gat_heads=heads)
    _full_check(w, g, dense_output=True)


@pytest.mark.parametrize("value", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("mode,heads,dims", [(tg.SAGE_MEAN, 1, (40, 24)), (tg.SAGE_MEAN, 1, (24, 48)), (tg.GCN_SYM, 1, (20, 16)),
                                             (tg.GIN_SUM, 1, (16, 130)), (tg.GAT, 1, (24, 32)), (tg.GAT, 4, (24, 64))])
def test_a_row_that_is_not_finite_shows_in_its_destinations_only(mode, heads, dims, value):
    V, bad = 3_000, 1_234
    w = replace(tg.scaled(tg.WORKLOADS["mid"], V, chunk=512), dims=dims, fanout=(0,), pool_slots=V, hub_count=0, mode=mode, gat_heads=heads)
    g, model = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
    big = int(np.argmax(g.in_degree))
    assert g.in_degree[big] > 256                      # summed in segments
    x0 = tg.features(w.seed, 0, 0, V, dims[0])
    row = g.row_ptr
    # a source of the vertex whose in-list is summed in segments
    source = next(u for u in range(bad, V) if big in g.col_idx[row[u]:row[u + 1]] and u != big)
    x1 = x0.copy()
    x1[source, dims[0] // 2] = value
    touched = np.zeros(V, bool)
    touched[source] = True
    touched[g.col_idx[row[source]:row[source + 1]]] = True
    clean = run_oracle(w, g, model, x0)["outs"][0]
    lib = run_library(w, g, model, x1, dense_output=True)
    got = lib["outs"][0]
    assert np.array_equal(~np.isfinite(got).all(axis=1), touched)
    err = np.abs(got[~touched] - clean[~touched]).max(axis=1) / (np.abs(clean[~touched]).max(axis=1) + 1e-6)
    assert err.max() <= 1e-4
    # nothing of it is left for the next pass over the same context
    import torch
    dense = torch.zeros((V, dims[1]), device="cuda:0")
    feat = torch.from_numpy(x0).cuda()
    ctx = lib["ctx"]
    ctx.layer_begin(0)
    src = feat
    chunks = [(s, min(s + w.chunk, V)) for s in range(0, V, w.chunk)]
    if mode == tg.GAT:
        src = torch.empty((V, dims[1]), device="cuda:0")
        for s, e in chunks:
            ctx.gat_project_chunk(s, e, feat[s:e], src[s:e], dims[1])
        ctx.gat_attention()
    ctx.layer_set_dense_output(dense, dims[1])
    for s, e in chunks:
        ctx.push_chunk(s, e, src[s:e])
    ctx.layer_end()
    again = dense.cpu().numpy()
    assert (np.abs(again - clean).max(axis=1) / (np.abs(clean).max(axis=1) + 1e-6)).max() <= 1e-4
