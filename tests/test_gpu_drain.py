"""taurus_drain_dense without an id buffer, where the kernel that places the rows also empties the buffer: a buffer that holds the rows
of one push at most, so that a count left standing overflows it, and drains with and without ids in turn."""
from dataclasses import replace

import numpy as np
import pytest

import taurus_gen as tg
from gpu_harness import row_error, run_oracle

pytestmark = pytest.mark.gpu


def _layer(w, g, model, feat, plan, drain_rows, with_ids):
    """Layer 0 with a drain after every push; with_ids: per push, whether the drain hands out ids.  Returns rows and counts."""
    import torch
    import paper_2607_17374_b200 as tb
    V, d_out = g.V, w.dims[1]
    ctx = tb.Context(V, g.E, g.row_ptr, g.col_idx, g.in_degree, w.mode, w.dims, model.W_neigh, model.W_self, model.bias, model.act, w.chunk,
                     w.pool_slots, w.hub_count, w.fanout, w.seed, 0 if w.pool_slots >= V else V - w.hub_count, drain_rows, w.gemm_mode, 0, 0, w.gin_eps)
    dense = torch.zeros((V, d_out), device="cuda")
    ids = torch.empty(V, dtype=torch.int64, device="cuda")
    placed, counts = [], []
    ctx.layer_begin(0)
    for i, (s, e) in enumerate(plan):
        ctx.push_chunk(s, e, feat[s:e])
        n = ctx.drain_dense(dense, d_out, V, ids if with_ids[i] else None)
        counts.append(n)
        if with_ids[i]:
            placed.append(ids[:n].cpu().numpy().copy())
        assert ctx.drain_dense(dense, d_out, V) == 0 and ctx.drain_dense(dense, d_out, V, ids) == 0
    assert ctx.layer_end()["completed"] == V
    out = dense.cpu().numpy()
    ctx.destroy()
    return out, counts, placed


@pytest.mark.parametrize("mode", [tg.SAGE_MEAN, tg.GIN_SUM])
@pytest.mark.parametrize("pool,step", [("all", 1024), ("all", 700), ("bounded", 1024)])   # resident on and off the chunk grid, evicting
def test_drains_without_ids(mode, pool, step):
    import torch
    V = 30_000
    w = tg.scaled(tg.WORKLOADS["large"], V, chunk=1024)
    w = replace(w, dims=(40, 37), fanout=(0,), hub_count=30, mode=mode, pool_slots=V if pool == "all" else 12_000)
    g, model = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
    x0 = tg.features(w.seed, 0, 0, V, w.dims[0])
    feat = torch.from_numpy(x0).cuda()
    plan = [(s, min(s + step, V)) for s in range(0, V, step)]
    orc = run_oracle(w, g, model, x0)
    want = orc["outs"][0]
    assert pool == "all" or orc["sims"][0].stats["evictions"] > 1_000
    every = [True] * len(plan)
    out, counts, placed = _layer(w, g, model, feat, plan, V, every)
    assert np.array_equal(np.sort(np.concatenate(placed)), np.arange(V)) and row_error(out, want)[0] <= 1e-4
    room = max(counts) + 256   # (the bound on a push's completions counts in blocks of 64 of either end)
    assert sum(counts) > 1.2 * room
    for with_ids in ([False] * len(plan), [i % 3 == 1 for i in range(len(plan))]):
        out, got, placed = _layer(w, g, model, feat, plan, room, with_ids)
        assert got == counts
        assert [p.size for p in placed] == [n for n, has in zip(counts, with_ids) if has]
        assert row_error(out, want)[0] <= 1e-4


@pytest.mark.parametrize("pinned", [False, True])
def test_a_drain_that_does_not_fit_takes_nothing(pinned):
    """Capacity below the rows that wait: refused, whole, and the next drain has them all.  Many blocks and one."""
    import torch
    import paper_2607_17374_b200 as tb
    for V, chunk in ((30_000, 8_192), (40, 40)):
        w = tg.scaled(tg.WORKLOADS["large"], V, chunk=chunk)
        w = replace(w, dims=(40, 37), fanout=(0,), hub_count=1, mode=tg.GIN_SUM, pool_slots=V)
        g, model = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
        x0 = tg.features(w.seed, 0, 0, V, w.dims[0])
        feat = torch.from_numpy(x0).cuda()
        ctx = tb.Context(V, g.E, g.row_ptr, g.col_idx, g.in_degree, w.mode, w.dims, model.W_neigh, model.W_self, model.bias, model.act, w.chunk,
                         w.pool_slots, w.hub_count, w.fanout, w.seed, 0, V, w.gemm_mode, 0, 0, w.gin_eps)
        dense = torch.zeros((V, 37), pin_memory=True) if pinned else torch.zeros((V, 37), device="cuda")
        total = 0
        ctx.layer_begin(0)
        for s in range(0, V, chunk):
            ctx.push_chunk(s, min(s + chunk, V), feat[s:s + chunk])
            before = dense.clone()
            if s + chunk >= V:
                with pytest.raises(tb.TaurusError):
                    ctx.drain_dense(dense, 37, V - total - 1)
                assert torch.equal(dense, before)
            total += ctx.drain_dense(dense, 37, V - total)
        assert total == V and ctx.layer_end()["completed"] == V
        assert row_error(dense.cpu().numpy(), run_oracle(w, g, model, x0)["outs"][0])[0] <= 1e-4
