"""Small pushes to pools that hold every vertex: their accounting runs in the first blocks of the launch that writes the rows, whichever kernel
that is, and either kernel of a push may come up while the one before it still runs.  Sizes on both sides of the rules (blocks that fit beside the
projection's, 65 536 rows), one row to several blocks; rows against the oracle in 64 bits, its accounting exact."""
from dataclasses import replace

import pytest

import taurus_gen as tg
from test_gpu_parity import _full_check
from gpu_harness import row_error, run_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dense", [False, True])
@pytest.mark.parametrize("mode,dims", [(tg.SAGE_MEAN, (64, 64)), (tg.GIN_SUM, (47, 33)), (tg.GCN_SYM, (20, 72)), (tg.SAGE_MEAN, (36, 100)), (tg.GAT, (64, 32))])
@pytest.mark.parametrize("V,chunk", [(40, 1), (900, 100), (5_000, 1_024), (17_000, 8_500), (30_000, 12_000), (66_000, 65_536), (66_000, 65_537)])
def test_sizes(V, chunk, mode, dims, dense):
    w = replace(tg.scaled(tg.WORKLOADS["large"], V, chunk=chunk), dims=dims, fanout=(0,), pool_slots=V, hub_count=min(7, V // 8), mode=mode)
    _full_check(w, dense_output=dense)


@pytest.mark.parametrize("fanout", [0, 5])
def test_rows_written_and_overwritten_on_the_stream(fanout):
    """One buffer, filled by a kernel in front of every push and spoilt by one behind it, pushes on two streams in turn."""
    import torch
    import paper_2607_17374_b200 as tb
    V, chunk = 20_000, 512
    w = replace(tg.scaled(tg.WORKLOADS["large"], V, chunk=chunk), dims=(64, 64, 16), fanout=(fanout, fanout), pool_slots=V, hub_count=9)
    g, model = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
    x0 = tg.features(w.seed, 0, 0, V, 64)
    want = run_oracle(w, g, model, x0)["outs"][1]
    x = torch.from_numpy(x0).cuda()
    ctx = tb.Context(V, g.E, g.row_ptr, g.col_idx, g.in_degree, w.mode, w.dims, model.W_neigh, model.W_self, model.bias, model.act, chunk, V, 9, w.fanout, w.seed, 0, V)
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    between, out = torch.empty(V, 64, device="cuda"), torch.empty(V, 16, device="cuda")
    bufs = [torch.empty(chunk, 64, device="cuda") for _ in range(2)]
    torch.cuda.synchronize()
    for _ in range(3):
        for l, (src, dst) in enumerate(((x, between), (between, out))):
            ctx.layer_begin(l, streams[0])
            ctx.layer_set_dense_output(dst, dst.shape[1])
            for i, b in enumerate(range(0, V, chunk)):
                k = i // 5 % 2   # five pushes on one stream, then five on the other
                with torch.cuda.stream(streams[k]):
                    n = min(chunk, V - b)
                    bufs[k][:n].copy_(src[b:b + n])
                    ctx.push_chunk(b, b + n, bufs[k][:n], streams[k])
                    bufs[k].fill_(float("nan"))
            assert ctx.layer_end()["completed"] == V
        assert row_error(out.cpu().numpy(), want)[0] <= 1e-4


@pytest.mark.parametrize("dims,fanout", [((64, 64), 0), ((24, 72), 0), ((64, 32), 4)])
def test_what_blocking_calls_find_after_the_last_push(dims, fanout):
    """The last push of a layer reports the control block by itself: statistics, drains, layer_end and another drain after it, in several orders."""
    import numpy as np
    import torch
    import paper_2607_17374_b200 as tb
    V, chunk = 5_000, 1_000
    w = replace(tg.scaled(tg.WORKLOADS["large"], V, chunk=chunk), dims=dims, fanout=(fanout,), pool_slots=V, hub_count=5)
    g, m = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
    x = torch.from_numpy(tg.features(w.seed, 0, 0, V, dims[0])).cuda()
    ctx = tb.Context(V, g.E, g.row_ptr, g.col_idx, g.in_degree, w.mode, w.dims, m.W_neigh, m.W_self, m.bias, m.act, chunk, V, 5, w.fanout, w.seed, 0, V + 1_024)
    out = torch.empty(V, dims[1], device="cuda")
    ids, rows = torch.empty(V, dtype=torch.int64, device="cuda"), torch.empty(V, dims[1], device="cuda")
    seen = []
    for order in range(5):
        ctx.layer_begin(0)
        if order == 4:
            ctx.layer_set_dense_output(out, dims[1])
        for b in range(0, V, chunk):
            ctx.push_chunk(b, b + chunk, x[b:b + chunk])
            if order == 0 and b == 2 * chunk:
                first = ctx.drain_dense(out, dims[1], V)
        if order == 0:
            assert ctx.get_stats()["completed"] == V
            assert ctx.drain_dense(out, dims[1], V) + first == V and ctx.drain_dense(out, dims[1], V) == 0
        elif order == 1:
            assert ctx.drain_completed(ids, rows, V) == V and ctx.drain_completed(ids, rows, V) == 0
        elif order == 2:
            assert ctx.get_stats()["completed"] == V and ctx.layer_end()["completed"] == V
            assert ctx.drain_dense(out, dims[1], V) == V and ctx.drain_completed(ids, rows, V) == 0
        elif order == 3:
            with pytest.raises(tb.TaurusError):
                ctx.drain_dense(out, dims[1], V - 1)
            assert ctx.drain_dense(out, dims[1], V, ids) == V and sorted(ids.tolist()) == list(range(V))
        st = ctx.layer_end()
        assert st["completed"] == V and st["chunks"] == V // chunk and st["free_slots"] == V
        seen.append({k: v for k, v in st.items()})
    assert all(s == seen[0] for s in seen)


@pytest.mark.parametrize("pool", ["all", "bounded"])
def test_rows_that_another_stream_writes_late(pool):
    """The rows of every push come from another stream, behind a kernel that takes its time, and the push waits for an event of it: directly behind
    that wait, with the kernels of the push before in front of it."""
    import torch
    import paper_2607_17374_b200 as tb
    V, chunk = 6_000, 500 if pool == "all" else 100
    w = replace(tg.scaled(tg.WORKLOADS["large"], V, chunk=chunk), dims=(64, 64), fanout=(0,), pool_slots=V if pool == "all" else 4_500, hub_count=9)
    g, model = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
    x0 = tg.features(w.seed, 0, 0, V, 64)
    want = run_oracle(w, g, model, x0)["outs"][0]
    x = torch.from_numpy(x0).cuda()
    ctx = tb.Context(V, g.E, g.row_ptr, g.col_idx, g.in_degree, w.mode, w.dims, model.W_neigh, model.W_self, model.bias, model.act, chunk, w.pool_slots, 9, w.fanout, w.seed,
                     0 if pool == "all" else V, V + 1_024)
    ours, other = torch.cuda.Stream(), torch.cuda.Stream()
    out = torch.empty(V, 64, device="cuda")
    rows = torch.empty(V, 64, device="cuda")
    for _ in range(3):
        rows.fill_(float("nan"))
        torch.cuda.synchronize()
        ctx.layer_begin(0, ours)
        ctx.layer_set_dense_output(out, 64)
        for b in range(0, V, chunk):
            with torch.cuda.stream(other):
                torch.cuda._sleep(200_000)
                rows[b:b + chunk].copy_(x[b:b + chunk])
                ready = torch.cuda.Event()
                ready.record(other)
            ours.wait_event(ready)
            ctx.push_chunk(b, b + chunk, rows[b:b + chunk], ours)
        assert ctx.layer_end()["completed"] == V
        assert row_error(out.cpu().numpy(), want)[0] <= 1e-4
