"""Calls of one context on several streams: what a caller puts on the stream of a layer that has ended is over before a layer begun on another stream
reads or writes anything."""
from dataclasses import replace

import pytest

import taurus_gen as tg
from gpu_harness import row_error, run_oracle

pytestmark = pytest.mark.gpu


def _context(w, g, flags=0):
    import paper_2607_17374_b200 as tb
    m = tg.make_model(w, bias_scale=0.3)
    return m, tb.Context(g.V, g.E, g.row_ptr, g.col_idx, g.in_degree, w.mode, w.dims, m.W_neigh, m.W_self, m.bias, m.act, w.chunk, w.pool_slots, w.hub_count, w.fanout,
                         w.seed, 0, 2 * g.V, 0, flags, 0, w.gin_eps)


@pytest.mark.parametrize("dims", [(64, 64, 32), (20, 72, 40)])
def test_work_between_two_layers_on_the_stream_of_the_first(dims):
    """The caller writes the second layer's input on the first one's stream, behind a kernel that takes its time."""
    import torch
    V, chunk = 5_000, 1_024
    w = replace(tg.scaled(tg.WORKLOADS["large"], V, chunk=chunk), dims=dims, fanout=(0, 0), pool_slots=V, hub_count=5)
    g = tg.make_graph(w)
    m, ctx = _context(w, g)
    x0 = tg.features(w.seed, 0, 0, V, dims[0])
    want = run_oracle(w, g, m, x0)["outs"][1]
    x = torch.from_numpy(x0).cuda()
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    raw, between, out = (torch.empty(V, d, device="cuda") for d in (dims[1], dims[1], dims[2]))
    for _ in range(3):
        between.fill_(float("nan"))
        torch.cuda.synchronize()
        for l, (src, dst, st) in enumerate(((x, raw, first), (between, out, second))):
            ctx.layer_begin(l, st)
            ctx.layer_set_dense_output(dst, dst.shape[1])
            for b in range(0, V, chunk):
                ctx.push_chunk(b, min(b + chunk, V), src[b:b + chunk], st)
            assert ctx.layer_end()["completed"] == V
            if l == 0:
                with torch.cuda.stream(first):
                    torch.cuda._sleep(20_000_000)   # some 10 ms
                    between.copy_(raw)
        assert row_error(out.cpu().numpy(), want)[0] <= 1e-4
