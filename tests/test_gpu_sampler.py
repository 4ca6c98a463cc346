"""The sampler at the limits of its kernels (fanouts of 16, 32 and 64, in-lists of one or two words of the entry mask and beyond), and the mask by CSR
edge, which pools that hold every vertex build only when somebody asks: inspection, the first pass over a layer, pushes off the chunk grid."""
from dataclasses import replace

import numpy as np
import pytest

import oracle
import taurus_gen as tg
from gpu_harness import row_error, run_oracle
from helpers import csr_from_edges

pytestmark = pytest.mark.gpu


def _lists(V, lengths, rng):
    """Vertex d has lengths[d] in-edges, multi-edges among them; every vertex sends at least one."""
    edges = [(int(u), d) for d, n in enumerate(lengths) for u in rng.integers(0, V, n)] + [(u, len(lengths) + u % (V - len(lengths))) for u in range(V)]
    row_ptr, col = csr_from_edges(V, edges)
    return tg.Graph(V, len(edges), row_ptr, col, np.bincount(col, minlength=V).astype(np.int32))


@pytest.mark.parametrize("push_form", [False, True])
@pytest.mark.parametrize("fanout", [1, 2, 15, 16, 17, 31, 32, 33, 63, 64])
def test_kept_edges(fanout, push_form):
    import paper_2607_17374_b200 as tb
    V = 700
    g = _lists(V, [0, 1, 2, fanout - 1, fanout, fanout + 1, 31, 32, 33, 40, 63, 64, 65, 66, 95, 97, 200, 1_000, 5_000, 0, 64, 64], np.random.default_rng(fanout))
    w = replace(tg.WORKLOADS["tiny"], V=V, E=g.E, dims=(8, 8), fanout=(fanout,), chunk=64, pool_slots=V, hub_count=0)
    m = tg.make_model(w)
    ctx = tb.Context(V, g.E, g.row_ptr, g.col_idx, g.in_degree, w.mode, w.dims, m.W_neigh, m.W_self, m.bias, m.act, 64, V, 0, w.fanout, w.seed, 0, V, 0, 16 if push_form else 0)
    ms = oracle.message_sets(oracle.build_in_lists(V, g.row_ptr, g.col_idx), fanout, w.seed, 0)
    want = np.packbits(ms.prop, bitorder="little")
    for _ in range(2):
        ctx.layer_begin(0)
        assert np.array_equal(ctx.get_sample_digest(), oracle.sample_digest(ms))
        assert (ctx.get_edge_mask().view(np.uint8)[:want.size] == want).all()
    ctx.destroy()


@pytest.mark.parametrize("mode", [tg.SAGE_MEAN, tg.GIN_SUM])
def test_pushes_off_the_grid_that_nobody_inspected(mode):
    import torch
    import paper_2607_17374_b200 as tb
    V = 20_000
    w = replace(tg.scaled(tg.WORKLOADS["sampled"], V, chunk=1_024), dims=(36, 64, 20), fanout=(6, 0), pool_slots=V, hub_count=9, mode=mode)
    g, m = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
    x0 = tg.features(w.seed, 0, 0, V, 36)
    orc = run_oracle(w, g, m, x0)
    ctx = tb.Context(V, g.E, g.row_ptr, g.col_idx, g.in_degree, w.mode, w.dims, m.W_neigh, m.W_self, m.bias, m.act, 1_024, V, 9, w.fanout, w.seed, 0, V, 0, 0, 0, w.gin_eps)
    x, between, out = torch.from_numpy(x0).cuda(), torch.empty(V, 64, device="cuda"), torch.empty(V, 20, device="cuda")
    for steps in ((1_024, 777), (777, 1_024), (1_024, 1_024), (500, 777)):   # by layer; completion ranks are known from the second pass on
        for l, (src, dst) in enumerate(((x, between), (between, out))):
            ctx.layer_begin(l)
            ctx.layer_set_dense_output(dst, dst.shape[1])
            for b in range(0, V, steps[l]):
                ctx.push_chunk(b, min(b + steps[l], V), src[b:b + steps[l]])
            st = ctx.layer_end()
            assert st["completed"] == V and st["total_messages"] == int(np.asarray(orc["msets"][l].m).sum())
        assert row_error(between.cpu().numpy(), orc["outs"][0])[0] <= 1e-4 and row_error(out.cpu().numpy(), orc["outs"][1])[0] <= 1e-4
