"""The projection in fp32 mode (operands split into two TF32 values) at the edges of its tiles and stages: one row to several tiles per
CTA, K with short last stages, one to eight blocks of output columns, columns that fill no 32, bias and per-row factors; elements of
very different magnitudes in a row of X, in a column of W.  Against the product in 64 bits, element by element of the magnitude sum:
a value cut after 11 + 11 bits is off by at most 2^-20, on either side, the dropped lo.lo by 2^-20, and K additions by 2^-24 each:
2^-18 + K 2^-24 covers them, whatever the magnitudes."""
from dataclasses import replace

import numpy as np
import pytest
import torch

import paper_2607_17374_b200 as tb
import taurus_gen as tg
from test_gpu_parity import _full_check

pytestmark = pytest.mark.gpu


def _project(x, W, chunk=None):
    """out = x W through a GIN layer of an edgeless graph whose own row has weight 1 (gin_eps = 0)."""
    V, K = x.shape
    N = W.shape[1]
    dev = torch.device("cuda:0")
    row_ptr, col, din = torch.zeros(V + 1, dtype=torch.int64, device=dev), torch.zeros(0, dtype=torch.int32, device=dev), torch.zeros(V, dtype=torch.int32, device=dev)
    ctx = tb.Context(V, 0, row_ptr, col, din, tb.GIN_SUM, [K, N], [torch.from_numpy(W)], [torch.from_numpy(W)], [torch.zeros(N)], [0], chunk or V, V, 0, None, 1,
                     0, V, tb.GEMM_FP32, 0, 0, 0.0)
    out = torch.empty(V, N, device=dev)
    st = torch.cuda.current_stream()
    ctx.layer_begin(0, st)
    ctx.layer_set_dense_output(out, N)
    xd = torch.from_numpy(x).to(dev)
    for b in range(0, V, chunk or V):
        ctx.push_chunk(b, min(b + (chunk or V), V), xd[b:b + (chunk or V)], st)
    ctx.layer_end()
    return out.cpu().numpy()


def _check(x, W, got):
    x64, W64 = x.astype(np.float64), W.astype(np.float64)
    ref, mag = x64 @ W64, np.abs(x64) @ np.abs(W64)
    assert (np.abs(got - ref) <= (2.0 ** -18 + x.shape[1] * 2.0 ** -24) * mag).all(), float((np.abs(got - ref) / mag).max())


@pytest.mark.parametrize("V", [1, 127, 700, 40_003])
@pytest.mark.parametrize("K,N", [(4, 4), (16, 96), (64, 64), (68, 48), (100, 64), (128, 128), (192, 100), (256, 64), (256, 256), (320, 132), (512, 260), (1024, 512)])
def test_shapes(V, K, N):
    if V > 1_000 and K * N > 70_000:
        V = 20_003
    rng = np.random.default_rng(K * 1000 + N + V)
    x, W = rng.standard_normal((V, K)).astype(np.float32), (rng.standard_normal((K, N)) / K ** 0.5).astype(np.float32)
    _check(x, W, _project(x, W))


def _rows(kind, V, K, rng):
    x = rng.standard_normal((V, K))
    if kind == "grow":        # every column larger than the one before it
        x *= 10.0 ** np.linspace(-8, 9, K)
    elif kind == "steps":     # ... at every K step, with empty ones in front
        x *= 10.0 ** (4 * (np.arange(K) // 32 % 4)) * (np.arange(K) >= 32)
    elif kind == "late":      # ... in some rows only, in the last column
        x[:, -1] *= np.where(rng.random(V) < 0.1, 1e6, 1.0)
    elif kind == "rows":
        x *= 10.0 ** rng.uniform(-30, 30, V)[:, None]
    elif kind == "zeros":
        x *= rng.random((V, K)) < 0.01
    return x.astype(np.float32)


@pytest.mark.parametrize("K,N", [(36, 20), (96, 128), (256, 256), (300, 340)])
@pytest.mark.parametrize("kind", ["grow", "steps", "late", "rows", "zeros"])
def test_rows_of_many_magnitudes(kind, K, N):
    V = 40_003
    rng = np.random.default_rng(K + N)
    x, W = _rows(kind, V, K, rng), (rng.standard_normal((K, N)) / K ** 0.5).astype(np.float32)
    _check(x, W, _project(x, W))


@pytest.mark.parametrize("weights", ["zero", "balancing"])
@pytest.mark.parametrize("at", [0, 31, 32, -1])
@pytest.mark.parametrize("size", [1e4, 1e6, 1e9])
def test_one_raw_column(size, at, weights):
    """An id, a count or a time stamp among N(0, 1) features, with no weight or with one that brings it back to their size."""
    V, K, N = 5_003, 100, 72
    rng = np.random.default_rng(int(size) + at)
    x, W = rng.standard_normal((V, K)), rng.standard_normal((K, N)) / K ** 0.5
    x[:, at] *= size
    W[at] *= 0 if weights == "zero" else 1 / size
    x, W = x.astype(np.float32), W.astype(np.float32)
    _check(x, W, _project(x, W))


@pytest.mark.parametrize("feature", ["zero", "balancing"])
@pytest.mark.parametrize("at", [0, 31, 32, -1])
@pytest.mark.parametrize("size", [1e6, 1e9])
def test_one_large_weight_a_column(size, at, feature):
    V, K, N = 5_003, 100, 72
    rng = np.random.default_rng(int(size) + at)
    x, W = rng.standard_normal((V, K)), rng.standard_normal((K, N)) / K ** 0.5
    W[at] *= size
    x[:, at] *= 0 if feature == "zero" else 1 / size
    x, W = x.astype(np.float32), W.astype(np.float32)
    _check(x, W, _project(x, W))


def test_worst_element_of_a_hub():
    """A sum over thousands of projected rows, where an error that the rows have in common adds up, element by element.  On top of a
    product's own error: the additions of a piece of an in-list (128 entries) and of its pieces, one after the other at most."""
    V, K, N, hub = 30_000, 64, 32, 20_003
    rng = np.random.default_rng(5)
    src = np.concatenate([rng.integers(0, V, hub), rng.integers(0, V, 700), rng.integers(0, V, 3 * V)])
    dst = np.concatenate([np.full(hub, 17), np.full(700, V - 1), rng.integers(0, V, 3 * V)])
    order = np.argsort(src, kind="stable")
    src, dst = src[order], dst[order]
    row_ptr = np.zeros(V + 1, np.int64)
    row_ptr[1:] = np.cumsum(np.bincount(src, minlength=V))
    x, W = (1 + rng.standard_normal((V, K))).astype(np.float32), (rng.standard_normal((K, N)) / K ** 0.5).astype(np.float32)
    dev = torch.device("cuda:0")
    ctx = tb.Context(V, len(src), torch.from_numpy(row_ptr).to(dev), torch.from_numpy(dst.astype(np.int32)).to(dev),
                     torch.from_numpy(np.bincount(dst, minlength=V).astype(np.int32)).to(dev), tb.GIN_SUM, [K, N], [torch.from_numpy(W)], [torch.from_numpy(W)],
                     [torch.zeros(N)], [0], 8192, V, 0, None, 1, 0, V, tb.GEMM_FP32, 0, 0, 0.0)
    out = torch.empty(V, N, device=dev)
    ctx.layer_begin(0)
    ctx.layer_set_dense_output(out, N)
    xd = torch.from_numpy(x).to(dev)
    for b in range(0, V, 8192):
        ctx.push_chunk(b, min(b + 8192, V), xd[b:b + 8192])
    ctx.layer_end()

    def layer(x, W):
        h = x @ W
        o = h.copy()
        np.add.at(o, dst, h[src])
        return o
    ref, mag = layer(x.astype(np.float64), W.astype(np.float64)), layer(np.abs(x).astype(np.float64), np.abs(W).astype(np.float64))
    err = np.abs(out.cpu().numpy() - ref)
    assert (err <= (2.0 ** -18 + (K + 128 + hub // 128 + 16) * 2.0 ** -24) * mag).all(), float((err / mag).max())


@pytest.mark.parametrize("spread", [0, 2, 15])
def test_columns_of_many_magnitudes(spread):
    V, K, N = 20_003, 100, 132
    rng = np.random.default_rng(spread)
    x = _rows("rows", V, K, rng) if spread < 15 else rng.standard_normal((V, K)).astype(np.float32)
    W = (rng.standard_normal((K, N)) * 10.0 ** rng.uniform(-spread, spread / 4, N)).astype(np.float32)
    W[:, 5] = 0
    _check(x, W, _project(x, W))


def test_rows_that_are_not_finite():
    V, K, N = 5_000, 96, 64
    rng = np.random.default_rng(1)
    x, W = rng.standard_normal((V, K)).astype(np.float32), rng.standard_normal((K, N)).astype(np.float32)
    clean = _project(x, W)
    x[7, 3], x[800, 90], x[801, 0], x[4_999, 40] = np.inf, -np.inf, np.nan, np.nan
    got = _project(x, W)
    bad = np.zeros(V, bool)
    bad[[7, 800, 801, 4_999]] = True
    assert np.isnan(got[bad]).all() and (got[~bad] == clean[~bad]).all()


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("K,N", [(132, 130), (228, 260), (232, 300), (516, 258), (260, 340), (800, 1024)])   # 2 (264), 3, 3, 3, 3, 8 blocks of columns
def test_blocks_of_columns(K, N, bf16):
    """SAGE rows [P | T] of several blocks, enough rows that a CTA takes several tiles; biases and in-degrees that show which columns
    they went to.  bf16 operands: 2^-9 on either side of a product."""
    V = 20_003
    dev, gen = torch.device("cuda:0"), torch.Generator()
    gen.manual_seed(K + N)
    din = torch.randint(0, 5, (V,), generator=gen)
    dst = torch.repeat_interleave(torch.arange(V), din)
    src = torch.randint(0, V, (dst.numel(),), generator=gen)
    order = torch.argsort(src, stable=True)
    row_ptr = torch.zeros(V + 1, dtype=torch.int64)
    row_ptr[1:] = torch.cumsum(torch.bincount(src, minlength=V), 0)
    x = torch.randn(V, K, generator=gen)
    Wn, Ws = (torch.randn(K, N, generator=gen) / K ** 0.5 for _ in range(2))
    bias = torch.randn(N, generator=gen)
    ctx = tb.Context(V, dst.numel(), row_ptr.to(dev), dst[order].to(torch.int32).to(dev), din.to(torch.int32).to(dev), tb.SAGE_MEAN, [K, N], [Wn], [Ws], [bias],
                     [0], V, V, 0, None, 1, 0, V, tb.GEMM_BF16 if bf16 else tb.GEMM_FP32)
    out = torch.empty(V, N, device=dev)
    ctx.layer_begin(0)
    ctx.layer_set_dense_output(out, N)
    ctx.push_chunk(0, V, x.to(dev))
    ctx.layer_end()

    def layer(x, Wn, Ws, b):
        mean = torch.zeros(V, K, dtype=torch.float64, device=dev).index_add_(0, dst.to(dev), x[src.to(dev)]) / din.to(dev).clamp(min=1)[:, None]
        return mean @ Wn + x @ Ws + b
    t = [a.to(dev).double() for a in (x, Wn, Ws, bias)]
    ref, mag = layer(*t), layer(*(a.abs() for a in t))
    rel = (2.0 ** -8 + 2.0 ** -17 if bf16 else 2.0 ** -18) + (K + 16) * 2.0 ** -24   # K additions of a product, a few of its rows
    assert bool(((out.double() - ref).abs() <= rel * mag).all()), float(((out.double() - ref).abs() / mag).max())


def test_attention_scalars_in_the_second_block():
    w = tg.scaled(tg.WORKLOADS["mid"], 20_000, chunk=20_000)
    w = replace(w, E=6 * 20_000, dims=(200, 256), fanout=(0,), pool_slots=20_000, hub_count=0, mode=tg.GAT, gat_heads=4)
    _full_check(w, tg.make_graph(w), dense_output=True)
