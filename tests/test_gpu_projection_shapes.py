"""The projection in fp32 mode (operands split into two TF32 values) at the edges of its tiles and stages: one row to several tiles per
CTA, K on both sides of the two stage widths and with short last stages, one to four blocks of output columns, columns that fill
no 32.  Against the product in 64 bits, element by element of the magnitude sum: a value cut after 11 + 11 bits is off by at
most 2^-20, on either side, the dropped lo.lo by 2^-20, and K additions by 2^-24 each: 2^-18 + K 2^-24 covers them."""
import numpy as np
import pytest
import torch

import paper_2607_17374_b200 as tb

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
