"""Projection by pairs of CTAs (chunks of more than two waves of 128-row tiles) against the FFMA kernel: last tiles that fill one
CTA, part of one, or none of the second; column blocks of 32 up to 256 + 32 and 2 x 256 columns; input widths that end inside a
K step.  Both kernels see the same sums, so the rows may differ by the products' rounding only: 2^-21 per term with the split
operands, 2^-8 with bf16 ones, times the square root of the few hundred terms' worth of cancellation."""
from dataclasses import replace

import numpy as np
import pytest

import taurus_gen as tg
from gpu_harness import run_library

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V,K,N", [(38_017, 36, 16), (38_144, 64, 48), (38_273, 100, 144), (38_400, 256, 256), (41_001, 32, 128)])
@pytest.mark.parametrize("mode,gemm", [(tg.SAGE_MEAN, tg.GEMM_FP32), (tg.GCN_SYM, tg.GEMM_FP32), (tg.SAGE_MEAN, tg.GEMM_BF16)])
def test_pairs_against_the_ffma_kernel(V, K, N, mode, gemm):
    w = tg.scaled(tg.WORKLOADS["tiny"], V, chunk=V)
    w = replace(w, dims=(K, N), fanout=(0,), pool_slots=V, hub_count=0, mode=mode, gemm_mode=gemm)
    g, model = tg.make_graph(w), tg.make_model(w, bias_scale=0.3)
    x0 = tg.features(w.seed, 0, 0, V, K)
    outs = []
    for flags, gm in ((8, gemm), (8 | 2, tg.GEMM_FP32)):   # project first; FFMA
        r = run_library(w, g, model, x0, flags=flags, gemm_mode=gm, dense_output=True)
        outs.append(r["outs"][0].astype(np.float64))
        r["ctx"].destroy()
    err = np.linalg.norm(outs[0] - outs[1]) / np.linalg.norm(outs[1])
    assert err <= (2e-6 if gemm == tg.GEMM_FP32 else 8e-3), err
