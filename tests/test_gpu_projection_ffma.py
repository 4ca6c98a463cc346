"""The FFMA projection (rows whose pitch is not a whole number of 16 bytes) at the edges of its 32 x 64 blocks and 32-column panels,
against the product in 64 bits: K roundings of 2^-24 of the magnitude sum."""
import numpy as np
import pytest

from test_gpu_projection_shapes import _project

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("V", [1, 31, 33, 700, 10_007])
@pytest.mark.parametrize("K,N", [(1, 1), (5, 4), (31, 36), (33, 40), (47, 36), (63, 64), (65, 68), (97, 100), (130, 48), (130, 132), (257, 64), (515, 260)])
def test_blocks_and_panels(V, K, N):
    rng = np.random.default_rng(K * 1000 + N + V)
    x, W = rng.standard_normal((V, K)).astype(np.float32), (rng.standard_normal((K, N)) / K ** 0.5).astype(np.float32)
    x64, W64 = x.astype(np.float64), W.astype(np.float64)
    got = _project(x, W, chunk=max(1, V // 2))
    assert (np.abs(got - x64 @ W64) <= (K + 2) * 2.0 ** -24 * (np.abs(x64) @ np.abs(W64))).all()
