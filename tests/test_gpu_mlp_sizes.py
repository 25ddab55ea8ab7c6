"""The predictor's gradient at the edges of its tiles (32 samples below 19456 = 152 x 128, else
128) against the float64 oracle. The last sample's target is large, so its share of every
gradient entry is a large part of the sum: a sample left out or counted twice shows at any n.
Tolerance: FP32 sums of at most 140-term chains and some 1100 serial additions, 6e-8 each, of
terms that may cancel tenfold: 1e-3 of the largest entry; the loss's terms are positive: 1e-4."""
import numpy as np
import pytest

from oracle import mlp
from paper_2508_16376_gb300 import rtlfs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 9729, 19455, 19456, 19457, 38913, 78000])
def test_gradient_at_tile_edges(n):
    from paper_2508_16376_gb300 import build
    build.build()
    rng = np.random.default_rng(n)
    w = mlp.f64_to_bf16_bits(rng.normal(0, 0.2, mlp.N_PARAMS))
    X = rng.uniform(0, 1, (n, 5)).astype(np.float32)
    t = rng.normal(2, 1, n).astype(np.float32)
    t[-1] = 2.0 + np.float32(n)
    ctx = rtlfs.rtlfs_create(0)
    try:
        rtlfs.rtlfs_mlp_set_weights(ctx, w)
        loss, g = rtlfs.rtlfs_mlp_grad(ctx, X, t)
        y = rtlfs.rtlfs_mlp_forward(ctx, X)
    finally:
        rtlfs.rtlfs_destroy(ctx)
    eloss, eg = mlp.loss_grad(w, X.astype(np.float64), t.astype(np.float64))
    assert abs(loss - eloss) <= 1e-4 * abs(eloss)
    assert np.abs(g - eg).max() <= 1e-3 * np.abs(eg).max()
    ey, _ = mlp.forward(w, X.astype(np.float64))
    assert np.allclose(y, ey, rtol=1e-4, atol=1e-5)
