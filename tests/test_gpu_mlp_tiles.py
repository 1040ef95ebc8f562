"""The fused rank-predictor pass takes tiles of 64 samples, one CTA per SM: row
counts around a tile, around one tile per CTA, and a single row, against the
NumPy network.  Bounds: FP32 chains of at most 64 terms through three hidden
layers stay below 3 * 64 * 2^-24 ~ 1.2e-5 of the values' scale; the gradient's
sums over the samples are exact to far below FP32, so the same chains and the
backward ones (twice as many) bound it."""

import numpy as np
import pytest

from oracle import mlp as ref
from paper_1905_10602_gb300 import build as _build

pytestmark = pytest.mark.gpu

_build.build()
from paper_1905_10602_gb300 import ifmm  # noqa: E402


@pytest.mark.parametrize("n", [1, 63, 64, 65, 152 * 64 - 1, 152 * 64 + 1, 2 * 152 * 64 + 33])
def test_forward_and_gradient_at_tile_edges(n):
    rng = np.random.default_rng(n)
    w = (rng.standard_normal(ref.nweights()) * 0.15).astype(np.float32)
    X = rng.uniform(-1, 1, (n, 9)).astype(np.float32)
    t = rng.uniform(0, 1, n).astype(np.float32)
    y = ifmm.ifmm_mlp_forward(w, X)
    yr, _ = ref.forward(w, X)
    tol = 3 * 64 * 2.0 ** -24
    assert np.abs(y - yr).max() <= tol * max(1.0, np.abs(yr).max())
    loss, g = ifmm.ifmm_mlp_grad(w, X, t)
    lr, gr = ref.loss_and_grad(w, X, t)
    assert abs(loss - lr) <= 2 * tol * max(1.0, lr)
    assert np.linalg.norm(g - gr) <= 10 * tol * np.linalg.norm(gr)
    loss2, g2 = ifmm.ifmm_mlp_grad(w, X, t)
    assert loss2 == loss and np.array_equal(g, g2)
