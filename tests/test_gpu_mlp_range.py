"""The rank predictor's gradient where products of its factors leave FP32's range:
its sums over the samples are those of FP64, whatever the products' size.

Overflow: products of about 1e39 whose sums may cancel; a sum above FP32's largest
is infinite, the others finite.  Underflow: 65,536 products of about 2^-152 each, below
FP32's smallest number, whose sum of about 2^-136 is one.  Bounds: the FP32 chains of at
most 64 terms in three layers forward and back (6 * 64 * 2^-24 of the largest sum of
magnitudes), in the second case with dy rounded to a multiple of 2^-149 as well."""

import numpy as np
import pytest

from oracle import mlp as ref
from paper_1905_10602_gb300 import build as _build

pytestmark = pytest.mark.gpu

_build.build()
from paper_1905_10602_gb300 import ifmm  # noqa: E402

FMAX = float(np.finfo(np.float32).max)


def _weights(rng):
    return (rng.standard_normal(ref.nweights()) * 0.15).astype(np.float32)


def _magnitudes(w, X, t):
    """Sums of |a g| for the gradient's entries."""
    y, acts = ref.forward(w, X)
    g = np.abs((y - t) / len(y))[:, None]
    flat = []
    for l, (W, _) in reversed(list(enumerate(ref.unpack(w)))):
        flat.append(((np.abs(acts[l]).T @ g).ravel(), g.sum(axis=0)))
        if l > 0:
            g = (g @ np.abs(W).T) * (acts[l] > 0)
    return np.concatenate([np.concatenate(f) for f in reversed(flat)])


@pytest.mark.parametrize("n", [2, 64, 1000, 152 * 64 + 7])
def test_products_above_fp32(n):
    rng = np.random.default_rng(n)
    w = _weights(rng)
    X = (rng.uniform(-1, 1, (n, 9)) * 2e20).astype(np.float32)
    t = (rng.uniform(-1, 1, n) * 2e20 * np.sqrt(n)).astype(np.float32)
    loss, g = ifmm.ifmm_mlp_grad(w, X, t)
    _, gr = ref.loss_and_grad(w, X, t)
    tol = 6 * 64 * 2.0 ** -24 * _magnitudes(w, X, t)
    assert np.isinf(loss) and not np.isnan(g).any()
    inside = np.abs(gr) + tol < FMAX
    assert inside.any() and (np.abs(gr) - tol > FMAX).any()
    assert np.all(np.abs(g[inside] - gr[inside]) <= tol[inside])
    over = np.abs(gr) - tol > FMAX
    assert np.all(np.isinf(g[over]) & (np.sign(g[over]) == np.sign(gr[over])))


def test_products_below_fp32():
    n = 65536
    rng = np.random.default_rng(3)
    w = _weights(rng)
    w[4800:4800 + 4096] *= np.float32(2.0 ** -20)  # W3
    w[8896:8960] = 0                               # b3
    w[8960:9024] = np.abs(w[8960:9024]) * np.float32(2.0 ** -96)  # W4: one sign, so the sums do not cancel
    w[9024] = 0
    X = rng.uniform(-1, 1, (n, 9)).astype(np.float32)
    t = np.zeros(n, np.float32)
    _, g = ifmm.ifmm_mlp_grad(w, X, t)
    _, gr = ref.loss_and_grad(w, X, t)
    mag = _magnitudes(w, X, t)
    _, acts = ref.forward(w, X)
    slack = np.zeros_like(gr)
    slack[8960:9024] = np.abs(acts[3]).sum(axis=0) * 2.0 ** -150
    slack[9024] = n * 2.0 ** -150
    tol = 6 * 64 * 2.0 ** -24 * mag + slack + 2.0 ** -149
    assert np.all(np.abs(g - gr) <= tol)
    assert np.abs(g[8960:9024]).max() > 2.0 ** -140
