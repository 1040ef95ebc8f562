"""The Gauss-Jordan inverse at the edges of its size classes (rows per thread and
per warp, one to sixteen CTAs per matrix, two rows per thread above 512) and in
batches that change the CTAs per matrix, on matrices that need an interchange at
almost every step; a permutation matrix, whose inverse is exact; a singular step
inside a cluster.

Bound: the residual of Gauss-Jordan with partial pivoting is of order
n u ||A|| ||X||; 8 n u allowed (u = 2^-53)."""

import numpy as np
import pytest

from paper_1905_10602_gb300 import build as _build

pytestmark = pytest.mark.gpu

_build.build()
from paper_1905_10602_gb300 import ifmm  # noqa: E402

U = 2.0 ** -53


@pytest.mark.parametrize("orders", [[24, 25, 26], [127, 128, 129], [255, 256, 257], [511, 512, 513], [600],
                                    [25] * 115, [26] * 230, [70] * 78, [1] * 400, [30] * 500])
def test_class_edges(orders):
    rng = np.random.default_rng(len(orders) + orders[0])
    mats = [rng.standard_normal((n, n)) for n in orders]
    X, info = ifmm.ifmm_inv_check(mats)
    assert not info.any()
    for A, Xi in zip(mats, X):
        n = len(A)
        assert np.linalg.norm(A @ Xi - np.eye(n)) <= 8 * n * U * np.linalg.norm(A) * np.linalg.norm(Xi)


@pytest.mark.parametrize("n", [5, 40, 200, 530])
def test_permutation_and_magnitudes_are_exact(n):
    """A permutation times powers of two (also beyond what the approximate
    reciprocal takes): every operation is exact."""
    rng = np.random.default_rng(n)
    e = rng.integers(-1020, 1020, n)
    A = np.zeros((n, n))
    A[rng.permutation(n), np.arange(n)] = np.exp2(e.astype(float))
    (X,), info = ifmm.ifmm_inv_check([A])
    want = np.zeros((n, n))
    nz = A.T != 0
    want[nz] = 1.0 / A.T[nz]
    assert info[0] == 0 and np.array_equal(X, want)


@pytest.mark.parametrize("n,step", [(33, 0), (200, 199), (300, 128), (520, 17)])
def test_singular_step(n, step):
    A = np.random.default_rng(n).standard_normal((n, n))
    A[:, step] = 0.0
    _, info = ifmm.ifmm_inv_check([A])
    assert info[0] == step + 1
