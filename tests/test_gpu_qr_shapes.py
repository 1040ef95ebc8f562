"""The register-resident QR at the edges of its shapes: rows per lane (multiples
of 32 rows in eight classes, 1,536 at most), columns per warp and per cluster, the
warp-per-problem kernel (16 columns, 64 or 128 rows), the finished 32-row blocks
that leave the registers on the way, wide blocks, tall ones reduced by chunks; and
a rank-deficient block, whose pivoted QR must stop.

Bounds as for any Householder QR: ||A^T A - R^T R|| <= (m + n) u ||A||_F^2."""

import numpy as np
import pytest

from paper_1905_10602_gb300 import build as _build

pytestmark = pytest.mark.gpu

_build.build()
from paper_1905_10602_gb300 import ifmm  # noqa: E402

U = {"fp32": 2.0 ** -24, "fp64": 2.0 ** -53}
SHAPES = [(1, 1), (16, 16), (64, 16), (65, 16), (128, 16), (129, 16), (128, 17), (129, 33), (256, 64), (257, 64),
          (384, 65), (385, 20), (640, 130), (641, 5), (1024, 66), (1536, 10), (1537, 10), (33, 200), (31, 100),
          (96, 260), (500, 200), (4000, 90)]


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("m,n", SHAPES)
def test_shapes(prec, m, n):
    A = np.random.default_rng(m * 7 + n).standard_normal((m, n)) * 1e-9
    if prec == "fp32":
        A = A.astype(np.float32).astype(np.float64)
    nA2 = np.linalg.norm(A) ** 2
    R = ifmm.ifmm_qr_check(A, prec)
    assert np.linalg.norm(A.T @ A - R.T @ R) <= (m + n) * U[prec] * nA2
    R, jp, k = ifmm.ifmm_qr_check(A, prec, pivoted=True)
    assert k == min(m, n) and sorted(jp.tolist()) == list(range(n))
    Ap = A[:, jp]
    assert np.linalg.norm(Ap.T @ Ap - R.T @ R) <= (m + n) * U[prec] * nA2
    d = np.abs(np.diag(R))
    assert np.all(d[1:] <= d[:-1] * (1 + 64 * U[prec]))


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("m,n,r", [(60, 12, 5), (200, 40, 33), (500, 100, 64), (300, 150, 1), (40, 9, 0)])
def test_low_rank(prec, m, n, r):
    """r independent integer columns, the others copies of them or zero: every
    product is exact, so the remaining norms fall to rounding after r steps."""
    g = np.random.default_rng(n)
    B = g.integers(-3, 4, (m, max(r, 1))).astype(float) * (1 if r else 0)
    A = B[:, np.arange(n) % max(r, 1)]
    R, jp, k = ifmm.ifmm_qr_check(A, prec, pivoted=True)
    assert k >= r and sorted(jp.tolist()) == list(range(n))
    Ap = A[:, jp]
    nA2 = np.linalg.norm(A) ** 2
    assert np.linalg.norm(Ap.T @ Ap - R[:k].T @ R[:k]) <= (m + n) * U[prec] * max(nA2, 1e-300)
    if r == 0:
        assert k == 0
