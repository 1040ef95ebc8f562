"""Tall blocks of 17 to 64 columns around the heights where the chunk size changes
(24 chunks of 256 rows at 64 columns, then 512, 1,024 and 1,536 rows a chunk), held
to ||A^T A - R^T R|| <= (m + n) u ||A||_F^2 (any Householder QR; each reduction is one
more orthogonal step over the same rows), with no launch of the global-memory
kernels."""

import numpy as np
import pytest

from paper_1905_10602_gb300 import build as _build

pytestmark = pytest.mark.gpu

_build.build()
from paper_1905_10602_gb300 import ifmm  # noqa: E402

U = {"fp32": 2.0 ** -24, "fp64": 2.0 ** -53}


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("m,n", [(6144, 64), (6200, 64), (7000, 64), (8000, 60), (12096, 64), (12289, 64), (24577, 64)])
def test_tall(prec, m, n):
    A = np.random.default_rng(m + n).standard_normal((m, n))
    if prec == "fp32":
        A = A.astype(np.float32).astype(np.float64)
    nA2 = np.linalg.norm(A) ** 2
    ifmm.ifmm_profile(False)
    R = ifmm.ifmm_qr_check(A, prec)
    Rp, jp, k = ifmm.ifmm_qr_check(A, prec, pivoted=True)
    assert ifmm.ifmm_profile_query().get("qr_global_" + prec, (0, 0.0))[0] == 0
    assert np.linalg.norm(A.T @ A - R.T @ R) <= (m + n) * U[prec] * nA2
    assert k == n and sorted(jp.tolist()) == list(range(n))
    Ap = A[:, jp]
    assert np.linalg.norm(Ap.T @ Ap - Rp.T @ Rp) <= (m + n) * U[prec] * nA2
