"""GMRES' vector operations work on chunks of at least 512 elements, one CTA each:
system sizes around one and two chunks, a single unknown, and restarts (every
cycle's first vector comes from the residual kernel), without a preconditioner,
against a dense solve.

Bound: GMRES stops at a true relative residual <= tol, so the error is at most
cond(A) tol (||x|| >= ||b|| / ||A||), plus the dense solve's own n u cond(A)."""

import numpy as np
import pytest

from paper_1905_10602_gb300 import build as _build
from paper_1905_10602_gb300.workloads import bumpy_sphere

pytestmark = pytest.mark.gpu

_build.build()
from paper_1905_10602_gb300 import ifmm  # noqa: E402


@pytest.mark.parametrize("n", [1, 2, 511, 512, 513, 1025])
@pytest.mark.parametrize("restart", [2, 30])
def test_gmres_chunk_edges(n, restart):
    pts = bumpy_sphere(n, 2)
    t = ifmm.ifmm_build_tree(pts, 2)
    b = np.random.default_rng(n).standard_normal(n)
    tol = 1e-11
    x, its, rel = ifmm.bem_gmres(t, b, restart=restart, tol=tol, maxit=400)
    assert rel <= tol and its >= 1
    r = np.sqrt(((pts[:, None] - pts[None]) ** 2).sum(-1))
    np.fill_diagonal(r, 1.0)
    A = 1.0 / n / r
    np.fill_diagonal(A, 0.5 + 1.0 / np.sqrt(n))
    xs = np.linalg.solve(A, b)
    bound = np.linalg.cond(A) * (tol + n * 2.0 ** -53)
    assert np.linalg.norm(x - xs) <= bound * np.linalg.norm(xs)
    x2, its2, rel2 = ifmm.bem_gmres(t, b, restart=restart, tol=tol, maxit=400)
    assert its2 == its and rel2 == rel and np.array_equal(x, x2)
