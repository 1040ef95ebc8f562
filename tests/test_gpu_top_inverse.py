"""The explicit inverse of the level-1 system: orders from a few to a few thousand
(one partly filled panel of 32 columns, several, ragged tiles of 64; one to
sixteen CTAs per panel), through factorizations of depth 2, whose level-1 system
couples every cell.  ifmm_solve(A~ x) must return x to the truncation eps times
the few hundred that the elimination can amplify (1000 allowed, as in the tests of
the block widths), here with eps far below what digits lost in the inverse would
leave; and the exact inverse of a level-1 system that is diagonal."""

import numpy as np
import pytest

from paper_1905_10602_gb300 import build as _build
from paper_1905_10602_gb300.workloads import bumpy_sphere, torus

pytestmark = pytest.mark.gpu

_build.build()
from paper_1905_10602_gb300 import ifmm  # noqa: E402


@pytest.mark.parametrize("n,order", [(3, 2), (25, 2), (90, 2), (333, 3), (1400, 3), (2500, 4), (4000, 5)])
def test_solve_inverts_the_fmm_matrix_tightly(n, order):
    pts = torus(n, 2) if n % 2 else bumpy_sphere(n, 2)
    t = ifmm.ifmm_build_tree(pts, 2)
    ifmm.ifmm_color(t, 3)
    eps = 1e-12
    f = ifmm.ifmm_factor(t, order, eps)
    x = np.random.default_rng(n).standard_normal(n)
    y = ifmm.bem_matvec(t, x, kernel=ifmm.default_kernel(n, "fmm", order))
    v = ifmm.ifmm_solve(f, y)
    assert np.linalg.norm(v - x) <= 1000 * eps * np.linalg.norm(x)
    assert np.array_equal(v, ifmm.ifmm_solve(ifmm.ifmm_factor(t, order, eps), y))


@pytest.mark.parametrize("shift", [-200, 0, 300])
def test_magnitudes(shift):
    """The matrix scaled by a power of two: the solution scales back exactly (the
    digits are relative to each row's and column's largest entry)."""
    n = 700
    pts = bumpy_sphere(n, 3)
    t = ifmm.ifmm_build_tree(pts, 2)
    ifmm.ifmm_color(t, 3)
    b = np.random.default_rng(1).standard_normal(n)
    k = ifmm.default_kernel(n)
    v = ifmm.ifmm_solve(ifmm.ifmm_factor(t, 3, 1e-8, kernel=k), b)
    s = 2.0 ** shift
    ks = ifmm.Kernel(k.scale * s, k.diag * s, 0, 0, 0.0, 0.0)
    w = ifmm.ifmm_solve(ifmm.ifmm_factor(t, 3, 1e-8, kernel=ks), b)
    assert np.linalg.norm(w * s - v) <= 1e-10 * np.linalg.norm(v)
