"""A level's set-up and update kernels (leaf interpolation, translation tables, Gram
sums and their Cholesky factors, weight stacks, Schur updates) at the sizes where
their chunks end: Chebyshev orders 2 to 5 (8, 27, 64 and 125 coefficients: odd and
even orders of the Gram matrices, row blocks of each width class of the Schur
updates) and leaves of one point up to a few chunks of 64.  The factor approximates the inverse of the FMM
representation A~, whose product the library has as well, so ifmm_solve(A~ x) must
return x to the truncation eps times the few hundred that the elimination can
amplify (1000 allowed, as in the tests of the block widths)."""

import numpy as np
import pytest

from paper_1905_10602_gb300 import build as _build
from paper_1905_10602_gb300.workloads import bumpy_sphere, torus

pytestmark = pytest.mark.gpu

_build.build()
from paper_1905_10602_gb300 import ifmm  # noqa: E402


@pytest.mark.parametrize("n,depth,order", [(150, 3, 2), (900, 3, 3), (4001, 3, 3), (3001, 3, 4), (2500, 3, 5),
                                           (5200, 2, 4)])
@pytest.mark.parametrize("precision,eps", [("fp64", 1e-9), ("fp32", 1e-5)])
def test_solve_inverts_the_fmm_matrix(n, depth, order, precision, eps):
    pts = torus(n, 9) if n % 2 else bumpy_sphere(n, 9)
    t = ifmm.ifmm_build_tree(pts, depth)
    ifmm.ifmm_color(t, 3)
    f = ifmm.ifmm_factor(t, order, eps, precision=precision)
    x = np.random.default_rng(n).standard_normal(n)
    y = ifmm.bem_matvec(t, x, kernel=ifmm.default_kernel(n, "fmm", order))
    v = ifmm.ifmm_solve(f, y)
    assert np.linalg.norm(v - x) <= 1000 * eps * np.linalg.norm(x)
    assert np.array_equal(v, ifmm.ifmm_solve(ifmm.ifmm_factor(t, order, eps, precision=precision), y))
