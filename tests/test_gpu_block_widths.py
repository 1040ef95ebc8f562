"""The recompression's kernels by block width: the leaves' point counts select the
width classes of the Jacobi rotations (at most 16, 48, 128, 256 columns and
wider) and of the QR.  The factor approximates the inverse of the FMM
representation A~, whose product the library has as well, so ifmm_solve(A~ x)
must return x to the truncation: the solution error of the truncated elimination
scales with eps (the oracle's pinned property), with a factor of a few hundred
on these well-conditioned systems; 1000 eps allowed (FP32: 1000 * 2^-24 / eps
instead where rounding dominates)."""

import numpy as np
import pytest

from paper_1905_10602_gb300 import build as _build
from paper_1905_10602_gb300.workloads import bumpy_sphere, torus

pytestmark = pytest.mark.gpu

_build.build()
from paper_1905_10602_gb300 import ifmm  # noqa: E402


@pytest.mark.parametrize("n,depth", [(400, 2), (500, 3), (1500, 2), (3000, 3), (6000, 2), (11000, 2), (17000, 2)])
@pytest.mark.parametrize("precision,eps", [("fp64", 1e-9), ("fp32", 1e-5)])
def test_solve_inverts_the_fmm_matrix(n, depth, precision, eps):
    pts = torus(n, 5) if n % 1000 else bumpy_sphere(n, 5)
    t = ifmm.ifmm_build_tree(pts, depth)
    ifmm.ifmm_color(t, 3)
    f = ifmm.ifmm_factor(t, 3, eps, precision=precision)
    x = np.random.default_rng(n).standard_normal(n)
    y = ifmm.bem_matvec(t, x, kernel=ifmm.default_kernel(n, "fmm", 3))
    v = ifmm.ifmm_solve(f, y)
    assert np.linalg.norm(v - x) <= 1000 * eps * np.linalg.norm(x)
    g = ifmm.ifmm_factor(t, 3, eps, precision=precision)
    assert np.array_equal(v, ifmm.ifmm_solve(g, y))
