"""The FP64 Jacobi rotations with a problem on a cluster of 2, 4 or 8 CTAs: trees of
depth 2 have few problems per launch, so clusters, and their leaves reach the width
classes up to 48, 128, 256 and wider columns, with odd and even column counts; trees
of depth 3 mix clusters with single CTAs.  The factor approximates the inverse of the
FMM representation A~, whose product the library has as well, so ifmm_solve(A~ x)
must return x to the truncation eps times the few hundred that the elimination can
amplify (1000 allowed, as in the tests of the block widths); a race between the CTAs
would show as a second factor that differs."""

import numpy as np
import pytest

from paper_1905_10602_gb300 import build as _build
from paper_1905_10602_gb300.workloads import bumpy_sphere, torus

pytestmark = pytest.mark.gpu

_build.build()
from paper_1905_10602_gb300 import ifmm  # noqa: E402


@pytest.mark.parametrize("n,depth,order", [(601, 2, 3), (1300, 2, 4), (3501, 2, 4), (7000, 2, 3), (9001, 2, 4),
                                           (16000, 2, 3), (7501, 3, 4)])
def test_solve_inverts_the_fmm_matrix(n, depth, order):
    pts = torus(n, 4) if n % 2 else bumpy_sphere(n, 4)
    t = ifmm.ifmm_build_tree(pts, depth)
    ifmm.ifmm_color(t, 3)
    eps = 1e-10
    x = np.random.default_rng(n).standard_normal(n)
    y = ifmm.bem_matvec(t, x, kernel=ifmm.default_kernel(n, "fmm", order))
    v = ifmm.ifmm_solve(ifmm.ifmm_factor(t, order, eps), y)
    assert np.linalg.norm(v - x) <= 1000 * eps * np.linalg.norm(x)
    assert np.array_equal(v, ifmm.ifmm_solve(ifmm.ifmm_factor(t, order, eps), y))
