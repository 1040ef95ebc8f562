"""The FP64 direct sums with each unordered pair evaluated once, against the plain
sums in NumPy, at point counts around the tiles of 64 (small problems) and 128
points (above about 6,200) and at magnitudes that leave the FP32 range (the start
value of 1/r comes from FP32 bits).

Bound per row: each term is off by at most 8 units of roundoff u (difference,
squares, 1/r, product), the Helmholtz phase by 4 u k r on top, and a sum of n
terms by n u of the absolute sum, on both sides: 2 (n + 8 + 4 k r_max) u sum |a_ij x_j|."""

import numpy as np
import pytest

from paper_1905_10602_gb300 import build as _build
from paper_1905_10602_gb300.workloads import bumpy_sphere, torus

pytestmark = pytest.mark.gpu

_build.build()
from paper_1905_10602_gb300 import ifmm  # noqa: E402

U = 2.0 ** -53


def _check(pts, x, kern, k):
    n = len(pts)
    t = ifmm.ifmm_build_tree(pts, 2)
    y = ifmm.bem_matvec(t, x, kernel=kern)
    assert np.array_equal(y, ifmm.bem_matvec(t, x, kernel=kern))
    for i0 in range(0, n, 1024):
        p = pts[i0:i0 + 1024]
        r = np.sqrt(((p[:, None, :] - pts[None, :, :]) ** 2).sum(-1))
        rows = np.arange(len(p))
        r[rows, i0 + rows] = 1.0
        A = kern.scale / r * (np.exp(1j * k * r) if k else 1.0)
        A[rows, i0 + rows] = complex(kern.diag, kern.diag_im) if k else kern.diag
        bound = 2 * (n + 8 + 4 * abs(k) * r.max()) * U * (np.abs(A) @ np.abs(x))
        assert np.all(np.abs(A @ x - y[i0:i0 + 1024]) <= bound)


@pytest.mark.parametrize("n", [1, 2, 31, 63, 64, 65, 129, 1000, 6500])
@pytest.mark.parametrize("k", [0.0, 7.5])
def test_matvec_tile_edges(n, k):
    pts = torus(n, 3)
    g = np.random.default_rng(n)
    x = g.standard_normal(n) + (1j * g.standard_normal(n) if k else 0.0)
    kern = ifmm.helmholtz_kernel(n, k) if k else ifmm.default_kernel(n)
    _check(pts, x, kern, k)


@pytest.mark.parametrize("scale", [1e-120, 1e-30, 1.0, 1e25, 1e110])
def test_laplace_magnitudes(scale):
    n = 300
    x = np.random.default_rng(5).standard_normal(n)
    _check(bumpy_sphere(n, 4) * scale, x, ifmm.default_kernel(n), 0.0)


@pytest.mark.parametrize("k", [-3.0, 1e-9, 4.0e5, 3.0e6])
def test_helmholtz_phase_ranges(k):
    """Negative, tiny and large phases, on both sides of the table's range (10^6)."""
    n = 200
    g = np.random.default_rng(6)
    x = g.standard_normal(n) + 1j * g.standard_normal(n)
    _check(bumpy_sphere(n, 4), x, ifmm.Kernel(1.0 / n, 0.5, 0, 0, k, 0.25), k)
