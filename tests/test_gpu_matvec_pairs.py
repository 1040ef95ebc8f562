"""The symmetric float-pair sum with tiles of 128 and of 256 points (one and two
targets per lane), forced, at point counts around the tiles, against the FP64 sum.

Bound per row: a pair-arithmetic term is accurate to about 2^-44 relative plus the
48-bit coordinates' 2^-46 R / r, the sums to 2^-44 of the absolute sum."""

import numpy as np
import pytest

from paper_1905_10602_gb300 import build as _build
from paper_1905_10602_gb300.workloads import bumpy_sphere, torus

pytestmark = pytest.mark.gpu

_build.build()
from paper_1905_10602_gb300 import ifmm  # noqa: E402


@pytest.mark.parametrize("tile,code", [("sym", 128), ("sym2", 256)])
@pytest.mark.parametrize("n", [1, 31, 127, 128, 129, 255, 256, 257, 511, 513, 1300])
def test_symmetric_tiles(monkeypatch, tile, code, n):
    monkeypatch.setenv("IFMM_MATVEC_TILE", tile)
    pts = torus(n, 7) if n % 2 else bumpy_sphere(n, 7)
    t = ifmm.ifmm_build_tree(pts, 2)
    x = np.random.default_rng(n).standard_normal(n)
    k = ifmm.default_kernel(n, "df")
    y = ifmm.bem_matvec(t, x, kernel=k)
    assert list(ifmm.ifmm_tree_query(t, 0, "matvec_block")) == [code, 3]
    r = np.sqrt(((pts[:, None] - pts[None]) ** 2).sum(-1))
    np.fill_diagonal(r, 1.0)
    A = k.scale / r
    np.fill_diagonal(A, k.diag)
    R = np.abs(pts).max()
    bound = (np.abs(A) * (2.0 ** -43 + 2.0 ** -46 * R / r)) @ np.abs(x)
    assert np.all(np.abs(A @ x - y) <= bound)
    assert np.array_equal(y, ifmm.bem_matvec(t, x, kernel=k))
