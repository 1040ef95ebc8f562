"""ifmm_solve with several right-hand sides: groups of four and two share one pass
over the coefficients and must give what single ones give (the same operations in
the same order: equal bits), for FP64 and reduced-precision factors and the
block-diagonal one, host and device vectors, in place as well."""

import numpy as np
import pytest

from paper_1905_10602_gb300 import build as _build
from paper_1905_10602_gb300.workloads import torus

pytestmark = pytest.mark.gpu

_build.build()
from paper_1905_10602_gb300 import ifmm  # noqa: E402


@pytest.mark.parametrize("kind", ["fp64", "fp32", "bd"])
@pytest.mark.parametrize("nrhs", [1, 2, 3, 4, 5, 7, 9])
def test_groups_equal_single_solves(kind, nrhs):
    import torch

    n = 1501
    t = ifmm.ifmm_build_tree(torus(n, 3), 3)
    ifmm.ifmm_color(t, 3)
    f = ifmm.ifmm_bd_factor(t, 3) if kind == "bd" else ifmm.ifmm_factor(t, 3, 1e-6, precision=kind)
    R = np.random.default_rng(nrhs).standard_normal((nrhs, n))
    one = np.stack([ifmm.ifmm_solve(f, R[c]) for c in range(nrhs)])
    assert np.array_equal(ifmm.ifmm_solve(f, R), one)
    d = torch.from_numpy(R).cuda()
    assert np.array_equal(ifmm.ifmm_solve(f, d).cpu().numpy(), one)
    ifmm._check(ifmm.lib.ifmm_solve(f.h, ifmm._ptr(d), ifmm._ptr(d), nrhs, ifmm._stream(d)))
    assert np.array_equal(d.cpu().numpy(), one)
