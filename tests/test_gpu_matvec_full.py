"""The FP64 full sums (a thread per target), which products take whose partial sums
would exceed 8 GiB or find no room: IFMM_MATVEC64_FULL sends every size there, in a
child process.  Against the dense product in NumPy, Laplace and Helmholtz; bound: n
terms of a few rounding errors each, (n + 16) u of the sum of magnitudes."""

import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = r"""
import json, sys
import numpy as np
sys.path.insert(0, %(root)r)
from paper_1905_10602_gb300 import build as _build
from paper_1905_10602_gb300.workloads import bumpy_sphere
_build.build()
from paper_1905_10602_gb300 import ifmm
out = []
for n in (1, 2, 31, 255, 256, 257, 2000):
    pts = bumpy_sphere(max(n, 2), 5)[:n]
    t = ifmm.ifmm_build_tree(pts, 2)
    ifmm.ifmm_color(t, 3)
    r = np.linalg.norm(pts[:, None] - pts[None], axis=2)
    np.fill_diagonal(r, 1.0)
    g = np.random.default_rng(n)
    for wk in (0.0, 7.0):
        k = ifmm.helmholtz_kernel(n, wk) if wk else ifmm.default_kernel(n)
        x = g.standard_normal(n) + (1j * g.standard_normal(n) if wk else 0)
        A = k.scale * np.exp(1j * wk * r) / r if wk else k.scale / r
        A[np.arange(n), np.arange(n)] = k.diag + (1j * k.diag_im if wk else 0)
        y = ifmm.bem_matvec(t, x, kernel=k)
        # the phase w r of a term is rounded as well: a few units of w r
        tol = (n + 16 + 4 * wk) * 2.0 ** -53 * (np.abs(A) @ np.abs(x))
        out.append(float(np.max(np.abs(y - A @ x) / tol)))
print(json.dumps(out))
"""


def _child(env):
    p = subprocess.run([sys.executable, "-c", CHILD % {"root": ROOT}], capture_output=True, text=True, timeout=600,
                       env=dict(os.environ, **env))
    assert p.returncode == 0, p.stderr[-3000:]
    return json.loads(p.stdout.strip().splitlines()[-1])


@pytest.mark.parametrize("full", ["0", "1"])
def test_full_sums(full):
    assert max(_child({"IFMM_MATVEC64_FULL": full})) <= 1.0
