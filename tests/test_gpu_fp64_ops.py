"""The FP64 reciprocal square root and reciprocal on their own, over every exponent and
at the values that leave the fast path.

rsqrt_fp64: the start value is off by 2^-21 at most, so the step's next term is below
2^-60; a * y0 is rounded once (2^-54 of the result), the last operation once: one ulp
and a little, 1.1 allowed.  rcp_fp64: the second Newton step leaves the rounding of the
last operation, half an ulp and a little, 0.6 allowed.  Zero, infinities, NaN,
negative and subnormal arguments give what IEEE arithmetic gives."""

import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1905_10602_gb300 import build as _build

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def ops(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("ops") / "libfp64_ops.so")
    subprocess.run([os.path.join(_build.CUDA, "bin", "nvcc"), _build.ARCH, "-O3", "-std=c++17", "-shared", "-Xcompiler",
                    "-fPIC", "-I" + _build.CSRC, os.path.join(HERE, "fp64_ops_check.cu"), "-o", so], check=True)
    lib = ctypes.CDLL(so)

    def f(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        r, q = np.empty_like(x), np.empty_like(x)
        p = [v.ctypes.data_as(ctypes.c_void_p) for v in (x, r, q)]
        assert lib.fp64_ops(p[0], len(x), p[1], p[2]) == 0
        return r, q

    return f


def _ulps(got, want):
    """|got - want| in units of the last place of want (long double)."""
    ulp = np.spacing(np.abs(want).astype(np.float64)).astype(np.longdouble)
    return np.max(np.abs(got.astype(np.longdouble) - want) / ulp)


def test_accuracy(ops):
    g = np.random.default_rng(1)
    m = np.concatenate([1 + g.random(40), 1 + 2.0 ** -g.uniform(1, 52, 20), 2 - 2.0 ** -g.uniform(1, 51, 20), [1.0, 1.5]])
    x = np.ldexp(m[None, :], np.arange(-1022, 1023)[:, None]).ravel()
    r, q = ops(x)
    xl = x.astype(np.longdouble)
    assert _ulps(r, 1 / np.sqrt(xl)) <= 1.1
    assert _ulps(q, 1 / xl) <= 0.6
    rn, qn = ops(-x)
    assert np.isnan(rn).all() and _ulps(qn, -1 / xl) <= 0.6


def test_special_values(ops):
    sub = np.ldexp(1.0, np.arange(-1074, -1022))
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, *sub, *-sub, np.finfo(float).max, np.finfo(float).tiny])
    r, q = ops(x)
    with np.errstate(all="ignore"):
        want = (1 / np.sqrt(x.astype(np.longdouble))).astype(np.float64)
        inv = 1 / x
    assert np.allclose(r, want, rtol=2.0 ** -51, atol=0, equal_nan=True)
    assert np.allclose(q, inv, rtol=2.0 ** -51, atol=0, equal_nan=True) and np.array_equal(np.signbit(q), np.signbit(inv))
