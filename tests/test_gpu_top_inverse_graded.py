"""The level-1 inverse on its own (big_inverse on a matrix in hand), by panels and by
launches per column: orders around a panel of 32 columns and a tile of 64, rows and
columns of very different size, many interchanges, exact cases, a singular step.

A Gauss-Jordan inverse with partial pivoting of a well-conditioned matrix R leaves
||R X - I||_F <= c n u ||R||_F ||X||_F with c of a few (8 here, growth and the check's
own product included).  Scaling rows and columns by powers of two changes nothing of
that: for A = D1 R D2 the bound is asked of X with the scales taken out again, so digits
lost to the grading would show in full."""

import ctypes

import kernel_calls
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

U = 2.0 ** -53


@pytest.fixture(scope="module")
def inverse(tmp_path_factory):
    kc = kernel_calls.load(kernel_calls.compile_to(str(tmp_path_factory.mktemp("kc") / "libkernel_calls.so")))
    from paper_1905_10602_gb300 import ifmm

    def f(A, columns):
        n = len(A)
        a, x, info = np.asfortranarray(A), np.zeros((n, n), order="F"), np.zeros(1, np.int32)
        vp = [v.ctypes.data_as(ctypes.c_void_p) for v in (a, x, info)]
        assert kc.kc_top_inverse(n, *vp, int(columns)) == 0, ifmm.lib.ifmm_last_error()
        return x, int(info[0])

    return f


def _grades(kind, n, g):
    if kind == "flat":
        return np.zeros(n, int)
    if kind == "two levels":
        return -40 * (np.arange(n) % 2)
    if kind == "smooth":
        return -np.rint(np.linspace(0, 60, n)).astype(int)
    return g.integers(-40, 1, n)


@pytest.mark.parametrize("columns", [False, True])
@pytest.mark.parametrize("rows,cols", [("flat", "flat"), ("two levels", "flat"), ("smooth", "flat"), ("random", "flat"),
                                       ("flat", "random"), ("random", "two levels")])
@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 63, 64, 65, 200, 1000])
def test_residual(inverse, n, rows, cols, columns):
    g = np.random.default_rng(n)
    R = g.standard_normal((n, n))
    R[np.arange(n), (np.arange(n) * 7 + 3) % n if n % 7 else np.arange(n)] += 3 * np.sqrt(n)  # interchanges everywhere
    d1, d2 = _grades(rows, n, g), _grades(cols, n, g)
    X, info = inverse(np.ldexp(R, d1[:, None] + d2[None, :]), columns)
    assert info == 0
    X = np.ldexp(X, d2[:, None] + d1[None, :])
    res = np.linalg.norm(R @ X - np.eye(n))
    assert res <= 8 * n * U * np.linalg.norm(R) * np.linalg.norm(X)


@pytest.mark.parametrize("columns", [False, True])
@pytest.mark.parametrize("n", [1, 32, 33, 65, 300])
def test_exact(inverse, n, columns):
    """A permutation times powers of two over 2^+-200, and a diagonal: no rounding at all."""
    g = np.random.default_rng(n)
    for p in (np.arange(n), g.permutation(n)):
        e = g.integers(-200, 200, n)
        A = np.zeros((n, n))
        A[np.arange(n), p] = np.ldexp(1.0, e)
        B = np.zeros((n, n))
        B[p, np.arange(n)] = np.ldexp(1.0, -e)
        X, info = inverse(A, columns)
        assert info == 0 and np.array_equal(X, B)


@pytest.mark.parametrize("columns", [False, True])
@pytest.mark.parametrize("n,k", [(1, 0), (33, 0), (33, 32), (100, 40)])
def test_singular_step(inverse, n, k, columns):
    """A zero column: step k finds no pivot (a triangular matrix otherwise, so the steps before it are exact)."""
    A = np.triu(np.random.default_rng(n).integers(-3, 4, (n, n)).astype(float), 1) + np.eye(n)
    A[:, k] = 0
    assert inverse(A, columns)[1] == k + 1


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_not_finite(inverse, bad):
    """A NaN is never a pivot and stays visible; an infinite pivot has the reciprocal 0, as in the plain elimination
    by columns."""
    A = np.eye(100) * 3 + np.random.default_rng(1).standard_normal((100, 100)) * 0.1
    A[70, 20] = bad
    (X, info), (Y, info_columns) = inverse(A, False), inverse(A, True)
    if np.isnan(bad):
        assert info != 0 or not np.isfinite(X).all()
    else:
        assert info == info_columns == 0
        assert np.array_equal(np.isfinite(X), np.isfinite(Y))
        f = np.isfinite(Y)
        # ||X - A^-1|| <= ||A^-1|| ||A X - I||, twice
        tol = 2 * 8 * 100 * U * np.linalg.norm(A[np.isfinite(A)]) * np.linalg.norm(Y[f]) ** 2
        assert np.linalg.norm(X[f] - Y[f]) <= tol
