"""One-sided Jacobi on A = B D, B well conditioned and D = diag(2^-k): singular values
and vectors to the relative accuracy that B's condition gives, however small a column
is (Demmel and Veselic), against the same method in NumPy.  k reaches 400 bits in FP64
(squares and products of the norms leave FP64's range) and 54 in FP32 (the tangent's
square leaves FP32's).  Widths: a warp per problem, each class of a CTA, and in FP64
clusters of CTAs.

With cond(B) below about 4 a column pair's error is a few n u; 32 n u is allowed, for
the values relatively and for the vectors' orthogonality."""

import ctypes

import kernel_calls
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def svd(tmp_path_factory):
    kc = kernel_calls.load(kernel_calls.compile_to(str(tmp_path_factory.mktemp("kc") / "libkernel_calls.so")))

    def f(fp32, A):
        n = len(A)
        a, v, sig = np.asfortranarray(A), np.zeros((n, n), order="F"), np.zeros(n)
        assert kc.kc_svd(int(fp32), n, *[x.ctypes.data_as(ctypes.c_void_p) for x in (a, v, sig)]) == 0
        return v, sig

    return f


def _reference(B, k):
    """Singular values of B diag(2^-k): Jacobi on columns kept with exponents of their own, so that no product
    leaves the range."""
    C, e, n = B.copy(), -k, B.shape[1]
    for _ in range(30):
        rotated = False
        for i in range(n - 1):
            for j in range(i + 1, n):
                a, b = (i, j) if e[i] >= e[j] else (j, i)  # a is not the smaller one
                r = 2.0 ** float(e[b] - e[a])
                x, y = C[:, a], C[:, b]
                al, be, g = x @ x, y @ y, x @ y
                if abs(g) <= 1e-15 * np.sqrt(al * be):
                    continue
                rotated = True
                # columns x, r y: t = tan, formed from g r and be r^2 - al
                if r < 2.0 ** -60:
                    tr = g / -al  # t / r
                    C[:, a], C[:, b] = x - (tr * r * r) * y, tr * x + y
                else:
                    z = (be * r * r - al) / (2 * g * r)
                    t = np.copysign(1.0, z) / (abs(z) + np.hypot(1.0, z))
                    c = 1 / np.sqrt(1 + t * t)
                    C[:, a], C[:, b] = c * x - (c * t * r) * y, (c * t / r) * x + c * y
        if not rotated:
            break
    assert not rotated
    return np.sort(np.ldexp(np.linalg.norm(C, axis=0), e))[::-1]


CASES = [(False, n, bits) for n in (12, 24, 60, 100) for bits in (40, 100, 160, 400)]
CASES += [(False, 200, 100), (False, 300, 160)]
CASES += [(True, n, bits) for n in (12, 24, 60, 100, 200) for bits in (20, 40, 54)]


@pytest.mark.parametrize("fp32,n,bits", CASES)
def test_graded_columns(svd, fp32, n, bits):
    g = np.random.default_rng(n + bits)
    B = np.eye(n) + 0.3 * g.standard_normal((n, n)) / np.sqrt(n)
    if fp32:
        B = B.astype(np.float32).astype(np.float64)
    k = g.permutation(np.rint(np.linspace(0, bits, n)).astype(int))
    V, sig = svd(fp32, np.ldexp(B, -k[None, :]))
    tol = 32 * n * (2.0 ** -24 if fp32 else 2.0 ** -53)
    assert np.all(sig > 0)
    assert np.max(np.abs(sig / _reference(B, k) - 1)) <= tol
    assert np.abs(V.T @ V - np.eye(n)).max() <= tol
