"""The dense bottom operator's products, called in the library itself: odd orders, batch
widths, non-finite columns, and rounding against exact sums."""
import ctypes
import math

import numpy as np
import pytest

from tests.helpers import to_dev, to_host

pytestmark = pytest.mark.gpu


def _fn(name):
    from paper_2504_13373_gb300 import gasa
    return gasa.load()[name]


def _ptr(t):
    return ctypes.c_void_p(t.data_ptr())


def _exact_rows(M, x):
    """sum_j M_ij x_j rounded once (products of 26-bit halves of M and FP32 x are exact)"""
    e = np.frexp(M)[1]
    hi = np.ldexp(np.round(np.ldexp(M, 25 - e)), e - 25)
    x = x.astype(np.float64)
    return np.array([math.fsum(np.concatenate([h * x, l * x])) for h, l in zip(hi, M - hi)])


def _cancelling(rng, n, spread):
    """(M, x): rows of ten decades whose products with x cancel to the rounding of their last"""
    M = rng.standard_normal((n, n)) * 10.0 ** rng.uniform(-spread, spread, (n, n))
    x = rng.standard_normal(n).astype(np.float32)
    if n > 1:
        M[:, -1] = 0.0
        M[:, -1] = -_exact_rows(M, x) / float(x[-1])
    return M, x


def _pitched(M):
    n = M.shape[0]
    ld = (n + 15) // 16 * 16 + 16
    out = np.zeros((n, ld))
    out[:, :n] = M
    return out, ld


@pytest.mark.parametrize("spread", [0.0, 5.0])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 255, 257, 816, 2048])
def test_batched_bottom_operator(n, spread):
    """On K columns: no further from the exact sum than a warp's FP64 chain at order 2,048
    (2.6 x 2^-53 of the products' norm, rms over the rows), the same bits at any K and beside
    non-finite columns."""
    f = _fn("_ZN4gasa19launch_bdense_splitEiiPKdPKfPfiP11CUstream_st")
    rng = np.random.default_rng(n)
    M, x = _cancelling(rng, n, spread)
    Mp, ld = _pitched(M)
    dM = to_dev(Mp)
    norm = np.sqrt(((M * x.astype(np.float64)) ** 2).sum(1))
    want = _exact_rows(M, x)
    first = None
    for K in (1, 2, 4, 8):
        B = rng.standard_normal((n, K)).astype(np.float32)
        c = K - 1
        if K > 2:
            B[n // 2, 0], B[0, 1] = np.inf, np.nan
        B[:, c] = x
        X = to_dev(np.zeros((n, K), np.float32))
        dB = to_dev(B)
        assert f(n, ld, _ptr(dM), _ptr(dB), _ptr(X), K, None) == 0
        got = to_host(X)
        assert np.isnan(got[:, 1]).all() if K > 2 else np.isfinite(got).all()
        err = (got[:, c].astype(np.float64) - want) / norm
        assert np.sqrt(np.mean(err ** 2)) <= 2.6 * 2.0 ** -53 + (2.0 ** -24 if n == 1 else 0.0)
        if first is None:
            first = got[:, c].copy()
        assert np.array_equal(got[:, c], first)


@pytest.mark.parametrize("n", [1, 5, 31, 33, 130, 515, 816, 1217, 2048, 2435])
def test_bottom_operator(n):
    """On one vector, orders on both sides of every split: with two FP32 words of the operator
    within 12 x 2^-53 of the products' norm (rms over the rows) of those words' exact sums;
    with FP64 multiply-adds to a warp's chain."""
    rng = np.random.default_rng(n)
    M, x = _cancelling(rng, n, 2.0)
    Mp, ld = _pitched(M)
    hi = Mp.astype(np.float32)
    lo = (Mp - hi).astype(np.float32)
    words = (hi.astype(np.float64) + lo)[:, :n]
    norm = np.sqrt(((M * x.astype(np.float64)) ** 2).sum(1))

    def rms(y, op):
        return np.sqrt(np.mean(((to_host(y).astype(np.float64) - _exact_rows(op, x)) / norm) ** 2))

    dM, dx = to_dev(Mp), to_dev(x)
    y = to_dev(np.zeros(n, np.float32))
    f = _fn("_ZN4gasa18launch_dense_mv_dsEiiPKfS1_S1_PfP11CUstream_st")
    dh, dl = to_dev(hi), to_dev(lo)
    one = 2.0 ** -24 if n == 1 else 0.0
    assert f(n, ld, _ptr(dh), _ptr(dl), _ptr(dx), _ptr(y), None) == 0
    assert rms(y, words) <= 12 * 2.0 ** -53 + one
    for t, m, v in ((np.float32, "If", dx), (np.float64, "Id", to_dev(x.astype(np.float64)))):
        y = to_dev(np.zeros(n, t))
        g = _fn("_ZN4gasa15launch_dense_mv%sEE9cudaErroriPKdPKT_PS4_P11CUstream_sti" % m)
        assert g(n, _ptr(dM), _ptr(v), _ptr(y), None, ld) == 0
        assert rms(y, M) <= 3 * 2.0 ** -53 + one
