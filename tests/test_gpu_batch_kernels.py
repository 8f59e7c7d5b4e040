"""Kernels of the request server and of setup that work on many columns at once, and the folded
smoothing step, called in the library itself: both sides of every size rule, odd orders, the
same bits at any batch width, non-finite columns beside healthy ones."""
import ctypes

import numpy as np
import pytest

from tests.helpers import to_dev, to_host

pytestmark = pytest.mark.gpu

MODES = {"assign": 0, "residual": 1, "add": 2}


def _call(name, *args):
    from paper_2504_13373_gb300 import gasa
    conv = []
    for a in args:
        if a is None:
            conv.append(ctypes.c_void_p(None))
        elif hasattr(a, "data_ptr"):
            conv.append(ctypes.c_void_p(a.data_ptr()))
        else:
            conv.append(ctypes.c_int64(a) if isinstance(a, np.int64) else ctypes.c_int(int(a)))
    assert gasa.load()[name](*conv) == 0


def _bsr(rng, n, ncols, br, bc, lo, hi):
    """lo..hi blocks a row in increasing columns, some rows empty where lo is 0"""
    counts = rng.integers(lo, hi + 1, n)
    rp = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    start = rng.integers(0, ncols, n)
    k = np.arange(rp[-1]) - np.repeat(rp[:-1], counts)
    col = ((np.repeat(start, counts) + 3 * k) % ncols).astype(np.int32)
    return rp, col, rng.standard_normal((int(rp[-1]), br, bc))


def _apply(rp, col, val, X):
    """A X for X of (ncols, bc, K), in the precision of the arguments"""
    n, br = rp.size - 1, val.shape[1]
    y = np.zeros((n, br, X.shape[2]))
    step = 1 << 16
    rows = np.repeat(np.arange(n), np.diff(rp))
    for k in range(0, col.size, step):
        np.add.at(y, rows[k:k + step], np.einsum("kij,kjc->kic", val[k:k + step], X[col[k:k + step]]))
    return y


# few scalar rows are dealt to eight slices each (short rows by type, operation, number and
# length); many take a thread a row, or a warp from 16 blocks a row on (FP32 from 24
# blocks or 16,384 rows, FP64 from 155,648 rows)
SHAPES = [(1, 3, 3, 1, 1), (37, 5, 5, 0, 9), (700, 13, 13, 3, 30), (120, 28, 21, 2, 12),
          (3, 1, 1, 0, 2), (15565, 10, 10, 1, 4), (15563, 10, 10, 1, 4), (40000, 4, 4, 14, 20),
          (40000, 4, 9, 1, 3), (900, 10, 10, 20, 30), (2000, 10, 10, 14, 22), (1200, 10, 10, 0, 6),
          (1700, 10, 10, 1, 5), (39000, 4, 4, 16, 20)]


@pytest.mark.parametrize("t", ["f", "d"])
@pytest.mark.parametrize("n,br,bc,lo,hi", SHAPES)
def test_batched_products(n, br, bc, lo, hi, t):
    """Y = A X, B - A X and Y + A X on 1 to 8 columns: n terms of a row to n eps of
    sum |a x|; a column has the same bits at any width and beside non-finite columns."""
    dt, eps = (np.float32, 2.0 ** -23) if t == "f" else (np.float64, 2.0 ** -52)
    rng = np.random.default_rng(n + br)
    ncols = n if br == bc else 900
    rp, col, val = _bsr(rng, n, ncols, br, bc, lo, hi)
    val = val.astype(dt)
    x, b = rng.standard_normal((ncols, bc)).astype(dt), rng.standard_normal((n, br)).astype(dt)
    ax = _apply(rp, col, val.astype(np.float64), x[:, :, None].astype(np.float64))[:, :, 0]
    mag = _apply(rp, col, np.abs(val).astype(np.float64), np.abs(x)[:, :, None].astype(np.float64))[:, :, 0]
    tol = (hi * bc + 4) * eps * (mag + np.abs(b)) + 1e-300
    d = [to_dev(a) for a in (rp, col, val.ravel())]
    name = "_ZN4gasa10launch_bmvI%sEE9cudaErroriiiiPKiS3_PKT_S6_S6_PS4_iP11CUstream_stl" % t
    for mode, m in MODES.items():
        ref = {"assign": ax, "residual": b - ax, "add": b + ax}[mode]
        first = None
        for K in (1, 2, 4, 8):
            X, B = rng.standard_normal((ncols, bc, K)).astype(dt), rng.standard_normal((n, br, K)).astype(dt)
            c = K // 2
            if K > 2:
                X[:, :, 0], X[0, 0, K - 1] = np.inf, np.nan
            X[:, :, c], B[:, :, c] = x, b
            dB = to_dev(B)
            Y = dB.clone()
            _call(name, m, n, br, bc, *d, to_dev(X), dB, Y, K, None, np.int64(col.size))
            got = to_host(Y).reshape(n, br, K)[:, :, c]
            assert np.all(np.abs(got - ref) <= tol), (mode, K)
            first = got.copy() if first is None else first
            assert np.array_equal(got, first), (mode, K)


@pytest.mark.parametrize("t", ["f", "d"])
@pytest.mark.parametrize("n,bs,lo,hi", [(s[0], s[1], s[3], s[4]) for s in SHAPES if s[1] == s[2]])
def test_batched_smoothing_steps(n, bs, lo, hi, t):
    """Xo = X + W (B - A X) and Xo = W B on 1 to 8 columns, as above."""
    dt, eps = (np.float32, 2.0 ** -23) if t == "f" else (np.float64, 2.0 ** -52)
    rng = np.random.default_rng(n + bs)
    rp, col, val = _bsr(rng, n, n, bs, bs, lo, hi)
    val = val.astype(dt)
    W = (rng.standard_normal((n, bs, bs)) / bs).astype(dt)
    x, b = (rng.standard_normal((n, bs)).astype(dt) for _ in range(2))
    f64 = lambda a: a.astype(np.float64)
    ax = _apply(rp, col, f64(val), f64(x)[:, :, None])[:, :, 0]
    mag = _apply(rp, col, np.abs(f64(val)), np.abs(f64(x))[:, :, None])[:, :, 0]
    d = [to_dev(a) for a in (rp, col, val.ravel(), W.ravel())]
    name = "_ZN4gasa14launch_bjacobiI%sEE9cudaErroriiiPKiS3_PKT_S6_S6_S6_PS4_iP11CUstream_stl" % t
    for mode in (0, 1):                # a step; the first step from zero
        res = b - ax if mode == 0 else f64(b)
        ref = np.einsum("nij,nj->ni", f64(W), res) + (x if mode == 0 else 0.0)
        rtol = (hi * bs + 4) * eps * (mag + np.abs(b)) if mode == 0 else 0.0 * mag
        tol = np.einsum("nij,nj->ni", np.abs(f64(W)), rtol + bs * eps * np.abs(res))
        tol = tol + eps * (np.abs(x) + np.abs(ref)) + 1e-300
        first = None
        for K in (1, 2, 4, 8):
            X, B = (rng.standard_normal((n, bs, K)).astype(dt) for _ in range(2))
            c = K // 2
            if K > 2:
                X[:, :, 0], B[0, 0, K - 1] = np.inf, np.nan
            X[:, :, c], B[:, :, c] = x, b
            Xo = to_dev(np.zeros((n, bs, K), dt))
            _call(name, mode, n, bs, *d, to_dev(X), to_dev(B), Xo, K, None, np.int64(col.size))
            got = to_host(Xo)[:, :, c]
            assert np.all(np.abs(got - ref) <= tol), (mode, K)
            first = got.copy() if first is None else first
            assert np.array_equal(got, first), (mode, K)


@pytest.mark.parametrize("n,br,bc,ncol", [(1, 1, 1, 1), (5, 5, 5, 31), (40, 13, 13, 33), (9, 8, 8, 64),
                                          (30, 33, 33, 70), (12, 160, 160, 40), (17, 7, 24, 65), (6, 40, 9, 32)])
def test_setup_products_on_many_columns(n, br, bc, ncol):
    """The products and steps that form the dense bottom operator, and their unit vectors:
    FP64, n terms of a row to n 2^-52 of sum |a x|."""
    eps = 2.0 ** -52
    rng = np.random.default_rng(n + br)
    ncols = n if br == bc else 20
    rp, col, val = _bsr(rng, n, ncols, br, bc, 0, min(6, ncols))
    X, B = rng.standard_normal((ncols, bc, ncol)), rng.standard_normal((n, br, ncol))
    W = rng.standard_normal((n, br, br)) / br
    ax, mag = _apply(rp, col, val, X), _apply(rp, col, np.abs(val), np.abs(X))
    d = [to_dev(a) for a in (rp, col, val.ravel())]
    dX, dB, dW = to_dev(X), to_dev(B), to_dev(W.ravel())
    name = "_ZN4gasa9launch_mmEiiiiiPKiS1_PKdS3_S3_S3_PdP11CUstream_st"
    tol = (6 * bc + 4) * eps * (mag + np.abs(B)) + 1e-300
    wres = lambda r, rt: np.einsum("nij,njc->nic", np.abs(W), rt + br * eps * np.abs(r))
    res = B - ax
    steps = []
    if br == bc:
        steps.append((3, X + np.einsum("nij,njc->nic", W, res), wres(res, tol) + 4 * eps * (np.abs(X) + 1)))
        steps.append((4, np.einsum("nij,njc->nic", W, B), wres(B, 0.0) + 4 * eps))
    for op, ref, lim in [(0, ax, tol), (1, res, tol), (2, B + ax, tol)] + steps:
        Y = dB.clone()
        _call(name, op, n, br, bc, ncol, *d, dW, dX, dB, Y, None)
        assert np.all(np.abs(to_host(Y).reshape(n, br, ncol) - ref) <= lim), op
    m = n * br
    E = to_dev(np.ones((m, ncol)))
    _call("_ZN4gasa18launch_mm_identityEiiiPdP11CUstream_st", m, 2, ncol, E, None)
    assert np.array_equal(to_host(E).reshape(m, ncol), np.eye(m, ncol + 2)[:, 2:])
    D = rng.standard_normal((m, m))
    Y = to_dev(np.zeros((m, ncol)))
    _call("_ZN4gasa15launch_mm_denseEiiPKdS1_PdP11CUstream_st", m, ncol, to_dev(D), dB, Y, None)
    Bm = B.reshape(m, ncol)
    assert np.all(np.abs(to_host(Y).reshape(m, ncol) - D @ Bm) <= (m + 4) * eps * (np.abs(D) @ np.abs(Bm)) + 1e-300)


@pytest.mark.parametrize("bs", range(1, 13))
@pytest.mark.parametrize("n,lo,hi", [(1, 1, 1), (33, 0, 5), (5000, 3, 4), (300, 5, 40)])
def test_folded_step(n, bs, lo, hi):
    """x + (c - A x) in FP32, a lane per block up to 8 x 8 and a thread per row beyond."""
    eps = 2.0 ** -23
    rng = np.random.default_rng(n + bs)
    rp, col, val = _bsr(rng, n, n, bs, bs, lo, min(hi, n))
    val = val.astype(np.float32)
    x, c = (rng.standard_normal((n, bs)).astype(np.float32) for _ in range(2))
    ax = _apply(rp, col, val.astype(np.float64), x[:, :, None].astype(np.float64))[:, :, 0]
    mag = _apply(rp, col, np.abs(val).astype(np.float64), np.abs(x)[:, :, None].astype(np.float64))[:, :, 0]
    out = to_dev(np.zeros((n, bs), np.float32))
    _call("_ZN4gasa19launch_folded_sweepIfEE9cudaErroriiPKiS3_PKT_S6_S6_PS4_P11CUstream_stl", n, bs,
          to_dev(rp), to_dev(col), to_dev(val.ravel()), to_dev(x), to_dev(c), out, None,
          np.int64(col.size))
    tol = (hi * bs + 4) * eps * (mag + np.abs(c) + np.abs(x))
    assert np.all(np.abs(to_host(out) - (x + (c - ax))) <= tol)


def test_many_short_rows_are_not_sliced():
    """150,000 scalar rows of four blocks and eight columns: no slower than six times the
    15,000 that are dealt to slices (a thread a row takes about four times their time, slices
    take ten)."""
    import torch
    rng = np.random.default_rng(0)

    def ms(n):
        rp, col, val = _bsr(rng, n, n, 10, 10, 4, 4)
        X = to_dev(rng.standard_normal((n, 10, 8)).astype(np.float32))
        Y = torch.empty_like(X)
        d = [to_dev(a) for a in (rp, col, val.astype(np.float32).ravel())]
        name = "_ZN4gasa10launch_bmvIfEE9cudaErroriiiiPKiS3_PKT_S6_S6_PS4_iP11CUstream_stl"
        best = np.inf
        for _ in range(6):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda.synchronize()
            a.record()
            for _ in range(50):
                _call(name, 0, n, 10, 10, *d, X, Y, Y, 8, None, np.int64(col.size))
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) / 50)
        return best

    assert ms(15000) <= 6 * ms(1500)


@pytest.mark.parametrize("n,br,bc,per,limit", [(150, 17, 17, 98, 1.5e-7), (300, 13, 13, 25, 9.4e-8),
                                               (900, 4, 4, 75, 8.9e-8), (150, 20, 28, 20, 1.17e-7),
                                               (500, 12, 12, 17, 9.0e-8)])
def test_batched_products_rounding(n, br, bc, per, limit):
    """FP32 sums of long rows on few columns round like lanes that take whole blocks each: the
    rms error of random sums in units of their rms, to that (1.43e-7, 8.9e-8, 8.4e-8, 1.11e-7,
    8.5e-8) and about 5 %."""
    rng = np.random.default_rng(n)
    ncols = max(n, 3 * per + 1) if br != bc else n
    rp = (per * np.arange(n + 1)).astype(np.int32)
    col = ((np.arange(per)[None, :] + np.arange(n)[:, None]) % ncols).astype(np.int32).ravel()
    val = rng.standard_normal((n * per, br, bc)).astype(np.float32)
    err = []
    for K in (1, 8):
        X = rng.standard_normal((ncols, bc, K)).astype(np.float32)
        ref = _apply(rp, col, val.astype(np.float64), X.astype(np.float64))
        Y = to_dev(np.zeros((n, br, K), np.float32))
        _call("_ZN4gasa10launch_bmvIfEE9cudaErroriiiiPKiS3_PKT_S6_S6_PS4_iP11CUstream_stl", 0, n, br, bc,
              to_dev(rp), to_dev(col), to_dev(val.ravel()), to_dev(X), Y, Y, K, None, np.int64(col.size))
        err.append(np.sqrt(np.mean((to_host(Y) - ref) ** 2) / np.mean(ref ** 2)))
    assert max(err) <= limit, err
