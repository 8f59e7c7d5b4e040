"""Kernels and launch paths chosen by size, against the general path or the oracle."""
import numpy as np
import pytest

from tests.helpers import gpu_setup, problem, rel_err, to_dev

pytestmark = pytest.mark.gpu


def _gasa():
    from paper_2504_13373_gb300 import gasa
    return gasa


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("name", ["p3_16", "uneq6", "cd_q2_16"])
def test_vcycle_graph_same_bits(name, prec):
    """From the second V-cycle on the launches come from one graph: the same kernels on the
    same data as the first call's direct launches, for any vectors and after a new setup."""
    import torch
    gasa = _gasa()
    pr = problem(name)
    ctx, _ = gpu_setup(name)
    try:
        rng = np.random.default_rng(5)
        rs = [to_dev(rng.standard_normal(pr.n_dofs)) for _ in range(3)]
        first = torch.empty_like(rs[0])
        gasa.gasa_vcycle(ctx, rs[0], first, prec)
        for r in (rs[1], rs[2], rs[0]):
            z = torch.empty_like(r)
            gasa.gasa_vcycle(ctx, r, z, prec)
            fresh, _ = gpu_setup(name)
            try:
                ref = torch.empty_like(r)
                gasa.gasa_vcycle(fresh, r, ref, prec)     # a first call: direct launches
                assert torch.equal(z, ref)
            finally:
                gasa.gasa_destroy(fresh)
        assert torch.equal(z, first)
        same = rs[0].clone()
        gasa.gasa_vcycle(ctx, same, same, prec)           # in place
        assert torch.equal(same, first)
    finally:
        gasa.gasa_destroy(ctx)


@pytest.mark.parametrize("n_units,bs,size,r,s_next", [
    (24, 10, 8, 80, 13),      # the 3-D workload's level 0
    (16, 17, 8, 80, 22),      # more rows than candidates, five lane strides
    (24, 3, 4, 37, 5),        # fewer rows than candidates, an odd count
    (6, 2, 3, 256, 6),        # the most candidates: several rounds of ten pairs a warp
    (32, 10, 4, 4, 4),        # two pairs
    (22, 1, 11, 21, 1),       # eleven rows, a short last chunk of pairs
])
def test_tentative_packed_sums(n_units, bs, size, r, s_next):
    """Candidates of ten decades of singular values against LAPACK: singular values to the
    rounding of sigma_1, kept vectors to that over their gap, orthonormal columns."""
    from oracle import gasa_oracle as O
    gasa = _gasa()
    rng = np.random.default_rng(n_units * 100 + r)
    n = n_units * bs
    agg = np.arange(n_units) // size
    n_agg = int(agg.max()) + 1
    B = rng.standard_normal((n, r))
    for J in range(n_agg):
        rows = np.nonzero(np.repeat(agg, bs) == J)[0]
        U, S, V = np.linalg.svd(B[rows], full_matrices=False)
        B[rows] = (U * 10.0 ** (-10.0 * np.arange(S.size) / S.size)) @ V
    Tw, _, sv = O.tentative(B, agg, np.arange(n_units + 1) * bs, n_agg, 3.0, keep=[s_next] * n_agg)
    T, sig = to_dev(np.zeros(n * s_next)), to_dev(np.zeros(n_agg * r))
    gasa.gasa_tentative(n_units, bs, n_agg, to_dev(agg.astype(np.int32)),
                        to_dev(B.ravel(order="F")), r, s_next, T, sig)
    Tg, sg = T.cpu().numpy().reshape(n, s_next), sig.cpu().numpy().reshape(n_agg, r)
    for J in range(n_agg):
        rows = np.nonzero(np.repeat(agg, bs) == J)[0]
        Td = Tw.tocsr()[rows][:, J * s_next:(J + 1) * s_next].toarray()
        s = sv[J]
        gap = np.min(np.abs(np.diff(s[:s_next + 1]))) / s[0] if s.size > 1 else 1.0
        eps = 1e-15 * max(rows.size, r)
        assert np.max(np.abs(sg[J, :s.size] - s)) <= eps * s[0]
        assert np.max(np.abs(Tg[rows] - Td)) <= 10 * eps / gap, J
        assert np.max(np.abs(Tg[rows].T @ Tg[rows] - np.eye(s_next))) <= 1e-12


def _random_bsr(rng, n, ncols, br, bc, lo, hi):
    """(row_ptr, col, val) with lo..hi blocks per row (one row empty when lo is 0)."""
    counts = rng.integers(lo, hi + 1, n)
    rp = np.concatenate([[0], np.cumsum(counts)]).astype(np.int32)
    col = np.concatenate([np.sort(rng.choice(ncols, c, replace=False)) for c in counts] or
                         [np.zeros(0)]).astype(np.int32)
    return rp, col, rng.standard_normal((int(rp[-1]), br, bc))


def _bsr_apply(rp, col, val, x):
    n, br, bc = rp.size - 1, val.shape[1], val.shape[2]
    y = np.zeros((n, br))
    prod = np.einsum("kij,kj->ki", val, x.reshape(-1, bc)[col])
    np.add.at(y, np.repeat(np.arange(n), np.diff(rp)), prod)
    return y.ravel()


@pytest.mark.parametrize("br,bc", [(9, 9), (13, 13), (17, 17), (12, 12), (22, 22), (31, 31),
                                   (36, 36), (40, 40), (38, 38), (33, 33), (39, 13), (4, 30),
                                   (13, 10), (1, 40), (40, 9)])
@pytest.mark.parametrize("n,lo,hi", [(1, 9, 9), (45, 0, 30), (700, 8, 14)])
def test_wide_team_products(br, bc, n, lo, hi):
    """FP32 products and smoothing steps with wide blocks at every load width, team shape and
    a ragged last team: n terms of a row to n 2^-23 of sum |a x|."""
    gasa = _gasa()
    rng = np.random.default_rng(br * 100 + bc + n)
    ncols = max(n, hi)
    rp, col, val = _random_bsr(rng, n, ncols, br, bc, lo, hi)
    val = val.astype(np.float32)
    x, b = rng.standard_normal(ncols * bc).astype(np.float32), rng.standard_normal(n * br).astype(np.float32)
    ax = _bsr_apply(rp, col, val.astype(np.float64), x.astype(np.float64))
    mag = _bsr_apply(rp, col, np.abs(val).astype(np.float64), np.abs(x).astype(np.float64))
    tol = (hi * bc + 4) * 2.0 ** -23 * (mag + np.abs(b)) + 1e-30
    d = [to_dev(a) for a in (rp, col, val.ravel(), x, b)]
    for mode, ref in ((0, ax), (1, b - ax), (2, b + ax)):
        y = d[4].clone()
        gasa.gasa_bsr_mv_f32(mode, n, br, bc, *d[:4], d[4], y)
        assert np.all(np.abs(y.cpu().numpy() - ref) <= tol)
    if br != bc or ncols != n:
        return
    W = (rng.standard_normal((n, br, br)) / br).astype(np.float32)
    out = to_dev(np.zeros(n * br, np.float32))
    gasa.gasa_jacobi_sweep_f32(n, br, *d[:3], to_dev(W.ravel()), d[3], d[4], out)
    r = (b - ax).reshape(n, br)
    ref = x + np.einsum("nij,nj->ni", W.astype(np.float64), r).ravel()
    wtol = np.einsum("nij,nj->ni", np.abs(W).astype(np.float64),
                     (tol + np.abs(r).ravel() * br * 2.0 ** -23).reshape(n, br)).ravel()
    assert np.all(np.abs(out.cpu().numpy() - ref) <= wtol + 2.0 ** -23 * (np.abs(x) + np.abs(ref)))


@pytest.mark.parametrize("dtype", ["fp32", "fp64"])
@pytest.mark.parametrize("br,bc,n,lo,hi", [
    (10, 10, 7000, 0, 16),      # many scalar rows, short and long ones mixed: each takes its kernel
    (13, 13, 5100, 7, 8),       # lengths on both sides of the line
    (20, 20, 3300, 2, 12),      # no thread-per-row kernel at this width
    (10, 10, 900, 0, 12),       # few scalar rows
    (3, 3, 2048, 2, 5), (4, 4, 40000, 1, 9), (8, 8, 300, 20, 40), (1, 1, 5, 1, 3),
    (4, 10, 20000, 1, 12), (10, 4, 8000, 1, 4), (45, 45, 30, 1, 9),
])
def test_products_without_a_known_row_length(dtype, br, bc, n, lo, hi):
    """Single operations choose by sizes and by each row's own length: against the product
    in 64 bits, aligned and not, n terms of a row to n eps of sum |a x|."""
    import torch
    gasa = _gasa()
    rng = np.random.default_rng(br * 1000 + n)
    t, eps = (np.float32, 2.0 ** -23) if dtype == "fp32" else (np.float64, 2.0 ** -52)
    ncols = max(n, hi) if br == bc else 4000
    rp, col, val = _random_bsr(rng, n, ncols, br, bc, lo, hi)
    val = val.astype(t)
    x, b = rng.standard_normal(ncols * bc).astype(t), rng.standard_normal(n * br).astype(t)
    ax = _bsr_apply(rp, col, val.astype(np.float64), x.astype(np.float64))
    mag = _bsr_apply(rp, col, np.abs(val).astype(np.float64), np.abs(x).astype(np.float64))
    tol = (hi * bc + 4) * eps * (mag + np.abs(b)) + 1e-30
    f = gasa.gasa_bsr_mv_f32 if dtype == "fp32" else gasa.gasa_bsr_mv
    sweep = gasa.gasa_jacobi_sweep_f32 if dtype == "fp32" else gasa.gasa_jacobi_sweep
    drp, dcol, db = to_dev(rp), to_dev(col), to_dev(b)
    for shift in (0, 1):        # 1: values and x one element off their allocation's alignment
        dval = torch.empty(val.size + 1, dtype=torch.from_numpy(val).dtype, device="cuda")[shift:shift + val.size]
        dx = torch.empty(x.size + 1, dtype=dval.dtype, device="cuda")[shift:shift + x.size]
        dval.copy_(to_dev(val.ravel()))
        dx.copy_(to_dev(x))
        for mode, ref in ((0, ax), (1, b - ax), (2, b + ax)):
            y = db.clone()
            f(mode, n, br, bc, drp, dcol, dval, dx, db, y)
            assert np.all(np.abs(y.cpu().numpy() - ref) <= tol), (mode, shift)
        if br == bc and ncols == n:
            W = (rng.standard_normal((n, br, br)) / br).astype(t)
            out = torch.zeros_like(db)
            sweep(n, br, drp, dcol, dval, to_dev(W.ravel()), dx, db, out)
            r = (b - ax).reshape(n, br)
            ref = x + np.einsum("nij,nj->ni", W.astype(np.float64), r).ravel()
            wtol = np.einsum("nij,nj->ni", np.abs(W).astype(np.float64),
                             (tol + np.abs(r).ravel() * br * eps).reshape(n, br)).ravel()
            assert np.all(np.abs(out.cpu().numpy() - ref) <= wtol + eps * (np.abs(x) + np.abs(ref))), shift


@pytest.mark.parametrize("br,bc", [(12, 12), (16, 16), (21, 21), (13, 13), (64, 64), (4, 9),
                                   (36, 9), (1, 33), (40, 2), (6, 6)])
@pytest.mark.parametrize("n,lo,hi", [(1, 1, 1), (37, 0, 70), (300, 16, 40)])
def test_fp64_team_products(br, bc, n, lo, hi):
    """FP64 products on few rows, every split of a block's values over lanes and warps: n
    terms of a row to n 2^-52 of sum |a x|."""
    gasa = _gasa()
    rng = np.random.default_rng(br * 100 + bc + n)
    ncols = max(n, hi)
    rp, col, val = _random_bsr(rng, n, ncols, br, bc, lo, hi)
    x, b = rng.standard_normal(ncols * bc), rng.standard_normal(n * br)
    ax, mag = _bsr_apply(rp, col, val, x), _bsr_apply(rp, col, np.abs(val), np.abs(x))
    tol = (hi * bc + 4) * 2.0 ** -52 * (mag + np.abs(b)) + 1e-300
    d = [to_dev(a) for a in (rp, col, val.ravel(), x, b)]
    for mode, ref in ((0, ax), (1, b - ax), (2, b + ax)):
        y = d[4].clone()
        gasa.gasa_bsr_mv(mode, n, br, bc, *d[:4], d[4], y)
        assert np.all(np.abs(y.cpu().numpy() - ref) <= tol)
    if br == bc and ncols == n:
        W = rng.standard_normal((n, br, br)) / br
        out = to_dev(np.zeros(n * br))
        gasa.gasa_jacobi_sweep(n, br, *d[:3], to_dev(W.ravel()), d[3], d[4], out)
        r = (b - ax).reshape(n, br)
        ref = x + np.einsum("nij,nj->ni", W, r).ravel()
        wtol = np.einsum("nij,nj->ni", np.abs(W),
                         (tol + np.abs(r).ravel() * br * 2.0 ** -52).reshape(n, br)).ravel()
        assert np.all(np.abs(out.cpu().numpy() - ref) <= wtol + 2.0 ** -52 * (np.abs(x) + np.abs(ref)))


@pytest.mark.parametrize("n,b", [(160, 13), (64, 21), (35, 36), (40, 12), (16, 40)])
def test_vcycle_few_long_rows(n, b):
    """Few block rows of many blocks, each shared by a cluster of CTAs: the V-cycle on a
    random SPD operator, ragged rows, against the oracle's (FP64 to the conditioning of the
    kept vectors, FP32 to 1e-4, the bounds of the solver's V-cycle tests)."""
    from oracle import gasa_oracle as O
    from tests.test_gpu_solver import level_tolerances
    gasa = _gasa()
    rng = np.random.default_rng(n * 100 + b)
    keep = rng.random((n, n)) < 0.8
    keep = keep | keep.T | np.eye(n, dtype=bool)
    A = rng.standard_normal((n, b, n, b)) * keep[:, None, :, None]
    A = A.reshape(n * b, n * b)
    A = (A + A.T) / np.sqrt(8.0 * n * b) + 4.0 * np.eye(n * b)
    rp = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int32)
    row, col = np.nonzero(keep)
    val = np.ascontiguousarray(A.reshape(n, b, n, b)[row, :, col, :])
    agg = [np.arange(n, dtype=np.int32) // 8]
    B0 = rng.standard_normal((n * b, 2 * b))
    H = O.setup(rp, col.astype(np.int32), val, agg, B0=B0, r=2 * b, dim=2)
    ctx = gasa.gasa_create(0)
    try:
        gasa.gasa_setup(ctx, rp, col.astype(np.int32), val.ravel(), b, agg,
                        gasa.gasa_default_options(dim=2, n_cand=2 * b, dense_tail_dofs=0),
                        init_candidates=B0)
        f = rng.standard_normal(n * b)
        want = O.make_vcycle(H)(f)
        z = to_dev(np.zeros(n * b))
        gasa.gasa_vcycle(ctx, to_dev(f), z)
        assert rel_err(z.cpu().numpy(), want) <= 0.1 * level_tolerances(H)[-1]
        gasa.gasa_vcycle(ctx, to_dev(f), z, gasa.GASA_PREC_MIXED32)
        assert rel_err(z.cpu().numpy(), want) <= 1e-4
    finally:
        gasa.gasa_destroy(ctx)


@pytest.mark.parametrize("prec", ["mixed32", "mixed16"])
def test_mixed_cg_level0_blocks_wider_than_16(prec):
    """P3 tetrahedra (20 x 20 blocks): the double-single product of the Krylov step and its
    p . q partial sums, graph-resident and host-driven, against the oracle's mixed solve."""
    from oracle import gasa_oracle as O
    from synth import configs
    gasa = _gasa()
    pr = configs.poisson3d(3, 3, r=80)
    A = pr.A
    H = O.setup(A.row_ptr, A.col, A.val, pr.agg_of, B0=pr.B0, r=pr.r, dim=3)
    want = O.solve(H, pr.rhs, 1e-10, "cg", precision=prec, max_iter=500)
    P = gasa.GASA_PREC_MIXED32 if prec == "mixed32" else gasa.GASA_PREC_MIXED16
    ctx = gasa.gasa_create(0)
    try:
        gasa.gasa_setup(ctx, A.row_ptr, A.col, A.val.ravel(), A.b, pr.agg_of,
                        gasa.gasa_default_options(dim=3, n_cand=pr.r), adj_ptr=pr.adj_ptr,
                        adj_idx=pr.adj_idx, centroids=pr.centroids, init_candidates=pr.B0)
        for host_driven in (False, True):
            gasa.gasa_profile_enable(ctx, host_driven)
            x = np.zeros_like(pr.rhs)
            info = gasa.gasa_solve(ctx, pr.rhs, x, 1e-10, P)
            assert info.converged and info.rel_residual <= 1e-10
            assert abs(info.iterations - want.iterations) <= 1, (info.iterations, want.iterations)
    finally:
        gasa.gasa_destroy(ctx)


@pytest.mark.parametrize("n,b,per_row,limit", [
    (3000, 12, 25, 9.5e-8), (5400, 12, 17, 9.5e-8), (8000, 10, 15, 9.0e-8), (200, 36, 50, 1.2e-7),
    (4000, 13, 25, 9.5e-8), (3000, 16, 27, 9.8e-8)])
def test_wide_team_rounding(n, b, per_row, limit):
    """FP32 sums of wide blocks round like sums taken block by block in several groups: the
    rms error over the rows of random values, in units of the sums' rms, to that of eight
    groups of blocks (8.4e-8, 8.4e-8, 7.9e-8, 1.1e-7, 8.8e-8, 9.1e-8) and about 8 %."""
    gasa = _gasa()
    rng = np.random.default_rng(n + b)
    rp = (per_row * np.arange(n + 1)).astype(np.int32)
    col = np.sort(np.argsort(rng.random((n, max(2 * per_row, 60))), axis=1)[:, :per_row], axis=1)
    col = ((col + 7 * np.arange(n)[:, None]) % n).astype(np.int32).ravel()
    val = rng.standard_normal((n * per_row, b, b)).astype(np.float32)
    x = rng.standard_normal(n * b).astype(np.float32)
    want = np.einsum("nkij,nkj->ni", val.astype(np.float64).reshape(n, per_row, b, b),
                     x.astype(np.float64).reshape(n, b)[col].reshape(n, per_row, b)).ravel()
    y = to_dev(np.zeros(n * b, np.float32))
    gasa.gasa_bsr_mv_f32(0, n, b, b, to_dev(rp), to_dev(col), to_dev(val.ravel()), to_dev(x), y, y)
    err = np.sqrt(np.mean((y.cpu().numpy() - want) ** 2) / np.mean(want ** 2))
    assert err <= limit, err


@pytest.mark.parametrize("n,br,bc,per_row", [(8000, 10, 10, 15), (4300, 16, 16, 20), (9000, 8, 12, 9)])
def test_many_long_rows_of_unknown_length(n, br, bc, per_row):
    """Many rows, all of them long, in one call: no slower than four times the same rows in
    two calls that are few rows each (and take teams or lanes for all of them)."""
    import torch
    gasa = _gasa()
    rng = np.random.default_rng(n)
    rp = (per_row * np.arange(n + 1)).astype(np.int32)
    col = ((np.arange(per_row)[None, :] * 3 + np.arange(n)[:, None]) % n)
    col = np.sort(col, axis=1).astype(np.int32).ravel()
    val = rng.standard_normal((n * per_row, br, bc)).astype(np.float32)
    x = rng.standard_normal(n * bc).astype(np.float32)
    dv, dx, dc = to_dev(val.ravel()), to_dev(x), to_dev(col)
    y, y2 = to_dev(np.zeros(n * br, np.float32)), to_dev(np.zeros(n * br, np.float32))
    h = n // 2
    drp, drp1, drp2 = to_dev(rp), to_dev(rp[:h + 1]), to_dev(rp[h:] - rp[h])
    k = int(rp[h])

    def whole():
        gasa.gasa_bsr_mv_f32(0, n, br, bc, drp, dc, dv, dx, y, y)

    def halves():
        gasa.gasa_bsr_mv_f32(0, h, br, bc, drp1, dc, dv, dx, y2, y2)
        gasa.gasa_bsr_mv_f32(0, n - h, br, bc, drp2, dc[k:], dv[k * br * bc:], dx, y2[h * br:], y2[h * br:])

    def ms(f):
        best = np.inf
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(20):
                f()
            b.record()
            b.synchronize()
            best = min(best, a.elapsed_time(b) / 20)
        return best

    whole()
    halves()
    ref = _bsr_apply(rp, col, val.astype(np.float64), x.astype(np.float64))
    mag = _bsr_apply(rp, col, np.abs(val).astype(np.float64), np.abs(x).astype(np.float64))
    for got in (y, y2):
        assert np.all(np.abs(got.cpu().numpy() - ref) <= (per_row * bc + 4) * 2.0 ** -23 * mag)
    assert ms(whole) <= 4 * ms(halves)


@pytest.mark.parametrize("n,b", [(48, 37), (30, 33)])
def test_vcycle_odd_widths_beyond_a_warp(n, b):
    """Blocks wider than a warp that are read an entry at a time, in a hierarchy."""
    test_vcycle_few_long_rows(n, b)


@pytest.mark.parametrize("call", ["vcycle", "solve"])
def test_graphs_are_not_captured_on_the_callers_stream(call):
    """What another thread enqueues on the stream that the caller gave, while a graph is being
    built, runs once and does not become part of the graph."""
    import threading
    import torch
    gasa = _gasa()
    pr = problem("p3_16")
    A = pr.A
    stream = torch.cuda.Stream()
    ctx = gasa.gasa_create(0, stream)
    try:
        gasa.gasa_setup(ctx, A.row_ptr, A.col, A.val.ravel(), A.b, pr.agg_of,
                        gasa.gasa_default_options(dim=2, n_cand=pr.r), adj_ptr=pr.adj_ptr,
                        adj_idx=pr.adj_idx, centroids=pr.centroids, init_candidates=pr.B0)
        r = to_dev(pr.rhs)
        z, z2, x = torch.empty_like(r), torch.empty_like(r), torch.empty_like(r)
        count = torch.zeros(1, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        gasa.gasa_vcycle(ctx, r, z, 1)
        added, stop, started, errors = [0], threading.Event(), threading.Event(), []

        def other():
            try:
                with torch.cuda.stream(stream):
                    while not stop.is_set():
                        count.add_(1.0)
                        added[0] += 1
                        started.set()
            except Exception as e:      # a launch refused because of the capture
                errors.append(e)
                started.set()

        t = threading.Thread(target=other)
        t.start()
        started.wait()
        try:
            if call == "vcycle":
                gasa.gasa_vcycle(ctx, r, z2, 1)                       # builds its graph
            else:
                gasa.gasa_solve(ctx, r, x, 1e-8, 1, on_device=True)   # builds the CG graph
        finally:
            stop.set()
            t.join()
        for _ in range(3):
            gasa.gasa_vcycle(ctx, r, z2, 1)
        torch.cuda.synchronize()
        assert not errors and count.item() == added[0]
        assert torch.equal(z, z2)
    finally:
        gasa.gasa_destroy(ctx)


def test_launch_count_of_graphs_is_this_threads():
    """Launches of other threads while a V-cycle's graph is built are not counted as its own:
    every later V-cycle counts what a hierarchy built alone does."""
    import threading
    import torch
    gasa = _gasa()
    pr = problem("p3_16")

    def per_cycle(busy):
        ctx, _ = gpu_setup("p3_16", keep=False)
        stop = threading.Event()
        n = 4096
        x, y = (torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(2))
        rp, col = to_dev(np.arange(n + 1, dtype=np.int32)), to_dev(np.arange(n, dtype=np.int32))

        def other():
            s = torch.cuda.Stream()
            while not stop.is_set():
                gasa.gasa_bsr_mv(0, n, 1, 1, rp, col, x, x, x, y, s)

        t = threading.Thread(target=other)
        try:
            r = to_dev(pr.rhs)
            z = torch.empty_like(r)
            gasa.gasa_vcycle(ctx, r, z, 1)
            if busy:
                t.start()
            gasa.gasa_vcycle(ctx, r, z, 1)
            if busy:
                stop.set()
                t.join()
            torch.cuda.synchronize()
            k = gasa.gasa_kernel_launches()
            for _ in range(5):
                gasa.gasa_vcycle(ctx, r, z, 1)
            return (gasa.gasa_kernel_launches() - k) / 5
        finally:
            stop.set()
            gasa.gasa_destroy(ctx)

    alone = per_cycle(False)
    for _ in range(3):
        assert per_cycle(True) == alone


@pytest.mark.parametrize("n_agg,bs,size,r,s_next", [
    (160, 4, 3, 80, 6),       # many aggregates: ten pairs a warp, four warps
    (154, 2, 3, 256, 6),      # the most candidates: several rounds of ten pairs
    (170, 5, 4, 37, 5),       # an odd count, a short last chunk of pairs
    (153, 1, 2, 1, 1), (155, 3, 2, 21, 3),
])
def test_tentative_many_aggregates(n_agg, bs, size, r, s_next):
    """More aggregates than SMs, which share them: as the tests of few aggregates."""
    test_tentative_packed_sums(n_agg * size, bs, size, r, s_next)
