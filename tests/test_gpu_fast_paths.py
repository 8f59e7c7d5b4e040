"""Kernels and launch paths chosen by size, against the general path or the oracle."""
import numpy as np
import pytest

from tests.helpers import gpu_setup, problem, to_dev

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


@pytest.mark.parametrize("n_units,bs,size,r,s_next,rank", [
    (64, 10, 8, 80, 13, 80),      # square blocks
    (48, 13, 8, 40, 17, 40),      # more rows than candidates
    (24, 3, 4, 37, 5, 37),        # fewer rows than candidates
    (40, 1, 1, 16, 1, 16),        # one row per aggregate
    (36, 5, 5, 17, 5, 3),         # rank below the kept count (and a short last aggregate)
    (12, 4, 4, 16, 5, 0),         # zero candidates
    (6, 2, 3, 256, 6, 256),       # the most candidates
    (32, 10, 4, 4, 4, 4),         # the benchmark's r
    (8, 3, 2, 1, 1, 1),           # one candidate
])
def test_tentative_preconditioned(n_units, bs, size, r, s_next, rank):
    """The preconditioned Jacobi kernel against LAPACK's SVD: candidates whose
    singular values fall over ten decades, as relaxed ones do.  A kept vector is exact to
    1e-13 over its relative gap; null vectors are completed as in the oracle."""
    from oracle import gasa_oracle as O
    gasa = _gasa()
    rng = np.random.default_rng(n_units * 100 + r)
    n = n_units * bs
    agg = np.arange(n_units) // size
    n_agg = int(agg.max()) + 1
    B = np.zeros((n, r))
    for J in range(n_agg):
        rows = np.nonzero(np.repeat(agg, bs) == J)[0]
        k = min(rows.size, r, rank)
        if k:
            U = np.linalg.qr(rng.standard_normal((rows.size, k)))[0]
            V = np.linalg.qr(rng.standard_normal((r, k)))[0]
            B[rows] = (U * 10.0 ** (-8.0 * np.arange(k) / k)) @ V.T
    up = np.arange(n_units + 1) * bs
    Tw, _, sv = O.tentative(B, agg, up, n_agg, 3.0, keep=[s_next] * n_agg)
    T, sig = to_dev(np.zeros(n * s_next)), to_dev(np.zeros(n_agg * r))
    gasa.gasa_tentative(n_units, bs, n_agg, to_dev(agg.astype(np.int32)),
                        to_dev(B.ravel(order="F")), r, s_next, T, sig)
    Tg, sg = T.cpu().numpy().reshape(n, s_next), sig.cpu().numpy().reshape(n_agg, r)
    Tw = Tw.tocsr()
    for J in range(n_agg):
        rows = np.nonzero(np.repeat(agg, bs) == J)[0]
        Td = Tw[rows][:, J * s_next:(J + 1) * s_next].toarray()
        s = sv[J]
        if s[0] > 0:
            live = s[:s_next] > 1e-9 * s[0]
            gap = np.min(np.abs(np.diff(s[: min(len(s), s_next + 1)])[:max(1, live.sum())])) / s[0] \
                if len(s) > 1 else 1.0
            assert np.max(np.abs(sg[J, :len(s)] - s)) <= 1e-14 * len(rows) * s[0]
        else:
            gap = 1.0
        assert np.max(np.abs(Tg[rows] - Td)) <= max(1e-12, 1e-13 / max(gap, 1e-12)), J
        assert np.max(np.abs(Tg[rows].T @ Tg[rows] - np.eye(s_next))) <= 1e-13 * len(rows)
