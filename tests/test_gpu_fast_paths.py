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
