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
