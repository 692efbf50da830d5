"""The FP64 V-cycle's coarse end on a thread block cluster (-m gpu)."""
import numpy as np
import pytest

from oracle import multigrid as mg
from tests.gpu_util import rel_max

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ibrd():
    import paper_1306_3159_gb300 as p
    p.load_library()
    return p


# Grids that the cluster kernel takes whole: one and two shared levels; fewer
# plane pairs than CTAs, as many, more (uneven parts); two pairs (the
# neighbours above and below are the same CTA); sides that are no powers of two;
# and ones with levels above it (on separate kernels).
BOXES = [(16, 16, 16), (32, 32, 32), (24, 24, 24), (40, 16, 36), (12, 20, 80), (24, 16, 4), (32, 48, 16), (96, 96, 48),
         (64, 64, 64)]


@pytest.mark.parametrize("dims", BOXES)
@pytest.mark.parametrize("alpha,zero", [(0.0, True), (0.3, False)])
def test_coarse_end_on_a_cluster(ibrd, dims, alpha, zero):
    """The V-cycle against its definition, singular and shifted, from zero and
    from a guess, within the V-cycle's 1e-12."""
    import torch
    rng = np.random.default_rng(sum(dims))
    b, x0 = rng.standard_normal(dims[::-1]) + 0.5, rng.standard_normal(dims[::-1])
    g = ibrd.Grid(*dims, h=0.7, chi=1.3, alpha=alpha)
    x = g.vcycle(torch.from_numpy(b).cuda(), torch.from_numpy(x0).cuda(), zero)
    want = mg.vcycle(b, 0.7, 1.3, alpha, x0=None if zero else x0)
    assert rel_max(x.cpu().numpy(), want) < 1e-12


@pytest.mark.parametrize("nu1,nu2", [(0, 1), (1, 0), (1, 1), (3, 2)])
def test_sweep_counts_on_a_cluster(ibrd, nu1, nu2):
    """Preconditioners with other sweep counts (no sweep before: the residual of
    both colours; none after: both colours corrected) still solve the system."""
    import torch
    from oracle import direct
    from synthetic import loguniform_rates, rsa_positions
    dims = (32, 24, 16)
    q, kappa = rsa_positions(12, dims, 1.0, 3.0, 3), loguniform_rates(12, 0.1, 10.0, 4)
    rhs = np.random.default_rng(5).standard_normal(dims[::-1]) + 1.0
    g = ibrd.Grid(*dims)
    g.set_blobs(torch.from_numpy(q).cuda())
    c, info = g.solve_reaction(torch.from_numpy(kappa).cuda(), torch.from_numpy(rhs).cuda(), tol=1e-11, nu1=nu1,
                               nu2=nu2, max_iter=300)
    want, _, _ = direct.solve_reaction(q, kappa, rhs, 1.0, 1.0, 0.0)
    assert rel_max(c.cpu().numpy(), want) < 1e-9
