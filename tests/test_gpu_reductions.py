"""Streaming reductions at the edges of their forms, through the calls that use
them (-m gpu)."""
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


# 315 cells (less than one block's entries, an odd count) up to several blocks
# with a remainder
@pytest.mark.parametrize("dims", [(5, 7, 9), (10, 14, 6), (64, 48, 40)])
@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("start", [0, 1])
def test_mean_projection(ibrd, dims, bits, start):
    """The singular V-cycle sums its right-hand side and subtracts the mean of
    its result: whole vectors, remainders, and fields that start one value into
    an allocation (no 16-byte alignment). Bounds: those of the V-cycle tests
    (FP32 2e-5, FP64 1e-12); the mean of the result is that of rounding."""
    import torch
    kind = torch.float32 if bits == 32 else torch.float64
    n = dims[0] * dims[1] * dims[2]
    rng = np.random.default_rng(n + bits)
    b = (rng.standard_normal(dims[::-1]) + 3.0).astype(np.float32 if bits == 32 else np.float64)
    g = ibrd.Grid(*dims)
    bd, x = (torch.zeros(n + start, dtype=kind, device="cuda")[start:].view(dims[::-1]) for _ in (0, 1))
    bd.copy_(torch.from_numpy(b))
    (g.vcycle_f32 if bits == 32 else g.vcycle)(bd, x)
    exact = dict(exact_cells=32768, exact_side=64) if bits == 32 else {}
    want = mg.vcycle(b.astype(np.float64), 1.0, 1.0, 0.0, **exact)
    got = x.cpu().numpy().astype(np.float64)
    bound = 2e-5 if bits == 32 else 1e-12
    assert rel_max(got, want) < bound
    assert abs(got.mean()) < bound * np.abs(want).max()


@pytest.mark.parametrize("precision,tol", [(0, 1e-11), (2, 1e-11)])
@pytest.mark.parametrize("eta", [0.0, 0.70710678118654752, 1.0])
def test_orthogonalisation_over_groups(ibrd, precision, tol, eta):
    """More Krylov vectors than one projection launch takes (8), without, with
    a conditional and with an unconditional second pass: the solution is the
    direct solver's (the solve parity bound 1e-9 at this tolerance) and the
    passes are counted."""
    import torch
    from oracle import direct
    from synthetic import loguniform_rates, rsa_positions
    dims = (32, 16, 24)
    q, kappa = rsa_positions(30, dims, 1.0, 3.0, 7), 10.0 * loguniform_rates(30, 0.1, 10.0, 8)
    rhs = np.random.default_rng(9).standard_normal(dims[::-1]) + 1.0
    g = ibrd.Grid(*dims, alpha=0.01, precision=precision)
    g.set_blobs(torch.from_numpy(q).cuda())
    c, info = g.solve_reaction(torch.from_numpy(kappa).cuda(), torch.from_numpy(rhs).cuda(), tol=tol, reorth_eta=eta,
                               nu1=1, nu2=1, inner_tol=1e-6, max_iter=400)
    want, _, _ = direct.solve_reaction(q, kappa, rhs, 1.0, 1.0, 0.01)
    assert rel_max(c.cpu().numpy(), want) < 1e-9
    assert info["outer_iters"] > 8
    if eta != 0.70710678118654752:
        assert info["reorths"] == (info["outer_iters"] if eta == 1.0 else 0)
