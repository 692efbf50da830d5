"""The row-resident FP32 kernels at the edges of their forms (-m gpu)."""
import numpy as np
import pytest

from tests.gpu_util import rel_max
from oracle import multigrid as mg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ibrd():
    import paper_1306_3159_gb300 as p
    p.load_library()
    return p


# (nu1, nu2): every way the pre-smoothed black cells are handed on -- unpacked
# when no sweep follows, read by the fused prolongation when one does, in one
# or the other of the level's two fields by the parity of the sweeps -- and the
# cycles that keep the full field.
@pytest.mark.parametrize("nu1,nu2", [(1, 0), (1, 1), (1, 3), (2, 2), (3, 1), (0, 1), (0, 2)])
@pytest.mark.parametrize("dims", [(128, 8, 4), (256, 24, 16), (256, 32, 64)])
def test_black_cells_between_half_cycles(ibrd, dims, nu1, nu2):
    """The FP32 V-cycle from zero against its definition. Bound: a V-cycle of a
    few sweeps is a short chain of FP32 operations with weights below one, so
    its error stays within a few hundred units of 2^-24 of the largest value."""
    import torch
    rng = np.random.default_rng(11 + nu1 + 5 * nu2)
    b = rng.standard_normal(dims[::-1]).astype(np.float32)
    g = ibrd.Grid(*dims, alpha=0.1)
    x = g.vcycle_f32(torch.from_numpy(b).cuda(), nu1=nu1, nu2=nu2)
    want = mg.vcycle(b.astype(np.float64), 1.0, 1.0, 0.1, nu1=nu1, nu2=nu2, exact_cells=32768, exact_side=64)
    assert rel_max(x.cpu().numpy().astype(np.float64), want) < 2e-5


# Row lengths by how a warp holds them: part of one slot (32, 64, 96), one slot
# (128), part of two (160, 192, 224), two (256), two warps with part of two
# slots each (288, 320, 448) and with two full ones (512).
ROW_BOXES = [(32, 72, 16), (64, 72, 16), (96, 8, 4), (96, 40, 16), (128, 8, 4), (160, 16, 8), (192, 16, 8),
             (224, 16, 8), (256, 24, 16), (288, 32, 16), (320, 32, 16), (448, 32, 16), (512, 32, 16)]


@pytest.mark.parametrize("dims", ROW_BOXES)
@pytest.mark.parametrize("nu1,nu2,alpha,zero", [(1, 1, 0.0, True), (2, 2, 0.1, True), (1, 1, 0.1, False)])
def test_row_lengths(ibrd, dims, nu1, nu2, alpha, zero):
    """Every row length the kernels serve against the V-cycle's definition (the
    same bound), from zero and from a guess; alpha = 0 also checks the per-CTA
    sums that feed the mean projection."""
    import torch
    rng = np.random.default_rng(dims[0] + nu1)
    b = rng.standard_normal(dims[::-1]).astype(np.float32)
    x0 = rng.standard_normal(dims[::-1]).astype(np.float32)
    g = ibrd.Grid(*dims, alpha=alpha)
    x = g.vcycle_f32(torch.from_numpy(b).cuda(), torch.from_numpy(x0).cuda(), zero, nu1=nu1, nu2=nu2)
    want = mg.vcycle(b.astype(np.float64), 1.0, 1.0, alpha, x0=None if zero else x0.astype(np.float64), nu1=nu1,
                     nu2=nu2, exact_cells=32768, exact_side=64)
    assert rel_max(x.cpu().numpy().astype(np.float64), want) < 2e-5


@pytest.mark.parametrize("dims", [(96, 8, 4), (160, 16, 8), (320, 32, 16), (512, 32, 16)])
@pytest.mark.parametrize("zc", [0, 2, 6])
def test_fused_prolongation_of_other_row_lengths(ibrd, dims, zc):
    """The fused prolongation equals, bit for bit, the cycle with it kept
    separate, where lanes are idle or two warps share a row."""
    import torch
    rng = np.random.default_rng(dims[0] + zc)
    b = torch.from_numpy(rng.standard_normal(dims[::-1]).astype(np.float32)).cuda()
    out = []
    for separate in (0, 1):
        g = ibrd.Grid(*dims)
        if zc:
            ibrd.ibrd_tune_set(g.handle, 4, 0, *dims, 0, zc)
        ibrd.ibrd_tune_set(g.handle, 4, 2, *dims, separate, 0)
        out.append(g.vcycle_f32(b, nu1=1, nu2=1))
    assert torch.equal(out[0], out[1])
