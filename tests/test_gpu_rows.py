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
