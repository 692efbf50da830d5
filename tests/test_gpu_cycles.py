"""The launches of FP32 V-cycles whose passes are not all fused (-m gpu)."""
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


@pytest.mark.parametrize("dims", [(128, 64, 32), (64, 64, 64), (96, 64, 32)])
def test_passes_outside_the_fused_sweep(ibrd, dims):
    """One level above the exact one. With a row-resident sweep after it, the coarse
    correction rides on that sweep: as many launches with it as without a
    sweep (the correction alone), and one more where the two are kept
    apart or a tiled sweep is chosen; no pass that only rewrites the field. The
    result is the definition's (2e-5, the bound of the other FP32 V-cycle tests)."""
    import torch
    rng = np.random.default_rng(dims[0])
    b = rng.standard_normal(dims[::-1]).astype(np.float32)
    bd = torch.from_numpy(b).cuda()

    def launches(nu2, shape=None):
        g = ibrd.Grid(*dims, alpha=0.1)
        if shape:
            ibrd.ibrd_tune_set(g.handle, 4, shape[0], *dims, shape[1], 0)
        g.vcycle_f32(bd, nu1=1, nu2=nu2)  # (lays out what a handle keeps)
        ibrd.ibrd_profile_read(g.handle)
        x = g.vcycle_f32(bd, nu1=1, nu2=nu2)
        n = ibrd.ibrd_profile_read(g.handle)["launches"]
        want = mg.vcycle(b.astype(np.float64), 1.0, 1.0, 0.1, nu1=1, nu2=nu2, exact_cells=32768, exact_side=64)
        assert rel_max(x.cpu().numpy().astype(np.float64), want) < 2e-5
        return n

    fused = launches(1)
    assert launches(0) == fused
    assert launches(1, (2, 1)) == fused + 1
    assert launches(1, (0, 32)) == fused + 1
