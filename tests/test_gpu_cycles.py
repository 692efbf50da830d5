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


# 2048 rows and more, where the row-resident sweeps of a full field are the built-in
# ones: part of one slot, one, part of two, two; two warps with part of two
# slots (plain sweep only) and with two
@pytest.mark.parametrize("dims", [(96, 32, 64), (128, 64, 32), (160, 64, 32), (224, 32, 64), (256, 64, 32),
                                  (288, 64, 32), (448, 32, 64), (512, 64, 32), (64, 48, 32), (32, 64, 64)])
@pytest.mark.parametrize("nu,alpha,zero", [(2, 0.1, True), (1, 0.0, False), (2, 0.0, True)])
def test_sweeps_of_a_full_field(ibrd, dims, nu, alpha, zero):
    """Two sweeps on each side, or a guess: the cycles whose sweeps read a full
    field (2e-5 of the definition, the bound of the other FP32 V-cycle tests)."""
    import torch
    rng = np.random.default_rng(dims[0] + nu)
    b, x0 = (rng.standard_normal(dims[::-1]).astype(np.float32) for _ in (0, 1))
    g = ibrd.Grid(*dims, alpha=alpha)
    x = g.vcycle_f32(torch.from_numpy(b).cuda(), torch.from_numpy(x0).cuda(), zero, nu1=nu, nu2=nu)
    want = mg.vcycle(b.astype(np.float64), 1.0, 1.0, alpha, x0=None if zero else x0.astype(np.float64), nu1=nu,
                     nu2=nu, exact_cells=32768, exact_side=64)
    assert rel_max(x.cpu().numpy().astype(np.float64), want) < 2e-5


@pytest.mark.parametrize("dims", [(32, 256, 256), (64, 512, 512), (384, 16, 16), (96, 16, 16), (256, 256, 64)])
def test_built_in_sweeps_are_not_slower(ibrd, dims):
    """The built-in shapes of a cycle with two sweeps on each side against tiled
    sweeps on its finest level (5 % for the clock)."""
    import torch
    width = 64 if dims[0] % 64 == 0 else 32
    fields = [torch.randn(dims[::-1], device="cuda") for _ in range(3)]
    handles = [ibrd.Grid(*dims, alpha=0.1) for _ in (0, 1)]
    ibrd.ibrd_tune_set(handles[1].handle, 4, 0, *dims, width, 0)
    best = [1e9, 1e9]
    for k in range(24):
        g = handles[k % 2]
        for warm in (True, False):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(2 if warm else 12):
                g.vcycle_f32(fields[0], fields[1], nu1=2, nu2=2)
                g.vcycle_f32(fields[1], fields[2], nu1=2, nu2=2)
            e1.record()
            e1.synchronize()
        best[k % 2] = min(best[k % 2], e0.elapsed_time(e1))
    assert best[0] < 1.05 * best[1]


@pytest.mark.parametrize("dims", [(64, 256, 256), (96, 64, 64), (160, 32, 32), (128, 64, 32)])
def test_tuning_keeps_the_fused_cycle(ibrd, dims):
    """Tuned shapes change depths on levels the row-resident kernels serve, not the
    kernels: the cycle has as many launches as before."""
    import torch
    b = torch.randn(dims[::-1], device="cuda")
    g = ibrd.Grid(*dims, alpha=0.1)

    def launches():
        g.vcycle_f32(b, nu1=1, nu2=1)
        ibrd.ibrd_profile_read(g.handle)
        g.vcycle_f32(b, nu1=1, nu2=1)
        return ibrd.ibrd_profile_read(g.handle)["launches"]

    before = launches()
    for r in ibrd.ibrd_autotune(g.handle, 1, retune=True):
        if r["kind"] == 0 and r["nx"] % 32 == 0 and r["nx"] <= 512 and r["ny"] % 8 == 0:
            assert r["tx"] in (0, r["nx"] if r["nx"] in (128, 256) else 0)
    assert launches() == before


# the packed black cells' kernels where two warps per row begin (1024 rows), and
# one tile of rows
@pytest.mark.parametrize("dims", [(288, 32, 32), (320, 64, 32), (448, 32, 64), (512, 32, 32), (96, 8, 8),
                                  (256, 8, 16)])
@pytest.mark.parametrize("nu2,alpha,zc", [(0, 0.1, 0), (1, 0.0, 0), (1, 0.1, 2), (1, 0.0, 6), (2, 0.1, 0)])
def test_packed_cells_and_the_correction_apart(ibrd, dims, nu2, alpha, zc):
    """One sweep before: the cycle's definition (2e-5), and bit for bit the one with
    the correction kept apart."""
    import torch
    b = np.random.default_rng(dims[0] + zc).standard_normal(dims[::-1]).astype(np.float32)
    out = []
    for apart in (0, 1):
        g = ibrd.Grid(*dims, alpha=alpha)
        if zc:
            ibrd.ibrd_tune_set(g.handle, 4, 0, *dims, 0, zc)
        ibrd.ibrd_tune_set(g.handle, 4, 2, *dims, apart, 0)
        out.append(g.vcycle_f32(torch.from_numpy(b).cuda(), nu1=1, nu2=nu2).cpu().numpy())
    assert np.array_equal(out[0], out[1])
    want = mg.vcycle(b.astype(np.float64), 1.0, 1.0, alpha, nu1=1, nu2=nu2, exact_cells=32768, exact_side=64)
    assert rel_max(out[0].astype(np.float64), want) < 2e-5
