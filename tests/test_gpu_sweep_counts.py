"""FP64 V-cycles with other sweep counts than two, cell by cell, and solves whose
coarse levels want a cluster at the same time (-m gpu)."""
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


# on a cluster whole: two shared levels, one, more plane pairs than CTAs; with a
# level of separate kernels above it; with a tiled sweep chosen for that level
@pytest.mark.parametrize("dims,tile", [((32, 24, 16), 0), ((16, 16, 16), 0), ((12, 20, 80), 0), ((64, 64, 64), 0),
                                       ((96, 48, 96), 0), ((64, 64, 64), 32)])
@pytest.mark.parametrize("nu1,nu2", [(0, 1), (1, 0), (0, 2), (2, 0), (1, 1), (3, 2)])
def test_one_preconditioner_application(ibrd, dims, tile, nu1, nu2):
    """The first iterate of the flexible GMRES solve of A c = b (no blobs) is the
    preconditioner's V(b) times a number that minimises the residual: the cycle's
    definition cell by cell, within the V-cycle's 1e-12. No sweep before: the
    residual of both colours; none after: both colours corrected."""
    import torch
    alpha, h, chi = 0.3, 0.7, 1.3
    b = np.random.default_rng(sum(dims)).standard_normal(dims[::-1]) + 0.5
    g = ibrd.Grid(*dims, h=h, chi=chi, alpha=alpha)
    if tile:
        ibrd.ibrd_tune_set(g.handle, 8, 0, *dims, tile, 8)
    c = g.field()
    info = ibrd.ibrd_solve_reaction(g.handle, None, torch.from_numpy(b).cuda(), c,
                                    ibrd.ibrd_default_opts(nu1=nu1, nu2=nu2, mg_cycles=1, max_iter=1, tol=1e-15),
                                    raise_on_error=False)
    assert info["outer_iters"] == 1 and info["vcycles"] == 1
    want = mg.vcycle(b, h, chi, alpha, nu1=nu1, nu2=nu2)
    c = c.cpu().numpy()
    assert rel_max(c * ((c * want).sum() / (c * c).sum()), want) < 1e-12


@pytest.mark.parametrize("dims", [(32, 32, 32), (64, 64, 64)])
def test_solves_side_by_side(ibrd, dims):
    """Sixteen FP64 solves on streams of their own, each wanting its clusters when
    the others do: bit for bit the solves one after the other."""
    import torch
    count, size = 16, dims[0]
    rng = np.random.default_rng(size)
    streams = [torch.cuda.Stream() for _ in range(count)]
    grids = [ibrd.ibrd_grid_create(*dims, stream=s.cuda_stream) for s in streams]
    q = [torch.from_numpy(rng.uniform(0.0, size, (5, 3))).cuda() for _ in grids]
    kappa = [torch.from_numpy(rng.uniform(0.5, 2.0, 5)).cuda() for _ in grids]
    rhs = [torch.from_numpy(rng.standard_normal(dims[::-1]) + 1.0).cuda() for _ in grids]
    torch.cuda.synchronize()
    for g, p in zip(grids, q):
        ibrd.ibrd_set_blobs(g, p)
    out = []
    for threads in (1, 16):
        c = [torch.zeros(dims[::-1], dtype=torch.float64, device="cuda") for _ in grids]
        torch.cuda.synchronize()
        ibrd.ibrd_solve_reaction_batch(grids, kappa, rhs, c, ibrd.ibrd_default_opts(), threads)
        torch.cuda.synchronize()
        out.append(c)
    assert all(torch.equal(a, b) for a, b in zip(*out))
    for g in grids:
        ibrd.ibrd_grid_destroy(g)


# rows above 512 cells, which the row kernels don't serve: the sweep from zero and
# the restriction in one pass over tiles (levels of up to 2^21 cells)
@pytest.mark.parametrize("dims", [(544, 32, 32), (576, 32, 32), (640, 32, 32)])
@pytest.mark.parametrize("nu2,alpha", [(0, 0.1), (1, 0.1), (1, 0.0), (2, 0.1)])
def test_rows_above_512_cells(ibrd, dims, nu2, alpha):
    """FP32 cycles with one sweep before (2e-5, the bound of the other FP32 V-cycle
    tests)."""
    import torch
    b = np.random.default_rng(dims[0]).standard_normal(dims[::-1]).astype(np.float32)
    g = ibrd.Grid(*dims, alpha=alpha)
    x = g.vcycle_f32(torch.from_numpy(b).cuda(), nu1=1, nu2=nu2)
    want = mg.vcycle(b.astype(np.float64), 1.0, 1.0, alpha, nu1=1, nu2=nu2, exact_cells=32768, exact_side=64)
    assert rel_max(x.cpu().numpy().astype(np.float64), want) < 2e-5
