"""Calls that run out of device memory leave handles that can be used (-m gpu)."""
import contextlib

import numpy as np
import pytest

from oracle import operators as op
from tests.gpu_util import dev, host, rel_max

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def ibrd():
    import paper_1306_3159_gb300 as p
    p.load_library()
    return p


@contextlib.contextmanager
def only(megabytes):
    """Takes the device's free memory but for about that many MB."""
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    ballast = torch.empty(torch.cuda.mem_get_info()[0] - megabytes * MB, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del ballast
        torch.cuda.empty_cache()


def test_blobs_that_do_not_fit(ibrd):
    """A blob takes 216 bytes of positions, indices and weights and 64 and more of
    lists: with 500 MB free, two million blobs get the first (432 MB) and not
    the second. The call says so, the handle then has no blobs (sums over none
    are zero), and takes new ones."""
    import torch
    dims = (64, 32, 40)
    rng = np.random.default_rng(1)
    size = np.array(dims, dtype=float)
    g = ibrd.Grid(*dims)
    q = rng.uniform(0.0, 1.0, (50, 3)) * size
    lam = rng.uniform(0.5, 1.5, 50)
    c = rng.standard_normal(dims[::-1])
    many = torch.rand(2_000_000, 3, dtype=torch.float64, device="cuda")
    cd, out, back = dev(c), g.field(), torch.full((2_000_000,), 7.0, dtype=torch.float64, device="cuda")
    ld = dev(lam)
    g.set_blobs(dev(q))
    g.interp(cd, back)  # (the kernels are loaded)
    g.spread(ld, out)
    with only(500):
        with pytest.raises(ibrd.IbrdError) as e:
            g.set_blobs(many)
        assert "OOM" in str(e.value) and g.n_blobs == 0
        back.fill_(7.0)
        g.interp(cd, back)
        g.spread(ld, out)
    assert bool((back == 7.0).all()) and not bool(out.any())
    g.set_blobs(dev(q))
    assert rel_max(host(g.spread(ld)), op.spread(lam, q, dims, 1.0, 4)) < 1e-13


def test_refused_blobs_keep_the_old_ones(ibrd):
    """A position that is not finite is refused, and the blobs of before stay."""
    import torch
    dims = (16, 16, 16)
    rng = np.random.default_rng(2)
    g = ibrd.Grid(*dims)
    q, c = rng.uniform(0.0, 16.0, (9, 3)), dev(rng.standard_normal(dims[::-1]))
    g.set_blobs(dev(q))
    want = host(g.interp(c))
    bad = rng.uniform(0.0, 16.0, (3, 3))
    bad[1, 2] = np.inf
    with pytest.raises(ibrd.IbrdError):
        g.set_blobs(dev(bad))
    assert g.n_blobs == 9
    assert torch.equal(g.interp(c).cpu(), torch.from_numpy(want))


def test_model_that_does_not_fit(ibrd):
    """A blob takes about 8 KB here: 200 000 blobs do not fit 500
    MB. A smaller call on the same model then allocates what it needs."""
    import torch
    q = torch.rand(200_000, 3, dtype=torch.float64, device="cuda") * 400.0
    few = torch.rand(40, 3, dtype=torch.float64, device="cuda") * 40.0
    lam = torch.rand(40, dtype=torch.float64, device="cuda") + 0.5
    m = ibrd.GNN(6.0, 64)
    m.init_params(3)
    want, grad = m.predict(few, (40.0,) * 3, 40.0), m.loss_grad(few, (40.0,) * 3, lam)[1]
    out = torch.empty(200_000, dtype=torch.float64, device="cuda")
    with only(500):
        with pytest.raises(ibrd.IbrdError) as e:
            m.predict(q, (400.0,) * 3, 1.0, out)
        assert "OOM" in str(e.value)
    assert torch.equal(m.predict(few, (40.0,) * 3, 40.0), want)
    assert torch.equal(m.loss_grad(few, (40.0,) * 3, lam)[1], grad)
