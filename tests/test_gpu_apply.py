"""The operator at the edges of its blocks (-m gpu)."""
import numpy as np
import pytest

from oracle import operators as op
from tests.gpu_util import dev, host, rel_max

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ibrd():
    import paper_1306_3159_gb300 as p
    p.load_library()
    return p


# fewer cells than one block; odd sides; a remainder in x, in y and in the planes
# per block (1, 2 and more of them)
@pytest.mark.parametrize("dims", [(4, 4, 4), (5, 7, 9), (9, 7, 7), (36, 20, 28), (72, 40, 56)])
@pytest.mark.parametrize("alpha", [0.0, 0.3])
def test_apply_and_residual(ibrd, dims, alpha):
    """y = A x and b - A x. A cell's 8 roundings are each within 2^-53 of terms
    that sum to 6.3 |x| + 6 max|x| <= 12.3 max|x|, the oracle's as many: 3e-14 for
    |x| <= 5 and results of at least 8 at their largest, relative to those 4e-15;
    the bound is 1e-14."""
    rng = np.random.default_rng(sum(dims))
    c, b = rng.standard_normal(dims[::-1]), rng.standard_normal(dims[::-1])
    g = ibrd.Grid(*dims, alpha=alpha)
    want = op.apply_A(c, 1.0, 1.0, alpha)
    assert rel_max(host(g.apply_L(dev(c))), want) < 1e-14
    assert rel_max(host(g.residual(dev(b), dev(c))), b - want) < 1e-14
