"""Blob lists at the edges of their tiles (-m gpu)."""
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


# one tile smaller than a support's wrap; last tiles of one and two cells (three
# tiles under one support); more tiles than one scan block takes
@pytest.mark.parametrize("dims", [(4, 4, 4), (9, 7, 7), (18, 10, 10), (256, 256, 64)])
@pytest.mark.parametrize("kernel", [3, 4])
def test_lists_follow_the_blobs(ibrd, dims, kernel):
    """Spreading after one set of blobs has replaced another: a
    few, many in one tile (several passes of a warp over the tile's list),
    supports across every face, none, one. Weights and multipliers are positive,
    so a cell's sum of m products rounds to within (m + 8) 2^-53 of itself:
    1e-13 for the m <= 300 here."""
    rng = np.random.default_rng(sum(dims) + kernel)
    size = np.array(dims, dtype=float)
    g = ibrd.Grid(*dims, kernel=kernel)
    for n, place in [(5, "any"), (300, "corner"), (33, "face"), (0, "any"), (1, "face"), (200, "any")]:
        q = rng.uniform(-1.0, 2.0, (n, 3)) * size
        if place == "corner":
            q = rng.uniform(0.0, 1.5, (n, 3))
        elif place == "face":
            q = rng.integers(0, 2, (n, 3)) * size + rng.uniform(-2.5, 2.5, (n, 3))
        lam = rng.uniform(0.5, 1.5, n)
        g.set_blobs(dev(q))
        got = host(g.spread(dev(lam)))
        if n == 0:
            assert not got.any()
            continue
        qw = q - np.floor(q / size) * size
        assert rel_max(got, op.spread(lam, qw, dims, 1.0, kernel)) < 1e-13
