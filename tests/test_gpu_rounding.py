"""What rounding leaves in an FP64 V-cycle, against longer arithmetic (-m gpu)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

L = np.longdouble


@pytest.fixture(scope="module")
def ibrd():
    import paper_1306_3159_gb300 as p
    p.load_library()
    return p


def _neighbours(x):
    return sum(np.roll(x, s, a) for a in range(3) for s in (1, -1))


def _solve(A, b):
    """A x = b by elimination (a handful of unknowns, diagonally dominant)."""
    M = np.concatenate([A, b[:, None]], axis=1)
    for i in range(len(b)):
        M[i] /= M[i, i]
        for j in range(len(b)):
            if j != i:
                M[j] -= M[j, i] * M[i]
    return M[:, -1]


def _prolong(e):
    for a in range(3):
        out = np.empty([2 * n if k == a else n for k, n in enumerate(e.shape)], dtype=L)
        for odd in (0, 1):
            at = [slice(None)] * 3
            at[a] = slice(odd, None, 2)
            out[tuple(at)] = L(3) / 4 * e + L(1) / 4 * np.roll(e, -1 if odd else 1, a)
        e = out
    return e


def _vcycle(b, h, chi, alpha):
    """The definition (alpha > 0, two sweeps on each side, from zero) in the longest
    floating point type there is."""
    off, diag = chi / (h * h), alpha + 6 * chi / (h * h)
    if not all(n % 2 == 0 and n >= 4 for n in b.shape):
        A = np.zeros((b.size, b.size), dtype=L)
        for k in range(b.size):
            e = np.zeros(b.size, dtype=L)
            e[k] = 1
            e = e.reshape(b.shape)
            A[:, k] = (diag * e - off * _neighbours(e)).ravel()
        return _solve(A, b.ravel()).reshape(b.shape)
    k, j, i = np.meshgrid(*[np.arange(n) for n in b.shape], indexing="ij")
    red = (i + j + k) % 2 == 0

    def sweeps(x):
        for colour in (red, ~red) * 2:
            x = np.where(colour, (b + off * _neighbours(x)) / diag, x)
        return x

    x = sweeps(np.zeros_like(b))
    r = b - (diag * x - off * _neighbours(x))
    nz, ny, nx = b.shape
    r = r.reshape(nz // 2, 2, ny // 2, 2, nx // 2, 2).mean(axis=(1, 3, 5))
    return sweeps(x + _prolong(_vcycle(r, 2 * h, chi, alpha)))


# chi and alpha: alpha + 6 chi / h^2 is a double on every level, the double next to
# 1 / diag is within 0.12 x 2^-53 of it, and the one next to chi / h^2 times that
# one is not
CASES = [((32, 32, 32), 1.75, 0.52734375), ((32, 32, 32), 13.0, 3.802734375), ((32, 32, 32), 3.0, 1.3046875),
         ((64, 64, 64), 13.0, 3.802734375), ((48, 32, 64), 1.75, 0.52734375)]


@pytest.mark.parametrize("dims,chi,alpha", CASES)
def test_sweeps_do_not_scale_smooth_fields(ibrd, dims, chi, alpha):
    """Smooth fields pass through four half-sweeps per side and level almost
    unchanged, so that a relative error common to all cells of a sweep adds up.
    With 1 / diag rounded once it is 0.12 x 2^-53 here, at most half of 2^-53 in
    the last four; a cell's own last two roundings are 0.6 x 2^-53 rms each, and
    what the neighbours bring is averaged. In sum below 2 x 2^-53 rms."""
    import torch
    rng = np.random.default_rng(1)
    b = rng.standard_normal(dims[::-1])
    for a, n in enumerate(dims[::-1]):
        wave = 3.0 * np.sin(np.arange(n) * 2.0 * np.pi / n + rng.uniform(0.0, 6.0))
        b += wave.reshape([-1 if k == a else 1 for k in range(3)])
    g = ibrd.Grid(*dims, chi=chi, alpha=alpha)
    x = g.vcycle(torch.from_numpy(b).cuda()).cpu().numpy()
    want = _vcycle(b.astype(L), L(1), L(chi), L(alpha))
    if np.finfo(L).nmant < 60:
        pytest.skip("no longer floating point type than double here")
    err = x.astype(L) - want
    assert float(np.sqrt((err * err).mean() / (want * want).mean())) < 2.0 * 2.0 ** -53
