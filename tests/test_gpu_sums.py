"""What the streaming sums keep of their terms, through the launchers (-m gpu)."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

P, Z, D = ctypes.c_void_p, ctypes.c_size_t, ctypes.c_double


@pytest.fixture(scope="module")
def lib():
    import paper_1306_3159_gb300 as p
    return p.load_library()


def launcher(lib, name, *args):
    """A launcher of the library (C++ linkage; the last two arguments are its
    stream and its ticket, none here)."""
    import torch
    f = getattr(lib, name)
    f.argtypes, f.restype = list(args) + [P, P], None

    def call(*values):
        f(*[v.data_ptr() if isinstance(v, torch.Tensor) else v for v in values],
          torch.cuda.current_stream().cuda_stream, None)
    return call


def scratch():
    import torch
    return torch.zeros(2 * 608, dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")


# a few entries; fields summed in FP64 alone, up to the last such size; the first
# with runs, one and several vectors a thread, remainders
@pytest.mark.parametrize("n", [1, 7, 1000, 262144, 622591, 622592, 1000003, 4000002])
def test_runs_of_the_fp32_sum(lib, n):
    """FP32 entries are added in FP32 over four of them at most (none in fields
    below 622592): sums of four whole numbers below 2^22 (of one below 2^24) are
    exact, longer ones are not, so the total is exact."""
    import torch
    x = np.random.default_rng(n).integers(1, 1 << (24 if n < 622592 else 22), n)
    partial, out = scratch()
    launcher(lib, "_ZN4ibrd10launch_sumIfEEvPKT_mPdS4_dP11CUstream_stPj", P, Z, P, P, D)(
        torch.from_numpy(x.astype(np.float32)).cuda(), n, partial, out, 1.0)
    assert out.item() == float(x.sum())


@pytest.mark.parametrize("bits", [32, 64])
@pytest.mark.parametrize("n,start", [(1, 1), (2, 3), (3, 2), (1000, 1), (1000003, 2), (1000001, 3), (1 << 25, 1)])
def test_sum_off_a_boundary(lib, n, start, bits):
    """Fields that start anywhere are summed whole (below 2^22: as above) and, being
    bound by their one read, in the time of an aligned one, within a third."""
    import torch
    x = torch.randint(1, 1 << 22, (n + 4,), device="cuda")
    total = float(x[start:start + n].sum())
    x = x.to(torch.float32 if bits == 32 else torch.float64)
    partial, out = scratch()
    kind = "f" if bits == 32 else "d"
    add = launcher(lib, f"_ZN4ibrd10launch_sumI{kind}EEvPKT_mPdS4_dP11CUstream_stPj", P, Z, P, P, D)
    add(x[start:], n, partial, out, 1.0)
    assert out.item() == total
    if n < 1 << 25:
        return

    def time(field):
        best = 1e9
        for _ in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(4):
                add(field, n, partial, out, 1.0)
            e1.record()
            e1.synchronize()
            best = min(best, e0.elapsed_time(e1))
        return best

    assert time(x[start:]) < 4 / 3 * time(x)


# start 1: no 16-byte alignment
@pytest.mark.parametrize("n", [1, 7, 1000, 100003, 262145])
@pytest.mark.parametrize("start", [0, 1])
def test_terms_of_the_fp32_partial_sums(lib, n, start):
    """Squares, products and converted entries are added in FP32 over a warp of a
    small field's threads, one term each: 32 whole numbers of at most 700 x 700
    (of one below 2^24) are exact, 64 and more are not, so the totals are exact."""
    import torch
    rng = np.random.default_rng(n + start)
    a, b = (rng.integers(1, 701, n + start).astype(np.float64) for _ in (0, 1))
    x, y = torch.from_numpy(a).cuda()[start:], torch.empty(n + start, dtype=torch.float32, device="cuda")[start:]
    partial, out = scratch()
    launcher(lib, "_ZN4ibrd17launch_convert_sqEPKdPfmdPdS3_P11CUstream_stPj", P, P, Z, D, P, P)(
        x, y, n, 1.0, partial, out)
    assert out.item() == (a[start:] ** 2).sum() and torch.equal(y.double(), x)
    if n <= 155648:
        if start:  # (aligned, a thread's sum takes the four products of its vector)
            f, g = (torch.from_numpy(v).cuda().float()[start:] for v in (a, b))
            launcher(lib, "_ZN4ibrd10launch_dotIfEEvPKT_S3_mPdS4_dP11CUstream_stPj", P, P, Z, P, P, D)(
                f, g, n, partial, out, 1.0)
            assert out.item() == (a[start:] * b[start:]).sum()
        c = rng.integers(1, 1 << 24, n + start).astype(np.float64)
        both = torch.zeros(2, dtype=torch.float64, device="cuda")
        launcher(lib, "_ZN4ibrd18launch_convert_sumIdfEEvPKT_PT0_mPdS6_S6_P11CUstream_stPj", P, P, Z, P, P, P)(
            torch.from_numpy(c).cuda()[start:], y, n, partial, both, both[1:])
        assert both[0].item() == both[1].item() == c[start:].sum()
