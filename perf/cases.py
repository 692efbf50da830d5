"""The work that users of this library have it do, as measurable cases.

A case is one call sequence through the package's public entry points: whole
solves (one small problem, a medium one at the library's defaults, the two
solves of one large suspension, a batch of realisations), the multigrid V-cycle
alone in both precisions, the coupled operator and its residual, a move of the
blobs, and the learned multiplier predictor's inference and training gradient.
Grid sides are odd or even multiples of powers of two (the multigrid hierarchy
halves them), boxes are cubes or not, blob counts are arbitrary.

``exact`` states what each call returns in plain 64-bit torch: Fourier
transforms in place of multigrid, conjugate gradients on the blob unknowns in
place of FGMRES, and the definitions of the V-cycle, the kernels and the
network written out.
"""
import math

import numpy as np
import torch

import paper_1306_3159_gb300 as ibrd

# Solver settings of this library's benchmark for the mixed-precision solves.
REACTION = dict(mg_cycles=1, nu1=1, nu2=1, reorth_eta=0.0, inner_tol=1e-3)
SADDLE = dict(schur_inner=3, mg_cycles=1, nu1=1, nu2=1, reorth_eta=0.0, inner_tol=1e-4, lambda_guess=1,
              warm_cycles=1, precond=3)
# Relative residual of the solves: tight enough that a solution is set by the
# system and not by where the iteration stopped, and above the rounding floor
# of a few blobs in a large box (where c carries a large constant).
TOL = 5e-10
CUTOFF, NEIGHBOURS, BASES, WIDTH, LAYERS = 24.0, 256, 16, 64, 3


def listed():
    return [
        # the smallest whole call: one blob in a small box, library defaults
        # (a sweep over positions or box sizes makes thousands of these)
        dict(name="saddle_32_one_blob", kind="saddle", nx=32, ny=32, nz=32, blobs=1, alpha=0.0),
        # a medium problem as a new user writes it: FP64, every option at its default
        dict(name="reaction_96_defaults", kind="reaction", nx=96, ny=96, nz=96, blobs=512, alpha=0.0),
        # one configuration of a large suspension: blobs set, both solves,
        # mixed precision, each on its own handle and stream
        dict(name="step_256", kind="step", nx=256, ny=256, nz=256, blobs=4096),
        # disordered realisations of uneven size, solved together
        dict(name="batch_of_12", kind="batch", count=12, largest=160, most=2000),
        # the preconditioner of the mixed-precision solves, as they call it
        dict(name="vcycle_f32_256", kind="vcycle", nx=256, ny=256, nz=256, bits=32, nu1=1, nu2=1, alpha=0.0),
        # the same on the largest box
        dict(name="vcycle_f32_512", kind="vcycle", nx=512, ny=512, nz=512, bits=32, nu1=1, nu2=1, alpha=0.0),
        # an implicit time step's Helmholtz V-cycle in a box that is no cube and no power of two
        dict(name="vcycle_f32_box", kind="vcycle", nx=160, ny=96, nz=224, bits=32, nu1=2, nu2=2, alpha=0.1),
        # the FP64 V-cycle (the default precision's preconditioner)
        dict(name="vcycle_f64_128", kind="vcycle", nx=128, ny=128, nz=128, bits=64, nu1=2, nu2=2, alpha=0.0),
        # the coupled operator A c + S (kappa J c), as in an explicit step or a user's own iteration
        dict(name="operator_256", kind="operator", nx=256, ny=256, nz=256, blobs=4096, alpha=0.0, form="apply"),
        # the blobs moved: set up, source spread, concentrations read back
        dict(name="blobs_256", kind="blobs", nx=256, ny=256, nz=256, blobs=4096, width=4),
        # inference of the learned multipliers on a large suspension
        dict(name="predict_4096", kind="predict", side=256, blobs=4096),
        # one training configuration's loss and gradient
        dict(name="train_1000", kind="train", side=128, blobs=1000),
    ]


def _between(rng, lo, hi):
    """A whole number, its logarithm uniform over [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _box(rng, lo, hi, halvings):
    """Three sides in [lo, hi] that the hierarchy can halve `halvings` times
    down to at most 8 cells a side."""
    unit = 1 << halvings
    return [unit * rng.randint(max(2, -(-lo // unit)), max(2, min(8, hi // unit))) for _ in range(3)]


def draw(rng):
    kind = rng.choice(["saddle", "reaction", "step", "batch", "vcycle", "vcycle", "vcycle", "vcycle", "operator",
                       "blobs", "predict", "train"])
    case = dict(kind=kind)
    if kind in ("saddle", "reaction"):
        sides = _box(rng, 16, 96, rng.choice([3, 4]))
        cells = sides[0] * sides[1] * sides[2]
        case.update(nx=sides[0], ny=sides[1], nz=sides[2],
                    blobs=_between(rng, 1 + cells // 50000, max(2, cells // 1500)),
                    alpha=rng.choice([0.0, 0.0, 0.1, 0.3]))
    elif kind == "step":
        sides = _box(rng, 64, 224, 5)
        case.update(nx=sides[0], ny=sides[1], nz=sides[2],
                    blobs=_between(rng, 600, max(700, sides[0] * sides[1] * sides[2] // 3000)))
    elif kind == "batch":
        case.update(count=rng.randint(4, 11), largest=rng.choice([96, 128, 160]), most=_between(rng, 200, 2000))
    elif kind == "vcycle":
        bits = rng.choice([32, 32, 64])
        sides = _box(rng, 32, 320, rng.choice([5, 6])) if bits == 32 else _box(rng, 16, 160, rng.choice([4, 5]))
        nu = rng.choice([(1, 1), (2, 2)]) if bits == 32 else (2, 2)
        case.update(nx=sides[0], ny=sides[1], nz=sides[2], bits=bits, nu1=nu[0], nu2=nu[1],
                    alpha=rng.choice([0.0, 0.1]))
    elif kind in ("operator", "blobs"):
        sides = _box(rng, 32, 256, rng.choice([4, 5]))
        cells = sides[0] * sides[1] * sides[2]
        case.update(nx=sides[0], ny=sides[1], nz=sides[2], blobs=_between(rng, 1, max(2, cells // 1000)))
        case.update(dict(alpha=rng.choice([0.0, 0.1]), form=rng.choice(["apply", "residual"]))
                    if kind == "operator" else dict(width=rng.choice([3, 4])))
    else:
        side = rng.choice([128, 160, 192, 256] if kind == "predict" else [96, 128, 160])
        case.update(side=side, blobs=_between(rng, 30, min(4096, side ** 3 // 500)))
    return case


# ---------------------------------------------------------------- inputs
def _rng(seed, stream=0):
    return np.random.default_rng([int(seed), int(stream)])


def _field(dims, seed, scale=1.0):
    """A smooth field plus noise, as a concentration or a residual is: [nz][ny][nx], FP64."""
    nx, ny, nz = dims
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    out = torch.randn(nz, ny, nx, dtype=torch.float64, device="cuda", generator=gen)
    phase = _rng(seed, 7).uniform(0.0, 2.0 * math.pi, 3)
    for axis, n in enumerate((nz, ny, nx)):
        wave = torch.sin(torch.arange(n, dtype=torch.float64, device="cuda") * (2.0 * math.pi / n) + phase[axis])
        out += 3.0 * wave.reshape([-1 if a == axis else 1 for a in range(3)])
    return out.mul_(scale)


def _positions(dims, count, seed, spacing=4.0):
    """Blob centres at least `spacing` apart: distinct sites of a lattice, each
    moved by up to half of what its cell leaves. (count, 3) FP64, h = 1."""
    rng = _rng(seed, 1)
    gap = spacing + 1.0
    while True:
        sites = [max(1, int(n // gap)) for n in dims]
        if sites[0] * sites[1] * sites[2] >= count:
            break
        gap -= 0.1
    pick = rng.permutation(sites[0] * sites[1] * sites[2])[:count]
    ijk = np.stack([pick % sites[0], pick // sites[0] % sites[1], pick // (sites[0] * sites[1])], axis=1)
    cell = np.array([n / s for n, s in zip(dims, sites)])
    room = np.maximum(cell - spacing, 0.2)
    return np.ascontiguousarray((ijk + 0.5) * cell + rng.uniform(-0.5, 0.5, (count, 3)) * room + rng.uniform(0, 1, 3))


def _rates(count, seed):
    """Reaction rates, log-uniform in [0.1, 10]."""
    return np.exp(_rng(seed, 2).uniform(math.log(0.1), math.log(10.0), count))


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()


def _realisations(case, seed):
    """(side, blob positions, rates) of a batch's problems: sides between 64 and
    the largest, blob counts log-uniform in [16, most]."""
    out = []
    sides = [s for s in (64, 96, 128, 160) if s <= case["largest"]]
    sizes = _rng(case["count"] * 1000 + case["most"], 5)  # which sizes there are is the case's, not the seed's
    for i in range(case["count"]):
        side = sides[-1 - i % len(sides)]
        n = int(round(math.exp(sizes.uniform(math.log(16), math.log(case["most"])))))
        out.append((side, _positions((side,) * 3, n, seed * 64 + i, 3.0), _rates(n, seed * 64 + i)))
    return out


def _network(seed):
    """Network parameters as a trained model's: weights of every size between
    +-1/sqrt(fan in), small biases. FP32, in the library's order."""
    rng = _rng(seed, 3)
    parts = [rng.uniform(-0.25, 0.25, WIDTH * BASES), rng.uniform(-0.05, 0.05, WIDTH)]
    for _ in range(LAYERS):
        parts += [rng.uniform(-0.25, 0.25, WIDTH * BASES), rng.uniform(-0.05, 0.05, WIDTH),
                  rng.uniform(-0.125, 0.125, 2 * WIDTH * WIDTH), rng.uniform(-0.05, 0.05, WIDTH)]
    parts += [rng.uniform(-0.125, 0.125, WIDTH), rng.uniform(-0.05, 0.05, 1)]
    return np.concatenate(parts).astype(np.float32)


def _multipliers(count, seed):
    return np.exp(_rng(seed, 4).normal(0.0, 0.2, count))


def _dims(case):
    return (case["nx"], case["ny"], case["nz"])


# ---------------------------------------------------------------- the calls
def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind in ("saddle", "reaction", "step", "operator", "blobs"):
        dims = _dims(case)
        q = _dev(_positions(dims, case["blobs"], seed))
        s.update(q=q, kappa=_dev(_rates(case["blobs"], seed)))
    if kind in ("saddle", "reaction"):
        s["grid"] = ibrd.Grid(*dims, alpha=case["alpha"])
        s["grid"].set_blobs(q)
        s.update(rhs=s["grid"].field(1.0), c=s["grid"].field(), lam=torch.zeros_like(s["kappa"]))
    elif kind == "step":
        s["streams"] = [torch.cuda.Stream(), torch.cuda.Stream(priority=-1)]
        s["grids"] = [ibrd.Grid(*dims, precision=ibrd.IBRD_MIXED_REFINE, stream=t.cuda_stream) for t in s["streams"]]
        s.update(rhs=s["grids"][0].field(1.0), c=[g.field() for g in s["grids"]], lam=torch.zeros_like(s["kappa"]),
                 opts=[ibrd.ibrd_default_opts(tol=TOL, precision=ibrd.IBRD_MIXED_REFINE, max_iter=3000, **o)
                       for o in (REACTION, SADDLE)])
    elif kind == "batch":
        s.update(streams=[], grids=[], kappa=[], rhs=[], c=[])
        for side, q, kappa in _realisations(case, seed):
            s["streams"].append(torch.cuda.Stream())
            g = ibrd.Grid(side, side, side, precision=ibrd.IBRD_MIXED_REFINE, stream=s["streams"][-1].cuda_stream)
            q = _dev(q)
            torch.cuda.synchronize()  # the handle's stream does not wait for torch's
            g.set_blobs(q)
            s["grids"].append(g)
            s["kappa"].append(_dev(kappa))
            s["rhs"].append(g.field(1.0))
            s["c"].append(g.field())
        s["opts"] = ibrd.ibrd_default_opts(tol=TOL, precision=ibrd.IBRD_MIXED_REFINE, max_iter=3000, **REACTION)
    elif kind == "vcycle":
        s["grid"] = ibrd.Grid(*_dims(case), alpha=case["alpha"])
        s["rhs"] = _field(_dims(case), seed).to(torch.float32 if case["bits"] == 32 else torch.float64)
        s["x"] = torch.zeros_like(s["rhs"])
    elif kind == "operator":
        s["grid"] = ibrd.Grid(*dims, alpha=case["alpha"])
        s["grid"].set_blobs(q)
        s.update(c=_field(dims, seed), rhs=_field(dims, seed + 500000), y=s["grid"].field(),
                 jc=torch.zeros_like(s["kappa"]))
    elif kind == "blobs":
        s["grid"] = ibrd.Grid(*dims, kernel=case["width"])
        s.update(c=_field(dims, seed), y=s["grid"].field(), jc=torch.zeros_like(s["kappa"]))
    else:
        side = case["side"]
        s.update(box=np.array([float(side)] * 3), q=_dev(_positions((side,) * 3, case["blobs"], seed, 3.0)),
                 model=ibrd.GNN(CUTOFF, NEIGHBOURS), lam=_dev(_multipliers(case["blobs"], seed)))
        s["model"].set_params(_network(seed))
    torch.cuda.synchronize()
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "saddle":
        s["grid"].solve_saddle(s["rhs"], c=s["c"], lam=s["lam"], tol=TOL)
        return s["c"], s["lam"]
    if kind == "reaction":
        s["grid"].solve_reaction(s["kappa"], s["rhs"], c=s["c"], tol=TOL)
        return s["c"]
    if kind == "step":
        a, b = s["grids"]
        ibrd.ibrd_solve_many([
            dict(kind="reaction", grid=a.handle, q=s["q"], kappa=s["kappa"], rhs=s["rhs"], c=s["c"][0],
                 opts=s["opts"][0]),
            dict(kind="saddle", grid=b.handle, q=s["q"], rhs=s["rhs"], c=s["c"][1], lam=s["lam"],
                 opts=s["opts"][1])], threads=2)
        return s["c"][0], s["c"][1], s["lam"]
    if kind == "batch":
        ibrd.ibrd_solve_reaction_batch([g.handle for g in s["grids"]], s["kappa"], s["rhs"], s["c"], s["opts"],
                                       threads=16)
        return s["c"]
    if kind == "vcycle":
        if case["bits"] == 64:
            return s["grid"].vcycle(s["rhs"], s["x"])
        return s["grid"].vcycle_f32(s["rhs"], s["x"], nu1=case["nu1"], nu2=case["nu2"])
    if kind == "operator":
        g = s["grid"]
        g.interp(s["c"], s["jc"])
        if case["form"] == "apply":
            g.apply_L(s["c"], s["y"])
            return g.spread(s["kappa"] * s["jc"], s["y"], accumulate=True)
        g.residual(s["rhs"], s["c"], s["y"])
        return g.spread(-s["kappa"] * s["jc"], s["y"], accumulate=True)
    if kind == "blobs":
        s["grid"].set_blobs(s["q"])
        return s["grid"].spread(s["kappa"], s["y"]), s["grid"].interp(s["c"], s["jc"])
    if kind == "predict":
        return s["model"].predict(s["q"], s["box"], float(case["side"] ** 3))
    loss, grad = s["model"].loss_grad(s["q"], s["box"], s["lam"])
    return loss, grad


def work(case):
    """Each input read once, each output written once; the arithmetic of one
    application of what the call defines (for a solve: of its operator)."""
    kind = case["kind"]
    if kind == "batch":
        cells = sum(side ** 3 for side, _, _ in _realisations(case, 0))
        return {"bytes": 16.0 * cells, "flops": 8.0 * cells}
    if kind in ("predict", "train"):
        n = case["blobs"]
        edges = n * min(NEIGHBOURS, (n - 1) * (4.0 / 3.0) * math.pi * CUTOFF ** 3 / case["side"] ** 3)
        flops = LAYERS * (edges * WIDTH * (2 * BASES + 3) + n * 4 * WIDTH * WIDTH)
        params = 4.0 * ibrd.ibrd_gnn_num_params()
        return {"bytes": 32.0 * n + params * (1 if kind == "predict" else 2),
                "flops": flops * (1 if kind == "predict" else 3)}
    cells = float(case["nx"] * case["ny"] * case["nz"])
    if kind == "vcycle":
        return {"bytes": 2.0 * case["bits"] / 8 * cells,
                "flops": cells * (9.0 * (case["nu1"] + case["nu2"]) + 20.0) * 8.0 / 7.0}
    n = case["blobs"]
    if kind == "step":
        return {"bytes": 24.0 * cells + 40.0 * n, "flops": 16.0 * cells + 600.0 * n}
    if kind == "blobs":
        return {"bytes": 8.0 * cells + 8.0 * 64 * n + 40.0 * n, "flops": 500.0 * n}
    if kind == "operator" and case["form"] == "residual":
        return {"bytes": 24.0 * cells + 40.0 * n, "flops": 9.0 * cells + 300.0 * n}
    return {"bytes": 16.0 * cells + 40.0 * n, "flops": 8.0 * cells + 300.0 * n}


# ---------------------------------------------------------------- what the calls return, in 64 bits
def _apply(c, alpha, h=1.0):
    lap = -6.0 * c
    for axis in range(3):
        lap += torch.roll(c, 1, axis) + torch.roll(c, -1, axis)
    return alpha * c - lap / (h * h)


def _symbol(shape, alpha, h=1.0):
    """Eigenvalues of alpha I - L on the half spectrum of rfftn, 0 where singular."""
    nz, ny, nx = shape
    out = 0.0
    for axis, (n, m) in enumerate(((nz, nz), (ny, ny), (nx, nx // 2 + 1))):
        k = torch.arange(m, dtype=torch.float64, device="cuda")
        lam = (2.0 - 2.0 * torch.cos(2.0 * math.pi * k / n)) / (h * h)
        out = out + lam.reshape([-1 if a == axis else 1 for a in range(3)])
    return out + alpha


def _green(b, alpha, h=1.0):
    """A^-1 b (the pseudo-inverse when alpha = 0)."""
    lam = _symbol(b.shape, alpha, h)
    if alpha == 0.0:
        lam[0, 0, 0] = math.inf
    return torch.fft.irfftn(torch.fft.rfftn(b) / lam, s=b.shape)


def _peskin(r, width):
    r = r.abs()
    if width == 4:
        near = (3.0 - 2.0 * r + torch.sqrt((1.0 + 4.0 * r - 4.0 * r * r).clamp_min(0.0))) / 8.0
        far = (5.0 - 2.0 * r - torch.sqrt((-7.0 + 12.0 * r - 4.0 * r * r).clamp_min(0.0))) / 8.0
        return torch.where(r < 1.0, near, torch.where(r < 2.0, far, torch.zeros_like(r)))
    near = (1.0 + torch.sqrt((1.0 - 3.0 * r * r).clamp_min(0.0))) / 3.0
    far = (5.0 - 3.0 * r - torch.sqrt((1.0 - 3.0 * (1.0 - r) ** 2).clamp_min(0.0))) / 6.0
    return torch.where(r <= 0.5, near, torch.where(r < 1.5, far, torch.zeros_like(r)))


class _Blobs:
    """J and S (h = 1) as a gather and a scatter over each blob's 5^3 cells."""

    def __init__(self, q, dims, width=4):
        self.dims = dims
        u = q - 0.5
        base = torch.floor(u)
        off = torch.arange(-2, 3, dtype=torch.float64, device="cuda")
        cells = base[:, :, None] + off
        w = _peskin(u[:, :, None] - cells, width)
        n = torch.tensor(dims, dtype=torch.float64, device="cuda")
        i = torch.remainder(cells, n[None, :, None]).long()
        nx, ny, _ = dims
        self.at = ((i[:, 2, :, None, None] * ny + i[:, 1, None, :, None]) * nx + i[:, 0, None, None, :]).reshape(-1)
        self.w = (w[:, 2, :, None, None] * w[:, 1, None, :, None] * w[:, 0, None, None, :]).reshape(len(q), 125)

    def interp(self, c):
        return (c.reshape(-1)[self.at].reshape(self.w.shape) * self.w).sum(1)

    def spread(self, lam):
        nx, ny, nz = self.dims
        out = torch.zeros(nx * ny * nz, dtype=torch.float64, device="cuda")
        out.index_add_(0, self.at, (self.w * lam[:, None]).reshape(-1))
        return out.reshape(nz, ny, nx)


def _constrained(q, dims, rhs, alpha, kappa):
    """(c, lambda) of A c + S lambda = rhs with J c = lambda / kappa (J c = 0
    without kappa), by conjugate gradients on the blob unknowns."""
    blobs = _Blobs(q, dims)

    def matrix(v):
        out = blobs.interp(_green(blobs.spread(v), alpha))
        return out if kappa is None else out + v / kappa

    lam = torch.zeros(len(q), dtype=torch.float64, device="cuda")
    free = (lambda v: v - v.mean()) if alpha == 0.0 else (lambda v: v)
    if alpha == 0.0:
        lam += rhs.sum() / len(q)
    b = blobs.interp(_green(rhs, alpha))
    r = free(b - matrix(lam))
    p, rr = r.clone(), torch.dot(r, r)
    size = torch.dot(b, b) + rr
    for _ in range(1000):
        if not rr > 1e-30 * size:
            break
        mp = free(matrix(p))
        step = rr / torch.dot(p, mp)
        lam += step * p
        r -= step * mp
        new = torch.dot(r, r)
        p = r + (new / rr) * p
        rr = new
    c = _green(rhs - blobs.spread(lam), alpha)
    if alpha == 0.0:
        jc = 0.0 if kappa is None else lam / kappa
        c += (jc - blobs.interp(c)).mean()
    return c, lam


def _sweep(x, b, h, alpha, red):
    for colour in (red, ~red):
        nb = torch.zeros_like(x)
        for axis in range(3):
            nb += torch.roll(x, 1, axis) + torch.roll(x, -1, axis)
        x = torch.where(colour, (b + nb / (h * h)) / (alpha + 6.0 / (h * h)), x)
    return x


def _prolong(e):
    for axis in range(3):
        pair = torch.stack([0.75 * e + 0.25 * torch.roll(e, 1, axis), 0.75 * e + 0.25 * torch.roll(e, -1, axis)],
                           axis + 1)
        e = pair.flatten(axis, axis + 1)
    return e


def _vcycle(b, h, alpha, nu1, nu2, single):
    shape = b.shape
    halve = all(n % 2 == 0 and n >= 4 for n in shape)
    if not halve or (single and b.numel() <= 32768 and max(shape) <= 64):
        return _green(b, alpha, h)
    i = [torch.arange(n, device="cuda").reshape([-1 if a == axis else 1 for a in range(3)])
         for axis, n in enumerate(shape)]
    red = (i[0] + i[1] + i[2]) % 2 == 0
    x = torch.zeros_like(b)
    for _ in range(nu1):
        x = _sweep(x, b, h, alpha, red)
    r = b - _apply(x, alpha, h)
    r = r.reshape(shape[0] // 2, 2, shape[1] // 2, 2, shape[2] // 2, 2).mean(dim=(1, 3, 5))
    x = x + _prolong(_vcycle(r, 2.0 * h, alpha, nu1, nu2, single))
    for _ in range(nu2):
        x = _sweep(x, b, h, alpha, red)
    return x


def _outputs(theta, q, side):
    """The network's outputs y, differentiable in theta."""
    n = len(q)
    src, dst, dist = [], [], []
    for lo in range(0, n, 1024):
        d = q[lo:lo + 1024, None, :] - q[None, :, :]
        d -= side * torch.round(d / side)
        r = d.square().sum(2).sqrt()
        r[torch.arange(len(r), device="cuda"), torch.arange(lo, lo + len(r), device="cuda")] = math.inf
        i, j = torch.nonzero(r < CUTOFF, as_tuple=True)
        dst.append(i + lo)
        src.append(j)
        dist.append(r[i, j])
    src, dst, s = torch.cat(src), torch.cat(dst), torch.cat(dist) / CUTOFF
    fc = (1.0 - s) ** 2
    centre = torch.arange(BASES, dtype=torch.float64, device="cuda") / (BASES - 1)
    basis = fc[:, None] * torch.exp(-((s[:, None] - centre) * ((BASES - 1) / 1.5)) ** 2)

    def gather(values):
        return torch.zeros(n, values.shape[1], dtype=torch.float64, device="cuda").index_add(0, dst, values)

    at = 0

    def take(*shape):
        nonlocal at
        size = math.prod(shape)
        at += size
        return theta[at - size:at].reshape(shape)

    w0, c0 = take(WIDTH, BASES), take(WIDTH)
    h = torch.relu(gather(basis) @ w0.T + c0)
    for _ in range(LAYERS):
        e, eb, w, v, c = take(WIDTH, BASES), take(WIDTH), take(WIDTH, WIDTH), take(WIDTH, WIDTH), take(WIDTH)
        m = gather(fc[:, None] * torch.relu(basis @ e.T + eb) * h[src])
        h = h + torch.relu(m @ w.T + h @ v.T + c)
    return h @ take(WIDTH) + take(1)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("predict", "train"):
        theta = _dev(_network(seed)).requires_grad_(kind == "train")
        q = _dev(_positions((case["side"],) * 3, case["blobs"], seed, 3.0))
        y = _outputs(theta, q, float(case["side"]))
        if kind == "predict":
            return float(case["side"] ** 3) * torch.softmax(y, 0)
        t = torch.log(_dev(_multipliers(case["blobs"], seed)))
        loss = ((y - y.mean()) - (t - t.mean())).square().mean()
        loss.backward()
        return loss.detach(), theta.grad
    if kind == "batch":
        out = []
        for side, q, kappa in _realisations(case, seed):
            rhs = torch.ones(side, side, side, dtype=torch.float64, device="cuda")
            out.append(_constrained(_dev(q), (side,) * 3, rhs, 0.0, _dev(kappa))[0])
        return out
    dims = _dims(case)
    if kind == "vcycle":
        b = _field(dims, seed)
        if case["bits"] == 32:
            b = b.to(torch.float32).to(torch.float64)
        if case["alpha"] == 0.0:
            b = b - b.mean()
        x = _vcycle(b, 1.0, case["alpha"], case["nu1"], case["nu2"], case["bits"] == 32)
        return x - x.mean() if case["alpha"] == 0.0 else x
    q, kappa = _dev(_positions(dims, case["blobs"], seed)), _dev(_rates(case["blobs"], seed))
    if kind == "operator":
        blobs, c = _Blobs(q, dims), _field(dims, seed)
        y = _apply(c, case["alpha"]) + blobs.spread(kappa * blobs.interp(c))
        return y if case["form"] == "apply" else _field(dims, seed + 500000) - y
    if kind == "blobs":
        blobs = _Blobs(q, dims, case["width"])
        return blobs.spread(kappa), blobs.interp(_field(dims, seed))
    rhs = torch.ones(dims[2], dims[1], dims[0], dtype=torch.float64, device="cuda")
    if kind == "reaction":
        return _constrained(q, dims, rhs, case["alpha"], kappa)[0]
    if kind == "saddle":
        return _constrained(q, dims, rhs, case["alpha"], None)
    c, lam = _constrained(q, dims, rhs, 0.0, None)
    return _constrained(q, dims, rhs, 0.0, kappa)[0], c, lam
