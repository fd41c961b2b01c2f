"""The calls that a user of this library spends time in, as cases to measure.

A case is one pair of magnets and one call (or the few calls that belong
together) on it:

  stray      set_displacement and both stray fields: one point of an offset
             sweep;
  torque     compute_torque of the slider: one whole field evaluation (both
             demagnetising fields, both stray fields, forces) and the
             right-hand side;
  step       a trajectory of a few fixed Dormand-Prince steps from a given
             state (the launches of an adaptive step, at step sizes that do
             not depend on rounding);
  gradients  backward_energy of both magnetisations and of the displacement;
  batch      step_batch of many uneven pairs on several streams;
  eddy       eddy_field of a conducting magnet.

`exact` restates each in 64 bits: the kernels by closed forms and quadrature,
the convolutions by FFT on a grid of its own, the spline as dense operators
per axis, the Neumann problem by cosine transforms.
"""

import math

import torch

from paper_1801_04181_gb300 import pair_context, step_batch

MU0 = 4e-7 * math.pi
GAMMA_LL = 1.7595e11  # rad / (s T)
MARGIN = 4            # box margin in cells (the library's default)


# ---------------------------------------------------------------- what is measured
class _Material:
    def __init__(self, Ms, Aex, Ku=0.0, alpha=0.5):
        self.Ms, self.Aex, self.Ku, self.ku_axis, self.alpha = Ms, Aex, Ku, (0.0, 0.0, 1.0), alpha


class _Mechanics:
    def __init__(self, mass, k, v_drive, gamma_v, x0_spring=0.0):
        self.mass, self.k, self.v_drive, self.gamma_v, self.x0_spring = mass, k, v_drive, gamma_v, x0_spring
        self.dir = (1.0, 0.0, 0.0)


# material and mechanics of the repository's workloads, by name
_MATERIALS = {
    "plain": _Material(8e5, 1.3e-11),
    "pma": _Material(1.1e6, 1.5e-11, Ku=1.0e6),
    "cocrpt": _Material(3.5e5, 5e-12, Ku=1.225e5, alpha=0.05),
}
_SPRING = _Mechanics(2.5e-18, 1e-3, 1.0, 4e7)
_FRICTION = _Mechanics(3.5e-11 ** 2 / 0.02, 0.005, 2.0, 0.02 / 3.5e-11, x0_spring=80e-9)


class _Pair:
    """A pair description as pair_context takes it, from a case's values."""

    def __init__(self, c):
        self.n_base = (c["nx"], c["ny"], c["nz"])
        self.n_slider = (c.get("sx", c["nx"]), c.get("sy", c["ny"]), c.get("sz", c["nz"]))
        self.cell = (c["cell_nm"] * 1e-9,) * 3
        beyond = [c["nx"] + c["gap"], 0, 0] if c["beside"] else [0, 0, c["nz"] + c["gap"]]
        self.offsets = [(0, 0, 0), tuple(beyond)]
        self.mat_base = self.mat_slider = _MATERIALS[c["material"]]
        self.mech = _FRICTION if c["material"] == "cocrpt" else _SPRING
        self.H_ext = (0.0, 0.0, 0.0)
        self.u0 = (c["ux"], c["uy"], 0.0)
        self.periodic = 3 if c["periodic"] else 0
        self.pbc_images = 2

    @property
    def sizes(self):
        return (self.n_base, self.n_slider)


def _case(op, n, slider=None, **more):
    c = dict(op=op, nx=n[0], ny=n[1], nz=n[2], gap=5, cell_nm=4.0, material="pma", pattern="domains", beside=False,
             ux=0.3125, uy=0.0, periodic=False, precision="fp32", steps=0)
    if slider is not None:
        c.update(sx=slider[0], sy=slider[1], sz=slider[2])
    c.update(more)
    return c


def _plain(op, n, **more):
    return _case(op, n, **{**dict(gap=1, material="plain", pattern="random", uy=0.25), **more})


def _cubes(op, n, **more):
    return _case(op, n, **{**dict(gap=3, cell_nm=2.0, material="plain", pattern="vortex", beside=True), **more})


def listed():
    return [
        # one offset of the plain-film sweep: the smallest call, launches and latency
        dict(_plain("stray", (64, 64, 1)), name="stray_64x64x1"),
        # films of unequal, odd extents, as cut from a measured sample: no power of two anywhere
        dict(_case("torque", (355, 145, 3), slider=(301, 127, 2), ux=17.6, uy=-2.3), name="torque_odd_355x145x3"),
        # the headline workload: spring-pulled domain films, a short trajectory
        dict(_case("step", (1024, 256, 2), steps=3), name="step_stick_slip_1024x256x2"),
        # the same films with the reduced-precision transforms
        dict(_case("torque", (1024, 256, 2), precision="mixed"), name="torque_mixed_1024x256x2"),
        # one square film over another, a single layer each: long y lines in the fused pass
        dict(_case("torque", (1024, 1024, 1)), name="torque_1024x1024x1"),
        # eight layers: z by the direct sum, the largest single pair
        dict(_case("torque", (512, 512, 8)), name="torque_512x512x8"),
        # the friction films, periodic in the film plane
        dict(_case("step", (256, 256, 5), material="cocrpt", pattern="stripes", periodic=True, steps=2),
             name="step_friction_256x256x5"),
        # vortex cubes side by side: z by FFT
        dict(_cubes("torque", (64, 64, 64)), name="torque_cubes_64"),
        # their energy gradients, one iteration of an optimisation
        dict(_cubes("gradients", (64, 64, 64)), name="gradients_cubes_64"),
        # many uneven pairs stepped together, the parameter-study form
        dict(_case("batch", (512, 256, 4), steps=1, pairs=16), name="batch_16_pairs"),
        # the eddy field of a conducting cube
        dict(_cubes("eddy", (64, 64, 64)), name="eddy_cube_64"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _film(rng, nx, ny, nz, most):
    while True:
        n = (_log(rng, *nx), _log(rng, *ny), rng.randint(*nz))
        # the fused pass of thin films holds 4 nz + 3 lines of a padded y extent on chip
        if n[0] * n[1] * n[2] <= most and (n[2] > 4 or (4 * n[2] + 3) * n[1] <= 11000):
            return n


def _shift(rng, lo, hi):
    """A displacement in cells that a short trajectory does not take over a cell's edge."""
    return rng.randint(lo, hi - 1) + round(rng.uniform(0.02, 0.98), 4)


def _moved(rng):
    return dict(ux=_shift(rng, -20, 20), uy=_shift(rng, -3, 3))


def draw(rng):
    kind = rng.choice(["stray", "stray", "torque", "torque", "step", "step", "mixed", "layers", "friction", "cubes",
                       "gradients", "batch", "eddy"])
    if kind == "stray":
        return _plain("stray", _film(rng, (16, 512), (16, 256), (1, 4), 1 << 19), gap=rng.randint(1, 8), **_moved(rng))
    if kind == "torque":
        n = _film(rng, (64, 1024), (64, 1024), (1, 4), 1 << 20)
        s = tuple(max(16, int(v * rng.uniform(0.5, 1.0))) for v in n[:2]) + (rng.randint(1, n[2]),)
        return _case("torque", n, slider=s if rng.random() < 0.5 else None, **_moved(rng))
    if kind == "step":
        return _case("step", _film(rng, (64, 1024), (64, 256), (1, 4), 1 << 19), steps=rng.randint(1, 3), **_moved(rng))
    if kind == "mixed":
        return _case("torque", _film(rng, (64, 1024), (64, 512), (1, 8), 1 << 19), precision="mixed", **_moved(rng))
    if kind == "layers":
        return _case("torque", _film(rng, (64, 512), (64, 512), (5, 8), 1 << 21), **_moved(rng))
    if kind == "friction":
        sizes = [n for n in range(64, 257, 2) if _smooth(n)]
        return _case("step", (rng.choice(sizes), rng.choice(sizes), rng.randint(1, 5)), material="cocrpt",
                     pattern="stripes", periodic=True, steps=rng.randint(1, 2), ux=_shift(rng, -20, 20))
    if kind == "cubes":
        return _cubes("torque", tuple(_log(rng, 16, 64) for _ in range(3)), ux=_shift(rng, 0, 8))
    if kind == "gradients":
        return _cubes("gradients", tuple(_log(rng, 8, 64) for _ in range(3)), ux=_shift(rng, 0, 8))
    if kind == "batch":
        return _case("batch", (_log(rng, 96, 512), _log(rng, 96, 256), rng.randint(1, 4)), steps=1,
                     pairs=rng.randint(4, 16))
    return _cubes("eddy", tuple(_log(rng, 16, 64) for _ in range(3)))


def _smooth(n):
    for p in (2, 3, 5):
        while n % p == 0:
            n //= p
    return n == 1


# ---------------------------------------------------------------- inputs
def _pattern(kind, n, g, slant=20):
    """Unit magnetisation (3, nz, ny, nx) float32 on the generator's device."""
    nx, ny, nz = n
    dev = g.device
    tilt = torch.randn((3, nz, ny, nx), generator=g, device=dev, dtype=torch.float64)
    if kind == "random":
        m = tilt
    elif kind in ("domains", "stripes"):  # up / down domains of `slant` cells, a small in-plane tilt
        shift = torch.randint(0, 2 * slant, (2,), generator=g, device=dev)
        ix = (torch.arange(nx, device=dev) + shift[0]) // slant
        iy = (torch.arange(ny, device=dev) + shift[1]) // slant
        if kind == "stripes":
            mz = (1.0 - 2.0 * (ix % 2).double()).expand(ny, nx)
        else:
            signs = torch.randint(0, 2, (ny // slant + 4, nx // slant + 4), generator=g, device=dev).double() * 2 - 1
            mz = signs[iy][:, ix]
        m = 0.05 * tilt
        m[2] = mz
    else:  # vortex
        r = torch.rand(4, generator=g, device=dev, dtype=torch.float64)
        z, y, x = torch.meshgrid(*(torch.arange(k, device=dev, dtype=torch.float64) for k in (nz, ny, nx)),
                                 indexing="ij")
        x, y = x - (nx - 1) / 2 - 8 * (r[2] - 0.5), y - (ny - 1) / 2 - 8 * (r[3] - 0.5)
        chi, pol = (1.0 - 2.0 * (v > 0.5).double() for v in r[:2])
        m = torch.stack([-chi * y, chi * x, pol * torch.exp(-(x * x + y * y) / 16.0)])
    return (m / m.norm(dim=0, keepdim=True)).float()


def _pairs_of(case):
    """The pairs of a case: one, or a batch of uneven sizes up to the case's."""
    if case["op"] != "batch":
        return [_Pair(case)]
    g = torch.Generator().manual_seed(case["nx"] * 1009 + case["ny"] * 31 + case["nz"])
    out = []
    for _ in range(case["pairs"]):
        r = torch.rand(4, generator=g, dtype=torch.float64).tolist()
        n = (64 + int(r[0] * (case["nx"] - 63)), 64 + int(r[1] * (case["ny"] - 63)), 1 + int(r[2] * case["nz"]))
        out.append(_Pair(dict(case, nx=n[0], ny=n[1], nz=n[2], ux=50.0 * r[3])))
    return out


def _inputs(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    ms = [[_pattern(case["pattern"], n, g) for n in p.sizes] for p in _pairs_of(case)]
    extra = None
    if case["op"] == "eddy":  # the rate of change of the flux density, T / s
        extra = 1e9 * torch.randn(ms[0][0].shape, generator=g, device="cuda", dtype=torch.float32)
    return ms, extra


_DT = 1e-13      # s, a step size the films accept at the default tolerance
_SIGMA = 1e6     # S / m
_LANES = 8       # streams of a batch


def prepare(case, seed):
    pairs = _pairs_of(case)
    ms, extra = _inputs(case, seed)
    lanes = [torch.cuda.Stream() for _ in range(_LANES)] if case["op"] == "batch" else None
    mms = []
    for i, (p, m) in enumerate(zip(pairs, ms)):
        mms.append(pair_context(p, m[0], m[1], adaptive=False, precision=case["precision"],
                                stream=lanes[i % _LANES] if lanes else None))
        mms[-1].compute_fields()  # plans the grids
    return dict(case=case, pairs=pairs, ms=ms, extra=extra, mms=mms, lanes=lanes)


def _start(s, i):
    """The state a trajectory starts from: m of both magnets, the slider moving at the drive's speed."""
    mm, p = s["mms"][i], s["pairs"][i]
    for g in (0, 1):
        mm.set_magnetization(g, s["ms"][i][g])
    mm.set_displacement(tuple(u * d for u, d in zip(p.u0, p.cell)))
    mm.set_slider_state(0.0, p.mech.v_drive, 0.0)


def run(s):
    case, mm = s["case"], s["mms"][0]
    op = case["op"]
    if op == "stray":
        p = s["pairs"][0]
        mm.set_displacement(tuple(u * d for u, d in zip(p.u0, p.cell)))
        return dict(H=[mm.compute_stray_field(1), mm.compute_stray_field(0)])
    if op == "torque":
        mm.set_magnetization(1, s["ms"][0][1])
        dm, H = mm.compute_torque(1)
        return dict(dm=dm, H=H)
    if op == "step":
        _start(s, 0)
        mm.step(case["steps"], _DT)
        return dict(m=[mm.get_magnetization(g) for g in (0, 1)],
                    slider=torch.tensor(mm.get_slider_state(), dtype=torch.float32))
    if op == "gradients":
        for g in (0, 1):
            mm.set_magnetization(g, s["ms"][0][g])
        du, gs, gt = mm.backward_energy(0)
        return dict(du=torch.tensor(du, dtype=torch.float32), src=gs, tgt=gt)
    if op == "batch":
        for i in range(len(s["mms"])):
            _start(s, i)
        step_batch(s["mms"], case["steps"], [_DT] * len(s["mms"]))
        return dict(m=[[m.get_magnetization(g) for g in (0, 1)] for m in s["mms"]])
    H, J, sweeps = mm.eddy_field(0, s["extra"], _SIGMA)
    return dict(H=H, J=J, sweeps=sweeps)


# ---------------------------------------------------------------- least work
def _fft_flops(*q):
    n = math.prod(q)
    return 2.5 * n * math.log2(n)  # one real transform


def _evaluation(p, what):
    """(bytes, flops) of field evaluations of a pair: `what` counts the demag
    fields and the stray fields; every field is a transform of the source's m
    on a grid that holds the linear convolution and one back per output."""
    b = f = 0.0
    for s, (ns, nt) in enumerate((p.sizes, p.sizes[::-1])):
        cells, out = math.prod(ns), math.prod(nt)
        grid = [ns[a] if p.periodic and a < 2 else 2 * max(ns[a], nt[a]) for a in range(3)]
        if ns[2] == 1:
            grid[2] = 1
        f += _fft_flops(*grid) * 3
        if what["demag"]:
            f += _fft_flops(*grid) * 3 + 15.0 * math.prod(grid) / 2 * 2
        if what["stray"]:
            f += _fft_flops(*grid) + 5.0 * math.prod(grid) / 2 * 2
            f += 150.0 * out  # separable evaluation of the gradient and the Hessian
        b += 12.0 * cells * (1 + what["demag"]) + 12.0 * out * what["stray"]
    return b, f


def work(case):
    pairs = _pairs_of(case)
    both = dict(demag=1, stray=1)
    b = f = 0.0
    for p in pairs:
        cells = sum(math.prod(n) for n in p.sizes)
        if case["op"] == "stray":
            eb, ef = _evaluation(p, dict(demag=0, stray=1))
        elif case["op"] == "gradients":
            eb, ef = _evaluation(p, dict(demag=0, stray=1))
            eb, ef = eb / 2 + 24.0 * cells / 2, ef  # one direction there and one back
        elif case["op"] == "eddy":
            n = p.n_base
            eb = 36.0 * math.prod(n)
            # two cross products with S and the Poisson problem by fast transforms
            ef = 4 * 3 * _fft_flops(*[2 * k for k in n]) + 4 * _fft_flops(*n)
        elif case["op"] == "torque":
            eb, ef = _evaluation(p, both)
            eb, ef = eb + 24.0 * math.prod(p.n_slider), ef + 80.0 * math.prod(p.n_slider)
        else:
            evals = 6 * case["steps"] + 1
            eb, ef = _evaluation(p, both)
            eb, ef = evals * eb + 24.0 * cells, evals * (ef + 100.0 * cells)
        b, f = b + eb, f + ef
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------- in 64 bits
_DEVICE = "cuda"
_F64 = dict(dtype=torch.float64, device=_DEVICE)


def _gauss(n):
    """Gauss-Legendre nodes and weights on [-1/2, 1/2] (weights sum to 1), Golub-Welsch."""
    k = torch.arange(1, n, dtype=torch.float64)
    off = k / torch.sqrt(4 * k * k - 1)
    x, v = torch.linalg.eigh(torch.diag(off, 1) + torch.diag(off, -1))
    return [(float(a) / 2, float(b) ** 2) for a, b in zip(x, v[0])]


def _octant(nx, ny, nz):
    return torch.meshgrid(*(torch.arange(k, **_F64) for k in (nz, ny, nx)), indexing="ij")


def _S_points(x, y, z, rule):
    out = [torch.zeros_like(x) for _ in range(3)]
    for a, wa in rule:
        for b, wb in rule:
            for c, wc in rule:
                d = (x - a, y - b, z - c)
                r3 = (d[0] * d[0] + d[1] * d[1] + d[2] * d[2]) ** -1.5
                for k in range(3):
                    out[k] += (wa * wb * wc / (4 * math.pi)) * d[k] * r3
    return torch.stack(out)


def _S_octant(nx, ny, nz):
    """S of unit cubic cells at the offsets 0 <= d < n: (3, nz, ny, nx)."""
    z, y, x = _octant(nx, ny, nz)
    out = _S_points(x, y, z, _gauss(4))
    k = tuple(min(n, 7) for n in (nz, ny, nx))  # near: a finer rule; the own cell is zero by symmetry
    out[:, : k[0], : k[1], : k[2]] = _S_points(*(t[: k[0], : k[1], : k[2]] for t in (x, y, z)), _gauss(16))
    out[:, 0, 0, 0] = 0.0
    return out


def _ratio_asinh(num, den2):
    return torch.where(den2 > 0, torch.asinh(num / torch.sqrt(torch.where(den2 > 0, den2, 1.0))), 0.0)


def _ratio_atan(num, den):
    return torch.where(den != 0, torch.atan(num / torch.where(den != 0, den, 1.0)), 0.0)


def _newell_f(x, y, z):
    R = torch.sqrt(x * x + y * y + z * z)
    return (0.5 * y * (z * z - x * x) * _ratio_asinh(y, x * x + z * z)
            + 0.5 * z * (y * y - x * x) * _ratio_asinh(z, x * x + y * y)
            - x * y * z * _ratio_atan(y * z, x * R) + (2 * x * x - y * y - z * z) * R / 6)


def _newell_g(x, y, z):
    R = torch.sqrt(x * x + y * y + z * z)
    return (x * y * z * _ratio_asinh(z, x * x + y * y) + y * (3 * z * z - y * y) * _ratio_asinh(x, y * y + z * z) / 6
            + x * (3 * z * z - x * x) * _ratio_asinh(y, x * x + z * z) / 6 - z ** 3 * _ratio_atan(x * y, z * R) / 6
            - z * y * y * _ratio_atan(x * z, y * R) / 2 - z * x * x * _ratio_atan(y * z, x * R) / 2 - x * y * R / 3)


def _N_octant(nx, ny, nz):
    """N of unit cubic cells at the offsets 0 <= d < n: (6, nz, ny, nx), xx yy zz xy xz yz."""
    z, y, x = _octant(nx, ny, nz)
    rule = {}
    for t, wt in _gauss(4):  # the difference of a target and a source point
        for s, ws in _gauss(4):
            rule[round(t - s, 12)] = rule.get(round(t - s, 12), 0.0) + wt * ws
    out = torch.zeros((6, nz, ny, nx), **_F64)
    for a, wa in rule.items():
        for b, wb in rule.items():
            for c, wc in rule.items():
                d = (x + a, y + b, z + c)
                r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2]
                r2.clamp_(min=1e-6)  # only near offsets, replaced below
                w = (wa * wb * wc / (4 * math.pi)) * r2 ** -2.5
                for k in range(3):
                    out[k] += w * (r2 - 3 * d[k] * d[k])
                for k, (p, q) in enumerate(((0, 1), (0, 2), (1, 2))):
                    out[3 + k] -= 3 * w * d[p] * d[q]
    near = tuple(slice(0, 13) for _ in range(3))
    X, Y, Z = x[near], y[near], z[near]
    put = torch.zeros_like(out[(slice(None),) + near])
    for i, wi in ((-1, -1.0), (0, 2.0), (1, -1.0)):
        for j, wj in ((-1, -1.0), (0, 2.0), (1, -1.0)):
            for k, wk in ((-1, -1.0), (0, 2.0), (1, -1.0)):
                w, p = wi * wj * wk / (4 * math.pi), (X + i, Y + j, Z + k)
                put[0] += w * _newell_f(p[0], p[1], p[2])
                put[1] += w * _newell_f(p[1], p[0], p[2])
                put[2] += w * _newell_f(p[2], p[0], p[1])
                put[3] += w * _newell_g(p[0], p[1], p[2])
                put[4] += w * _newell_g(p[0], p[2], p[1])
                put[5] += w * _newell_g(p[1], p[2], p[0])
    out[(slice(None),) + near] = put
    return out


_TABLES = {}


def _table(make, reach):
    """The octant of a kernel up to `reach` offsets, or more: kept at its largest."""
    have = _TABLES.get(make)
    if have is None or any(h < r for h, r in zip(have.shape[:0:-1], reach)):
        had = have.shape[:0:-1] if have is not None else (0, 0, 0)
        _TABLES[make] = have = make(*(max(h, r) for h, r in zip(had, reach)))
    return have


# which axes (x, y, z) a kernel component is odd in
_ODD_S = ((1, 0, 0), (0, 1, 0), (0, 0, 1))
_ODD_N = ((0, 0, 0), (0, 0, 0), (0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1))
_N_OF = ((0, 3, 4), (3, 1, 5), (4, 5, 2))


class _Axis:
    """One axis of a convolution: offsets lo - (n - 1) .. lo + b - 1 on a circular
    grid of q points, or the images of one period (the offset of half a period
    averaged over its two truncations)."""

    def __init__(self, n, lo, b, period=0, images=2):
        self.nodes = torch.arange(lo, lo + b, device=_DEVICE)
        if period:
            self.q, at = period, []
            for c in range(period):
                s = c - period if 2 * c > period else c
                for e, w in (((s, 0.5), (-s, 0.5)) if 2 * s == period else ((s, 1.0),)):
                    at += [(c, e + i * period, w) for i in range(-images, images + 1)]
        else:
            span = n + b - 1
            self.q = next(q for q in range(span, 4 * span) if _smooth(q) and q % 2 == 0)
            at = [(d % self.q, d, 1.0) for d in range(lo - (n - 1), lo + b)]
        self.reach = 1 + max(abs(d) for _, d, _ in at)
        self.fold = []  # even and odd: circular index <- octant index
        for odd in (0, 1):
            A = torch.zeros((self.q, self.reach), dtype=torch.float64)
            for c, d, w in at:
                A[c, abs(d)] += w * (math.copysign(1.0, d) if odd else 1.0)
            self.fold.append(A.to(_DEVICE))

    def index(self):
        return self.nodes % self.q


class _Conv:
    """Spectra of a kernel over three axes (x, y, z) and the sums with them."""

    def __init__(self, make, odd, axes):
        self.axes = axes
        table = _table(make, [a.reach for a in axes])
        self.shape = tuple(a.q for a in axes[::-1])
        need = tuple(slice(0, a.reach) for a in axes[::-1])
        self.hat = []
        for comp, o in zip(table, odd):
            k = comp[need]
            k = torch.einsum("cz,zyx->cyx", axes[2].fold[o[2]], k)
            k = torch.einsum("cy,zyx->zcx", axes[1].fold[o[1]], k)
            k = torch.einsum("cx,zyx->zyc", axes[0].fold[o[0]], k)
            self.hat.append(torch.fft.rfftn(k))

    def forward(self, m):
        return torch.fft.rfftn(m, s=self.shape, dim=(-3, -2, -1))

    def back(self, spec):
        v = torch.fft.irfftn(spec, s=self.shape, dim=(-3, -2, -1))
        for d, a in zip((-1, -2, -3), self.axes):
            v = v.index_select(d, a.index())
        return v


def _spline_weights(t, order):
    s = 1 - t
    return (((s ** 3 / 6, (3 * t ** 3 - 6 * t * t + 4) / 6, (-3 * t ** 3 + 3 * t * t + 3 * t + 1) / 6, t ** 3 / 6)),
            (-s * s / 2, (9 * t * t - 12 * t) / 6, (-9 * t * t + 6 * t + 3) / 6, t * t / 2),
            (s, 3 * t - 2, 1 - 3 * t, t))[order]


class _Path64:
    """The stray field of magnet s inside magnet t of a pair."""

    def __init__(self, p, s, u):
        self.d = p.cell[0]
        ns, nt = p.sizes[s], p.sizes[1 - s]
        sign = 1.0 if s == 0 else -1.0
        axes, self.ops = [], []
        for a in range(3):
            off = p.offsets[1 - s][a] - p.offsets[s][a]
            shift = off + sign * u[a]
            per = ns[a] if p.periodic and a < 2 else 0
            lo = 0 if per else math.floor(shift) - 1 - MARGIN
            b = per or nt[a] + 3 + 2 * MARGIN
            axes.append(_Axis(ns[a], lo, b, per, p.pbc_images))
            # nodes -> coefficients -> value, first and second derivative at the targets
            B = torch.zeros((b, b), **_F64)
            for k in range(b):
                B[k, k] += 4 / 6
                for j in (k - 1, k + 1):
                    j = j % b if per else (1 if j < 0 else b - 2 if j >= b else j)
                    B[k, j] += 1 / 6
            B = torch.linalg.inv(B)
            base = math.floor(shift)
            ops = []
            for order in range(3):
                E = torch.zeros((nt[a], b), **_F64)
                i = torch.arange(nt[a], device=_DEVICE)
                for k, w in enumerate(_spline_weights(shift - base, order)):
                    j = i + base - 1 + k - lo
                    E[i, j % b if per else j] += w
                ops.append(E @ B / self.d ** order)
            self.ops.append(ops)
        self.conv = _Conv(_S_octant, _ODD_S, axes)

    def potential(self, M):
        f = self.conv.forward(M)
        return self.d * self.conv.back(sum(k * f[c] for c, k in enumerate(self.conv.hat)))

    def value(self, phi, ox, oy, oz):
        v = torch.einsum("tz,zyx->tyx", self.ops[2][oz], phi)
        v = torch.einsum("ty,zyx->ztx", self.ops[1][oy], v)
        return torch.einsum("tx,zyx->zyt", self.ops[0][ox], v)

    def gradient(self, phi):
        return torch.stack([self.value(phi, 1, 0, 0), self.value(phi, 0, 1, 0), self.value(phi, 0, 0, 1)])

    def force(self, phi, Mt):
        """Eq. (EQForce): -mu0 V sum_i Hess(phi) M_t."""
        F = []
        for a in range(3):
            s = 0.0
            for b in range(3):
                o = [int(k == a) + int(k == b) for k in range(3)]
                s = s + (self.value(phi, *o) * Mt[b]).sum()
            F.append(-MU0 * self.d ** 3 * s)
        return torch.stack(F)


class _Demag64:
    def __init__(self, p, g):
        n = p.sizes[g]
        axes = [_Axis(n[a], 0, n[a], n[a] if p.periodic and a < 2 else 0, p.pbc_images) for a in range(3)]
        self.conv = _Conv(_N_octant, _ODD_N, axes)

    def field(self, M):
        f = self.conv.forward(M)
        return -torch.stack([self.conv.back(sum(self.conv.hat[_N_OF[a][b]] * f[b] for b in range(3)))
                             for a in range(3)])


def _cross(a, b):
    return torch.linalg.cross(a, b, dim=0)


class _Pair64:
    """Right-hand side and Dormand-Prince steps of a pair."""

    def __init__(self, p):
        self.p, self.mat = p, (p.mat_base, p.mat_slider)
        self.demag = [_Demag64(p, g) for g in (0, 1)]

    def exchange(self, m, mat):
        d = self.p.cell[0]
        H = torch.zeros_like(m)
        for dim in (3, 2, 1):
            n = m.shape[dim]
            if n == 1:
                continue
            if self.p.periodic and dim > 1:
                H += m.roll(1, dim) + m.roll(-1, dim) - 2 * m
                continue
            step = m.narrow(dim, 1, n - 1) - m.narrow(dim, 0, n - 1)
            H.narrow(dim, 0, n - 1).add_(step)
            H.narrow(dim, 1, n - 1).sub_(step)
        return 2 * mat.Aex / (MU0 * mat.Ms * d * d) * H

    def rhs(self, m, x, v, t, only=None):
        """(dm / dt of both, H of both, acceleration of the slider)."""
        p = self.p
        u = (p.u0[0] + x / p.cell[0], p.u0[1], p.u0[2])
        dm, H, acc = [None, None], [None, None], 0.0
        for s in (0, 1):
            g, mat = 1 - s, self.mat[1 - s]
            if only is not None and g != only:
                continue
            path = _Path64(p, s, u)
            phi = path.potential(self.mat[s].Ms * m[s])
            h = -path.gradient(phi) + self.demag[g].field(mat.Ms * m[g]) + self.exchange(m[g], mat)
            h[2] += 2 * mat.Ku / (MU0 * mat.Ms) * m[g][2]
            c = _cross(m[g], h)
            dm[g] = -MU0 * GAMMA_LL / (1 + mat.alpha ** 2) * (c + mat.alpha * _cross(m[g], c))
            H[g] = h
            if g == 1:
                e = p.mech
                F = float(path.force(phi, mat.Ms * m[1])[0])
                acc = (e.k * (e.v_drive * t + e.x0_spring - x) - e.gamma_v * e.mass * v + F) / e.mass
        return dm, H, acc

    def steps(self, m, n, dt):
        A = ((1 / 5,), (3 / 40, 9 / 40), (44 / 45, -56 / 15, 32 / 9),
             (19372 / 6561, -25360 / 2187, 64448 / 6561, -212 / 729),
             (9017 / 3168, -355 / 33, 46732 / 5247, 49 / 176, -5103 / 18656),
             (35 / 384, 0.0, 500 / 1113, 125 / 192, -2187 / 6784, 11 / 84))
        C = (1 / 5, 3 / 10, 4 / 5, 8 / 9, 1.0, 1.0)
        y, t, k1 = [m[0], m[1], 0.0, self.p.mech.v_drive], 0.0, None

        def f(y, t):
            dm, _, acc = self.rhs(y[:2], y[2], y[3], t)
            return [dm[0], dm[1], y[3], acc]

        for _ in range(n):
            ks = [k1 or f(y, t)]
            for row, c in zip(A, C):
                z = [v + sum(dt * a * k[j] for a, k in zip(row, ks)) for j, v in enumerate(y)]
                ks.append(f(z, t + c * dt))
            y = [v / v.norm(dim=0, keepdim=True) for v in z[:2]] + z[2:]
            t, k1 = t + dt, ks[6]
        return y, t


def _eddy64(p, dB, sigma):
    n, d = p.n_base, p.cell[0]
    axes = [_Axis(k, 0, k) for k in n]
    conv = _Conv(_S_octant, _ODD_S, axes)

    def cross_sum(V):  # sum_j V(r_j) x S(r_i - r_j)
        f = conv.forward(V)
        return d * torch.stack([conv.back(conv.hat[(a + 2) % 3] * f[(a + 1) % 3] - conv.hat[(a + 1) % 3] * f[(a + 2) % 3])
                                for a in range(3)])

    E = -cross_sum(dB)
    b = torch.zeros_like(E[0])
    for a, dim in ((0, 2), (1, 1), (2, 0)):
        b.select(dim, n[a] - 1).sub_(E[a].select(dim, n[a] - 1) / d)
        b.select(dim, 0).add_(E[a].select(dim, 0) / d)
    b -= b.mean()
    # the cell-centred Neumann Laplacian is diagonal in the cosine basis
    phi, eig = b, 0.0
    basis = []
    for a in range(3):
        k, i = torch.arange(n[a], **_F64)[:, None], torch.arange(n[a], **_F64)[None]
        T = torch.cos(math.pi * k * (2 * i + 1) / (2 * n[a])) * math.sqrt(2 / n[a])
        T[0] /= math.sqrt(2)
        basis.append(T)
        e = (2 * torch.cos(math.pi * k[:, 0] / n[a]) - 2) / (d * d)
        eig = eig + e.reshape([-1 if j == 2 - a else 1 for j in range(3)])
    eig = eig.clone()
    eig[0, 0, 0] = 1.0
    phi = torch.einsum("pz,qy,rx,zyx->pqr", basis[2], basis[1], basis[0], phi) / eig
    phi[0, 0, 0] = 0.0
    phi = torch.einsum("pz,qy,rx,pqr->zyx", basis[2], basis[1], basis[0], phi)
    J = torch.empty_like(E)
    for a, dim in ((0, 2), (1, 1), (2, 0)):
        up, down = phi.roll(-1, dim), phi.roll(1, dim)  # ghosts by the boundary condition
        up.select(dim, n[a] - 1).copy_(phi.select(dim, n[a] - 1) + d * E[a].select(dim, n[a] - 1))
        down.select(dim, 0).copy_(phi.select(dim, 0) - d * E[a].select(dim, 0))
        J[a] = sigma * (E[a] - (up - down) / (2 * d))
    return dict(H=cross_sum(J), J=J, sweeps=None)


def exact(case, seed):
    pairs = _pairs_of(case)
    ms, extra = _inputs(case, seed)
    ms = [[m.double() for m in two] for two in ms]
    p, m, op = pairs[0], ms[0], case["op"]
    if op == "batch":
        got = []
        for q, mq in zip(pairs, ms):
            y, _ = _Pair64(q).steps(mq, case["steps"], _DT)
            got.append(y[:2])
        return dict(m=got)
    if op == "eddy":
        return _eddy64(p, extra.double(), _SIGMA)
    if op == "torque":
        dm, H, _ = _Pair64(p).rhs(m, 0.0, 0.0, 0.0, only=1)
        return dict(dm=dm[1], H=H[1])
    if op == "step":
        y, t = _Pair64(p).steps(m, case["steps"], _DT)
        return dict(m=y[:2], slider=torch.tensor([y[2], y[3], t], dtype=torch.float64))
    paths = [_Path64(p, s, p.u0) for s in (0, 1)]
    Ms = [mat.Ms for mat in (p.mat_base, p.mat_slider)]
    if op == "gradients":
        src, tgt = m[0].requires_grad_(), m[1].requires_grad_()
        phi = paths[0].potential(Ms[0] * src)
        V = MU0 * p.cell[0] ** 3
        E = V * Ms[1] * (paths[0].gradient(phi) * tgt).sum()
        gs, gt = torch.autograd.grad(E, (src, tgt))
        return dict(du=-paths[0].force(phi.detach(), Ms[1] * tgt.detach()), src=gs, tgt=gt)
    phi = [paths[s].potential(Ms[s] * m[s]) for s in (0, 1)]
    grad = [paths[s].gradient(phi[s]) for s in (0, 1)]
    return dict(H=[-grad[1], -grad[0]])
