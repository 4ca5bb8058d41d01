"""Performance cases of the B-TriRT solver: whole solves through the public classes.

A pass is what a user's program does with a lattice it keeps: set the initial field,
advance a number of steps, take phi back (``Lattice.init/step/phi``, ``Lattice3``,
``Batch``).  A case names the problem, the grid, the number of steps and the storage
options; ``prepare`` draws the physical coefficients and the initial field from the
seed, in the ranges of this repository's workloads.

Problems (``kind``), after the paper's tests and this repository's workloads:
  hill    advected anisotropic Gaussian hill, periodic, constant coefficients
  mms     manufactured solution between bounce-back walls, separable source
  modes   nonlinear fluxes and diffusion (B = u phi + phi^2/2 (1,1), A = (1 + phi^2) A0),
          periodic Fourier modes
  steady  diffusion between two walls marched towards its steady state, with the
          residual of every slice
  front   Burgers-Fisher front: power-law flux, reaction source, walls carrying the wave
  tensor  per-node diffusion tensor and per-node source
  hill3   the Gaussian hill on D3Q19
  state3  D3Q19, nonlinear, walls on y, constant source
  batch   independent hills and walled manufactured solutions of uneven size together
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1902_09813_gb300 import Batch, Lattice, Lattice3


def listed():
    return [
        # the 64^2 Gaussian hill of 500 steps, FP64: the smallest solve, bound by latency
        dict(name="hill_64_f64", kind="hill", nx=64, ny=64, steps=500, compute="f64", storage="f64", shift="ref"),
        # the headline workload: walled manufactured solution at 8192^2 in FP64
        dict(name="mms_8192_f64", kind="mms", nx=8192, ny=8192, steps=20, compute="f64", storage="f64", shift="ref"),
        # the nonlinear equation in FP64 on a ragged grid: reference runs of parameter studies
        dict(name="modes_1001x777_f64", kind="modes", nx=1001, ny=777, steps=40, compute="f64", storage="f64",
             shift="ref"),
        # the double-word format: FP64-class accuracy at FP32 rates, one size of the convergence sweep
        dict(name="mms_2048_df64", kind="mms", nx=2048, ny=2048, steps=50, compute="df64", storage="df64",
             shift="ref"),
        # FP32 storage, constant coefficients: the default of single-precision solves
        dict(name="mms_4096_f32", kind="mms", nx=4096, ny=4096, steps=100, compute="f32", storage="f32", shift="ref"),
        # the nonlinear workload at its full size with FP16 storage: the throughput format
        dict(name="modes_8192_f16", kind="modes", nx=8192, ny=8192, steps=100, compute="f32", storage="f16",
             shift="local"),
        # the accurate BF16 format on a ragged grid of the convergence sweep's size
        dict(name="mms_1023x1025_bf16", kind="mms", nx=1023, ny=1025, steps=200, compute="f32", storage="bf16",
             shift="moment_sr"),
        # a march to the steady state with a residual test every 100 steps: launches and host waits
        dict(name="steady_181x150_f32", kind="steady", nx=181, ny=150, steps=2000, slice=100, compute="f32",
             storage="f32", shift="ref"),
        # the three-dimensional lattice at its benchmark size, FP32 storage
        dict(name="hill3_384_f32", kind="hill3", nx=384, ny=384, nz=384, steps=20, compute="f32", storage="f32",
             shift="ref"),
        # three dimensions with FP16 storage, nonlinear with walls, ragged
        dict(name="state3_250x131x200_f16", kind="state3", nx=250, ny=131, nz=200, steps=40, compute="f32",
             storage="f16", shift="local"),
        # three dimensions in FP64, the default format
        dict(name="hill3_128_f64", kind="hill3", nx=128, ny=128, nz=128, steps=20, compute="f64", storage="f64",
             shift="ref"),
        # a serving slice: 64 uneven instances advanced 100 steps together
        dict(name="batch_64_f16", kind="batch", count=64, nmin=32, nmax=1024, steps=100, compute="f32",
             storage="f16", shift="local"),
    ]


# node-steps of the largest listed solves: FP64 and double-word, single precision, D3Q19
_CAP64, _CAP32, _CAP3 = 1.3e9, 6.7e9, 1.1e9
# forms of each storage format that a user picks
_FORMATS2 = [("f64", "f64", "ref"), ("f64", "f64", "ref"), ("df64", "df64", "ref"), ("f32", "f32", "ref"),
             ("f32", "f32", "local"), ("f32", "f32", "local_dw"), ("f32", "f16", "local"), ("f32", "f16", "local"),
             ("f32", "f16", "local_sr"), ("f32", "bf16", "local"), ("f32", "bf16", "moment_sr")]
_FORMATS3 = [("f64", "f64", "ref"), ("f32", "f32", "ref"), ("f32", "f32", "local"), ("f32", "f16", "local"),
             ("f32", "bf16", "local")]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.random()
    if what < 0.1:
        compute, storage, shift = rng.choice([("f32", "f16", "local"), ("f32", "bf16", "local"),
                                              ("f32", "f32", "ref"), ("f32", "f16", "local_sr"),
                                              ("f64", "f64", "ref")])
        return dict(kind="batch", count=rng.randint(16, 64), nmin=32, nmax=_log_int(rng, 256, 1024),
                    steps=rng.randint(20, 100), compute=compute, storage=storage, shift=shift)
    if what < 0.35:
        kind = rng.choice(["hill3", "state3"])
        nx, ny, nz = (_log_int(rng, 24, 384) for _ in range(3))
        compute, storage, shift = rng.choice(_FORMATS3)
        cap = _CAP3 * (0.25 if compute == "f64" else 1.0)
        steps = max(4, min(_log_int(rng, 10, 400), int(cap / (nx * ny * nz))))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, steps=steps, compute=compute, storage=storage, shift=shift)
    kind = rng.choice(["hill", "mms", "mms", "modes", "modes", "steady", "front", "tensor"])
    compute, storage, shift = rng.choice(_FORMATS2)
    most = {"steady": 1024, "front": 4096, "tensor": 1024}.get(kind, 8192)
    nx, ny = _log_int(rng, 32, most), _log_int(rng, 32, most)
    if kind == "mms":                       # the unit square: walls all round, nearly as many rows as columns
        ny = max(32, min(most, int(nx * rng.uniform(0.9, 1.1))))
    cap = (0.5 * _CAP64 if kind in ("modes", "front", "tensor") else _CAP64) if compute != "f32" else _CAP32 / 2
    steps = max(4, min(_log_int(rng, 10, 2000), int(cap / (nx * ny))))
    case = dict(kind=kind, nx=nx, ny=ny, steps=steps, compute=compute, storage=storage, shift=shift)
    if kind == "steady":
        case["slice"] = rng.choice([20, 50, 100])
    return case


# ---------------------------------------------------------------- problems
def _tensor2(l1, l2, th):
    c, s = math.cos(th), math.sin(th)
    return (l1 * c * c + l2 * s * s, (l1 - l2) * c * s, l1 * s * s + l2 * c * c)


def _problem(case, rng):
    """Everything of the case but the initial field: attributes as Lattice.from_problem takes them."""
    kind, nx, ny = case["kind"], case["nx"], case["ny"]
    p = SimpleNamespace(nx=nx, ny=ny, dx=1.0, dt=1.0, x0=0.0, y0=0.0, bc=(0, 0, 0, 0), u=(0.0, 0.0), b2=0.0,
                        b_dir=(1.0, 1.0), b_q=2.0, c3=0.0, A0=(0.0, 0.0, 0.0), a2=0.0, k0=1.0, k2_mode="hbb", k2=1.0,
                        source=SimpleNamespace(kind="none", const=0.0, exp=1.0, lam=0.0, k=math.pi,
                                               alpha=(0.0, 0.0, 0.0, 0.0)),
                        wall=(0.0, 0.0, 0.0, 0.0), wall_arrays=None, wall_lam=0.0, wall_fn=None, src_field=None,
                        A_field=None, t0=0.0, phi_ref=0.0)
    th, ang = rng.uniform(0.0, math.pi), rng.uniform(0.0, 2.0 * math.pi)
    if kind == "hill":
        p.A0 = _tensor2(*rng.uniform(0.005, 0.1, size=2), th)
        speed = rng.uniform(0.0, 0.1)
        p.u = (speed * math.cos(ang), speed * math.sin(ang))
    elif kind == "mms":
        kappa = 4.0
        p.dx = 1.0 / nx
        p.dt = kappa * p.dx * p.dx
        p.bc = (1, 1, 1, 1)
        p.A0 = _tensor2(rng.uniform(0.03, 0.06), rng.uniform(0.008, 0.02), th)
        p.u = tuple(rng.uniform(0.01, 0.06, size=2))
        pi, (axx, axy, ayy) = math.pi, p.A0
        p.source.kind, p.source.lam = "trig", -1.0
        p.source.alpha = (-1.0 + pi * pi * (axx + ayy), pi * p.u[1], pi * p.u[0], -2.0 * pi * pi * axy)
    elif kind == "modes":
        p.A0 = _tensor2(0.04, 0.008, th)
        p.u = (0.1 * math.cos(ang), 0.1 * math.sin(ang))
        p.b2, p.a2 = 1.0, 1.0
        p.dt = 0.05                          # 16 modes of amplitude up to 1/2: Courant number below 1/4 in the mean
    elif kind == "steady":
        alpha = rng.uniform(0.05, 0.15)
        p.dx = 1.0 / ny
        p.dt = p.dx * p.dx * (1.0 / 1.25 - 0.5) / (3.0 * alpha)
        p.bc = (0, 0, 1, 1)
        p.A0, p.u = (alpha, 0.0, alpha), (0.1, 0.0)
        p.wall = (0.0, 0.0, 0.0, rng.uniform(0.5, 1.5))
        p.source.kind, p.source.const = "const", 2.0 * alpha * p.wall[3]
    elif kind == "front":
        a, alpha, b, delta = rng.uniform(1.0, 2.0), rng.uniform(0.03, 0.06), 0.05, 1.5
        p.dx = 3.0 / max(nx, ny)
        p.dt = p.dx / 5.0
        p.x0 = p.y0 = -1.0
        p.bc = (1, 1, 1, 1)
        p.b2, p.b_dir, p.b_q = a, (1.0, 0.0), delta + 1.0
        p.A0 = (alpha, 0.0, alpha)
        p.source.kind, p.source.const, p.source.exp = "reaction", b, delta
        p.wave = -a * delta / (4.0 * alpha * (delta + 1.0))
        xs, ys = p.x0 + (np.arange(nx) + 0.5) * p.dx, p.y0 + (np.arange(ny) + 0.5) * p.dx
        sol = lambda s: (0.5 + 0.5 * np.tanh(p.wave * s)) ** (1.0 / delta)  # noqa: E731
        p.wall_arrays = [sol(p.x0 + ys), sol(p.x0 + nx * p.dx + ys), sol(xs + p.y0), sol(xs + p.y0 + ny * p.dx)]
    elif kind == "tensor":
        alpha = rng.uniform(0.5e-2, 2e-2)
        p.dx = 1.0 / nx
        p.dt = p.dx
        if alpha / p.dx > 0.5:               # the lattice diffusivity A dt / dx^2 stays moderate
            p.dt = 0.5 * p.dx * p.dx / alpha
        p.bc = (1, 1, 1, 1)
        p.u = tuple(rng.uniform(0.05, 0.1, size=2))
        p.A0 = (2.0 * alpha, 0.0, alpha)
        xs, ys = 2.0 * math.pi * (np.arange(nx) + 0.5) * p.dx, 2.0 * math.pi * (np.arange(ny) + 0.5) * p.dx
        ss = np.sin(ys)[:, None] * np.sin(xs)[None, :]
        p.A_field = (alpha * (2.0 - ss), np.zeros((ny, nx)), np.full((ny, nx), alpha))
        p.src_field = 0.1 * ss + 0.05 * np.cos(ys)[:, None] * np.sin(xs)[None, :]
        p.source.kind, p.source.lam = "field", -1.0
    return p


def _problem3(case, rng):
    p = SimpleNamespace(nx=case["nx"], ny=case["ny"], nz=case["nz"], dx=1.0, dt=1.0, x0=0.0, y0=0.0, z0=0.0,
                        bc=(0,) * 6, u=tuple(rng.uniform(-0.06, 0.06, size=3)), b2=0.0, b_dir=(1.0, 1.0, 1.0), b_q=2.0,
                        c3=0.0, a2=0.0, k0=1.0, k2_mode="hbb", k2=1.0,
                        source=SimpleNamespace(kind="none", const=0.0, exp=1.0, lam=0.0), src_field=None, wall=(0.0,) * 6,
                        wall_lam=0.0, phi_ref=0.0, t0=0.0)
    q, _ = np.linalg.qr(rng.standard_normal((3, 3)))
    m = (q * rng.uniform(0.01, 0.06, size=3)) @ q.T
    p.A0 = tuple(float(m[i, j]) for i, j in ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)))
    if case["kind"] == "state3":
        p.b2, p.c3, p.a2, p.k0 = 0.04, 0.02, 0.3, float(rng.uniform(0.8, 1.2))
        p.bc = (0, 0, 1, 1, 0, 0)
        p.wall = (0.0, 0.0, *(float(v) for v in rng.uniform(0.4, 1.0, size=2)), 0.0, 0.0)
        p.source.kind, p.source.const = "const", float(rng.uniform(-1e-3, 1e-3))
    return p


def _grid(n, d0, dx):
    return d0 + (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * dx


def _phi0(case, p, rng):
    """The initial field on the GPU, FP64."""
    kind = case["kind"]
    if kind in ("hill3", "state3"):
        ax = [_grid(n, 0.0, 1.0) for n in (p.nz, p.ny, p.nx)]
        if kind == "hill3":
            g = []
            for c, n in zip(ax, (p.nz, p.ny, p.nx)):
                mid, s0 = n * rng.uniform(0.4, 0.6), max(2.0, n / 16.0)
                g.append(torch.exp(-((c - mid) ** 2) / (2.0 * s0 * s0)))
            return g[0][:, None, None] * g[1][None, :, None] * g[2][None, None, :]
        out = torch.full((p.nz, p.ny, p.nx), float(rng.uniform(0.6, 0.9)), dtype=torch.float64, device="cuda")
        for _ in range(3):
            k, ph = rng.integers(1, 3, size=3), rng.uniform(0, 2 * math.pi, size=3)
            w = [torch.cos(2 * math.pi * int(k[i]) * ax[i] / (p.nz, p.ny, p.nx)[i] + ph[i]) for i in range(3)]
            out += float(rng.uniform(-0.1, 0.1)) * w[0][:, None, None] * w[1][None, :, None] * w[2][None, None, :]
        return out
    x, y = _grid(p.nx, p.x0, p.dx), _grid(p.ny, p.y0, p.dx)
    if kind == "hill":
        s0x, s0y = max(2.0, p.nx / 16.0), max(2.0, p.ny / 16.0)
        mx, my = p.nx * rng.uniform(0.4, 0.6), p.ny * rng.uniform(0.4, 0.6)
        return torch.exp(-((y - my) ** 2) / (2 * s0y * s0y))[:, None] * torch.exp(-((x - mx) ** 2) / (2 * s0x * s0x))
    if kind in ("mms", "tensor"):            # vanishing at the walls
        k = 1 if kind == "mms" else 2
        sx, sy = math.pi * _grid(p.nx, 0.0, 1.0 / p.nx), math.pi * _grid(p.ny, 0.0, 1.0 / p.ny)
        out = torch.sin(k * sy)[:, None] * torch.sin(k * sx)[None, :]
        for _ in range(3):
            i, j = rng.integers(1, 5, size=2)
            out += float(rng.uniform(-0.1, 0.1)) * torch.sin(int(j) * sy)[:, None] * torch.sin(int(i) * sx)
        return out
    if kind == "steady":
        return torch.zeros((p.ny, p.nx), dtype=torch.float64, device="cuda") + \
            float(rng.uniform(0.0, 0.1)) * (1.0 + torch.cos(2 * math.pi * x / (p.nx * p.dx)))
    if kind == "front":
        return (0.5 + 0.5 * torch.tanh(p.wave * (y[:, None] + x[None, :]))) ** (1.0 / 1.5)
    out = torch.zeros((p.ny, p.nx), dtype=torch.float64, device="cuda")
    for _ in range(16):                      # modes: cos(a + b) = cos a cos b - sin a sin b
        kx, ky = rng.integers(1, 9, size=2) * rng.choice([-1, 1], size=2)
        a = 2 * math.pi * int(kx) * x / p.nx
        b = 2 * math.pi * int(ky) * y / p.ny + float(rng.uniform(0, 2 * math.pi))
        amp = float(rng.uniform(-0.5, 0.5))
        out += amp * (torch.cos(b)[:, None] * torch.cos(a) - torch.sin(b)[:, None] * torch.sin(a))
    return out


def _inputs(case, seed):
    # a batch's sizes come from the case: the seed changes the instances' physics and fields
    rng = np.random.default_rng([seed, 17])
    if case["kind"] == "batch":
        sizes = np.random.default_rng(case["count"])
        out = []
        for k in range(case["count"]):
            n = int(round(math.exp(sizes.uniform(math.log(case["nmin"]), math.log(case["nmax"])))))
            c = dict(case, kind="hill" if k % 2 == 0 else "mms", nx=n, ny=n)
            p = _problem(c, rng)
            out.append((c, p, _phi0(c, p, rng)))
        return out
    p = (_problem3 if case["kind"] in ("hill3", "state3") else _problem)(case, rng)
    return p, _phi0(case, p, rng)


# ---------------------------------------------------------------- the user's program
def prepare(case, seed):
    form = dict(compute=case["compute"], storage=case["storage"], shift=case["shift"])
    if case["kind"] == "batch":
        members = _inputs(case, seed)
        lats = [Lattice.from_problem(p, **form).init(f, t0=p.t0) for _, p, f in members]
        batch = Batch(lats)
        batch.autotune()
        return SimpleNamespace(case=case, lats=lats, batch=batch, phi0=[f for _, _, f in members])
    p, phi0 = _inputs(case, seed)
    cls = Lattice3 if case["kind"] in ("hill3", "state3") else Lattice
    return SimpleNamespace(case=case, lat=cls.from_problem(p, **form), phi0=phi0, t0=p.t0)


def run(state):
    case = state.case
    if case["kind"] == "batch":
        for lat, phi0 in zip(state.lats, state.phi0):
            lat.init(phi0)
        state.batch.step(case["steps"])
        return [lat.phi() for lat in state.lats]
    lat = state.lat.init(state.phi0, t0=state.t0)
    if case["kind"] == "steady":
        done, resid = 0, []
        while done < case["steps"]:
            n = min(case["slice"], case["steps"] - done)
            resid.append(lat.step_residual(n))
            done += n
        return {"phi": lat.phi(), "residual": np.array(resid)}
    lat.step(case["steps"])
    return lat.phi()


def work(case):
    """Bytes: the initial field read, phi and the lattice's state (populations and phi plane) written once.
    Flops: the scheme's arithmetic per node and step (adds and multiplies, an FMA two), as the textbook
    moment form of Eq. 6 needs it with constant or per-node coefficients."""
    size = {"f64": 8, "df64": 8, "f32": 4, "f16": 2, "bf16": 2}
    real = 4 if case["compute"] == "f32" else 8
    if case["kind"] == "batch":
        sizes = np.random.default_rng(case["count"])
        nodes = sum(int(round(math.exp(sizes.uniform(math.log(case["nmin"]), math.log(case["nmax"]))))) ** 2
                    for _ in range(case["count"]))
    else:
        nodes = case["nx"] * case["ny"] * case.get("nz", 1)
    q = 19 if "nz" in case else 9
    per = {"hill": 70, "mms": 75, "steady": 70, "batch": 73, "modes": 150, "front": 180, "tensor": 150,
           "hill3": 165, "state3": 260}[case["kind"]]
    return {"bytes": nodes * (8 + real + q * size[case["storage"]] + real), "flops": nodes * case["steps"] * per}


# ---------------------------------------------------------------- the same in 64 bits with plain torch
_C9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_C19 = [(0, 0, 0)] + [tuple(s if i == a else 0 for i in range(3)) for a in range(3) for s in (1, -1)] + \
       [v for a, b in ((0, 1), (0, 2), (1, 2)) for v in
        [tuple(sa if i == a else sb if i == b else 0 for i in range(3)) for sb in (1, -1) for sa in (1, -1)]]


def _solve(p, phi0, steps, marks=()):
    """The scheme of Eq. 38 in population space and lattice units; returns phi and, for the step counts in
    `marks`, the 2-norm of that step's change of phi."""
    three = hasattr(p, "nz")
    C = _C19 if three else _C9
    dim, Q = len(C[0]), len(C)
    n2 = [sum(c * c for c in v) for v in C]
    w = [({0: 1 / 3, 1: 1 / 18, 2: 1 / 36} if three else {0: 4 / 9, 1: 1 / 9, 2: 1 / 36})[k] for k in n2]
    opp = [C.index(tuple(-c for c in v)) for v in C]
    shape, last = phi0.shape, phi0.dim() - 1
    s, sA = p.dt / p.dx, p.dt / (p.dx * p.dx)
    u = [v * s for v in p.u]
    bg = [p.b2 * s * d / p.b_q for d in p.b_dir]
    pairs = [(i, j) for i in range(dim) for j in range(i, dim)]
    A0 = {ij: a * sA for ij, a in zip(pairs, p.A0)}
    if getattr(p, "A_field", None) is not None:
        A0 = {ij: torch.tensor(np.asarray(a) * sA, device="cuda") for ij, a in zip(pairs, p.A_field)}
    src, field = p.source, None
    if src.kind == "field":
        field = torch.tensor(p.src_field, device="cuda")
    elif src.kind == "trig":
        x, y = _grid(p.nx, p.x0, p.dx), _grid(p.ny, p.y0, p.dx)
        a = src.alpha
        sx, cx, sy, cy = torch.sin(src.k * x), torch.cos(src.k * x), torch.sin(src.k * y), torch.cos(src.k * y)
        field = (a[0] * sy + a[1] * cy)[:, None] * sx + (a[2] * sy + a[3] * cy)[:, None] * cx

    def power(v, q):
        return v * v if q == 2.0 else v.clamp(min=0.0) ** q

    def flux(v):
        g = power(v, p.b_q) if p.b2 else 0.0
        return [u[d] * v + bg[d] * g if p.b2 else u[d] * v for d in range(dim)]

    def reaction(v):
        return src.const * v * (1.0 - power(v, src.exp))

    def collide(f, phi, prev, n, first):
        B = flux(phi)
        j = [sum((c[d] * f[i] for i, c in enumerate(C) if c[d]), 0.0 * phi) for d in range(dim)]
        dB = [torch.zeros_like(phi)] * dim if first else [b - a for b, a in zip(B, flux(prev))]
        scale = 1.0 + p.a2 * phi * phi if p.a2 else 1.0
        m = {ij: 3.0 * scale * a + (0.5 if ij[0] == ij[1] else 0.0) for ij, a in A0.items()}
        M = lambda i, k: m[(min(i, k), max(i, k))]  # noqa: E731
        tr = sum(M(i, i) for i in range(dim))
        if dim == 2:
            K = {(0, 0): M(1, 1), (0, 1): -M(0, 1), (1, 1): M(0, 0)}
            det = M(0, 0) * M(1, 1) - M(0, 1) * M(0, 1)
            k2 = 8.0 / 3.0 * (tr - 1.0) / (2.0 * tr - 1.0)
        else:
            K = {(i, k): M((i + 1) % 3, (k + 1) % 3) * M((i + 2) % 3, (k + 2) % 3)
                 - M((i + 1) % 3, (k + 2) % 3) * M((i + 2) % 3, (k + 1) % 3) for i, k in pairs}
            det = sum(M(0, k) * K[(0, k)] for k in range(3))
            k2 = 8.0 / 3.0 * (2.0 * tr - 3.0) / (4.0 * tr - 3.0)
        e = [B[d] - j[d] - 0.5 * dB[d] for d in range(dim)]
        V = [sum(K[(min(d, k), max(d, k))] * e[k] for k in range(dim)) / det + p.k0 * j[d] + dB[d] for d in range(dim)]
        Cm = p.c3 * phi ** 3 if p.c3 else 0.0
        N = {(a, b): sum(c[a] * c[b] * f[i] for i, c in enumerate(C) if c[a] and c[b]) for a, b in pairs}
        for d in range(dim):
            N[(d, d)] = N[(d, d)] - (phi + Cm) / 3.0
        t3 = sum(N[(d, d)] for d in range(dim)) / 3.0
        kap = 4.5 * (k2 - p.k0)
        tn = p.t0 + n * p.dt
        if src.kind in ("trig", "field"):
            Tn = math.exp(src.lam * tn)
            S = p.dt * 0.5 * (3.0 * Tn - (Tn if first else math.exp(src.lam * (tn - p.dt)))) * field
        elif src.kind == "reaction":
            Sn = reaction(phi)
            S = p.dt * (1.5 * Sn - 0.5 * (Sn if first else reaction(prev)))
        else:
            S = p.dt * src.const if src.kind == "const" else 0.0
        iso = p.k0 * phi + S
        for i, c in enumerate(C):
            H = -t3
            for a, b in pairs:
                if c[a] and c[b]:
                    H = H + (1.0 if a == b else 2.0) * c[a] * c[b] * N[(a, b)]
            g = iso - kap * H
            for d in range(dim):
                if c[d]:
                    g = g + 3.0 * c[d] * V[d]
            if p.c3:
                g = g + 1.5 * p.k0 * Cm * (n2[i] - (2.0 / 3.0 if dim == 2 else 1.0))
            f[i] = (1.0 - p.k0) * f[i] + w[i] * g
        return f

    walls = [(d, side) for d in range(dim) for side in (0, 1) if p.bc[2 * d]]

    def wall_value(d, side):
        arr = getattr(p, "wall_arrays", None)
        if arr is not None and arr[2 * d + side] is not None:
            v = torch.tensor(arr[2 * d + side], device="cuda")
            return v[:, None] if d == 0 else v[None, :]
        return torch.full((1,) * len(shape), float(p.wall[2 * d + side]), dtype=torch.float64, device="cuda")

    cross = {}
    for i, c in enumerate(C):                # nodes whose population i comes from beyond a wall, and its value
        val = torch.zeros(shape, dtype=torch.float64, device="cuda") if walls else None
        cnt = torch.zeros(shape, dtype=torch.float64, device="cuda") if walls else None
        for d, side in walls:
            if (c[d] == 1 and side == 0) or (c[d] == -1 and side == 1):
                at = [slice(None)] * len(shape)
                at[last - d] = slice(0, 1) if side == 0 else slice(shape[last - d] - 1, None)
                full = wall_value(d, side).expand(shape)
                val[tuple(at)] += full[tuple(at)]
                cnt[tuple(at)] += 1.0
        if walls and bool(cnt.any()):
            hit = cnt.nonzero(as_tuple=True)
            cross[i] = (hit, val[hit] / cnt[hit])
        del val, cnt

    phi = phi0.clone()
    B, Cm = flux(phi), (p.c3 * phi ** 3 if p.c3 else 0.0)
    f = [w[i] * (phi + 3.0 * sum(c[d] * B[d] for d in range(dim)) + 1.5 * Cm * (n2[i] - (2.0 / 3.0 if dim == 2 else 1.0)))
         for i, c in enumerate(C)]
    f = collide(f, phi, phi, 0, True)
    norms = []
    for n in range(1, steps + 1):
        fac = math.exp(p.wall_lam * (p.t0 + n * p.dt)) if p.wall_lam else 1.0
        bounced = {}
        for i, (hit, v) in cross.items():
            pw = v * fac
            dC = p.c3 * pw ** 3
            wt = 2.0 * w[i] * (pw + dC * ((3.0 * n2[i] - 2.0) * 0.5 if dim == 2 else 1.5 * (n2[i] - 1)))
            bounced[i] = wt - f[opp[i]][hit]
        for i, c in enumerate(C):
            if any(c):
                f[i] = torch.roll(f[i], c, dims=[last - d for d in range(dim)])
                if i in bounced:
                    f[i][cross[i][0]] = bounced[i]
        prev = phi
        phi = sum(f[1:], f[0])
        if n in marks:
            norms.append(float(torch.linalg.vector_norm(phi - prev)))
        f = collide(f, phi, prev, n, False)
    return phi, norms


def exact(case, seed):
    if case["kind"] == "batch":
        return [_solve(p, f, case["steps"])[0] for _, p, f in _inputs(case, seed)]
    p, phi0 = _inputs(case, seed)
    if case["kind"] == "steady":
        marks = list(range(case["slice"], case["steps"], case["slice"])) + [case["steps"]]
        phi, norms = _solve(p, phi0, case["steps"], marks)
        return {"phi": phi, "residual": np.array(norms)}
    return _solve(p, phi0, case["steps"])[0]
