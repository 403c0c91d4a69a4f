"""Performance cases of the framework: whole simulation runs and whole
differentiations through its public entry points, over the sizes, precision
forms and boundary kinds that its workloads have.

A pass of a simulation sets the initial state (``Lattice.init_equilibrium``),
takes a number of time steps (``Lattice.step``) and reads every field back
into device tensors (``Lattice.get``), as a parameter study does for each of
its points with one handle kept for the lattice.  A pass of a
differentiation runs the forward window and the reverse sweep, through
``autograd.run`` and ``backward`` or through the handle's own calls.

``exact`` restates the method in 64-bit torch for the inputs of a case (plain
gathers over the list of fluid cells, no code of the package's compute
path); the gradients come from torch's autograd through that restatement.
"""
import math

import numpy as np
import torch

from paper_1409_5645_gb300 import autograd, cases, fslbm

LIQ, IFC, GAS, WALL = 1, 2, 4, 8
FIELDS = ("flags", "f", "m", "phi", "rho", "u")


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the paper's film, the method's smallest use: 512 cells, a run of a few hundred
        # steps is all launches and latency; the FP64 form is the library's default
        dict(name="film_f64", kind="film", nx=4, ny=4, nz=32, precision="f64", rule=1, steps=400),
        # the convergence study's inclined film: link-wise (CLI) walls, shifted periodic
        # wrap, frozen interface
        dict(name="inclined_f64", kind="inclined", h=32, precision="f64", rule=1, steps=300),
        # the standing gravity-capillary wave at its own size: walled cube, surface tension
        # (curvature), FP64 as the reference run of the precision study ...
        dict(name="wave_f64", kind="wave", nx=128, ny=128, nz=128, precision="f64", rule=1, steps=25),
        # ... and FP16 storage as its reduced run
        dict(name="wave_f16", kind="wave", nx=128, ny=128, nz=128, precision="f16", loads="pairs", rule=1, steps=50),
        # a development-size splash (the benchmark's --small lattice), FP32
        dict(name="splash_small_f32", kind="splash", nx=128, ny=64, nz=64, precision="f32", loads="pairs", rule=1,
             steps=100),
        # rows that are no multiple of anything, the library's default loads, the first-order rule
        dict(name="splash_odd_f32", kind="splash", nx=187, ny=93, nz=101, precision="f32", loads="plain", rule=0,
             steps=60),
        # FP64 at a size that fills the chip
        dict(name="splash_f64", kind="splash", nx=256, ny=128, nz=128, precision="f64", rule=1, steps=25),
        # the throughput lattice, a developed splash with spray, both reduced forms
        dict(name="splash_large_f32", kind="splash", nx=512, ny=256, nz=256, precision="f32", loads="pairs", rule=1,
             steps=40),
        dict(name="splash_large_f16", kind="splash", nx=512, ny=256, nz=256, precision="f16", loads="pairs", rule=1,
             steps=40),
        # gradients of the surface velocity of a film, through torch.autograd
        dict(name="adjoint_film_f64", kind="adjoint_film", nx=8, ny=4, nz=64, precision="f64", rule=1, steps=200,
             K=50),
        # gradients through a splash with cell conversions, FP32 forward and reverse
        dict(name="adjoint_splash_f32", kind="adjoint_splash", nx=128, ny=64, nz=64, precision="f32", loads="pairs",
             rule=1, steps=16, K=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("film", "inclined", "wave", "splash", "splash", "splash", "adjoint_film", "adjoint_splash"))
    rule = 1 if kind.startswith("adjoint") else rng.choice((0, 1, 1))  # (FSK's populations do not see the fill levels)
    if kind == "film":
        return dict(kind=kind, nx=rng.randint(2, 9), ny=rng.randint(2, 9), nz=rng.randint(20, 80),
                    precision=rng.choice(("f64", "f32")), rule=rule, steps=_log_int(rng, 50, 400))
    if kind == "inclined":
        return dict(kind=kind, h=_log_int(rng, 8, 128), precision=rng.choice(("f64", "f64", "f32")), rule=rule,
                    steps=_log_int(rng, 50, 300))
    if kind == "adjoint_film":
        steps = rng.randint(40, 200)
        return dict(kind=kind, nx=rng.randint(4, 9), ny=rng.randint(3, 6), nz=rng.randint(40, 80),
                    precision=rng.choice(("f64", "f32")), rule=rule, steps=steps, K=rng.randint(20, 60))
    if kind == "adjoint_splash":
        return dict(kind=kind, nx=2 * _log_int(rng, 12, 64), ny=rng.randint(9, 64), nz=rng.randint(16, 64),
                    precision="f32", loads=rng.choice(("plain", "pairs")), rule=rule, steps=rng.randint(6, 16),
                    K=rng.randint(3, 8))
    if kind == "wave":
        nx = _log_int(rng, 24, 128)
        return dict(kind=kind, nx=nx, ny=nx + rng.randint(-5, 5), nz=nx, precision=rng.choice(("f64", "f32", "f16")),
                    loads=rng.choice(("plain", "pairs")), rule=rule, steps=rng.randint(10, 25))
    precision = rng.choice(("f64", "f32", "f32", "f16"))
    nx = _log_int(rng, 24, 256 if precision == "f64" else 512)
    if rng.random() < 0.5:
        nx += nx % 2  # even rows: the paired loads apply
    ny, nz = max(9, int(nx * rng.uniform(0.3, 0.5))), max(16, int(nx * rng.uniform(0.3, 0.5)))
    steps = int(min(100, max(10, 20 * (2 ** 23 / (nx * ny * nz)) ** 0.4)))
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, precision=precision, loads=rng.choice(("plain", "pairs", "pairs")),
                rule=rule, steps=steps)


# ---------------------------------------------------------------------------
# inputs (made on the GPU from the seed)
# ---------------------------------------------------------------------------
def _device():
    return torch.device("cuda", torch.cuda.current_device())


def _near_gas(gas):
    """Cells [z, y, x] with a gas cell along one of the 18 links; a face is no gas."""
    nz, ny, nx = gas.shape
    pad = torch.zeros((nz + 2, ny + 2, nx + 2), dtype=torch.bool, device=gas.device)
    pad[1:-1, 1:-1, 1:-1] = gas
    out = torch.zeros_like(gas)
    for cx, cy, cz in cases.LINKS[1:].tolist():
        out |= pad[1 + cz:1 + cz + nz, 1 + cy:1 + cy + ny, 1 + cx:1 + cx + nx]
    return out


def _walled(phi, surface, zc, g, params, u):
    """A walled box from fill levels [z, y, x]: kinds, hydrostatic density below ``surface``."""
    gas = phi <= 0.0
    ifc = ~gas & _near_gas(gas)
    flags = torch.where(gas, GAS, torch.where(ifc, IFC, LIQ)).to(torch.uint8)
    rho = 1.0 + 3.0 * g * torch.clamp(surface - zc, min=0.0)
    zero = torch.zeros((), dtype=torch.float64, device=phi.device)
    nz, ny, nx = phi.shape
    return dict(dims=(nx, ny, nz), params=params, flags=flags.reshape(-1),
                rho=torch.where(gas, zero + 1.0, rho).reshape(-1), u=torch.where(gas[..., None], zero, u).reshape(-1, 3),
                phi=torch.where(ifc, phi, zero).reshape(-1), noise=None, wall_delta=None)


def _grid(nx, ny, nz, dev):
    ax = [torch.arange(n, dtype=torch.float64, device=dev) + 0.5 for n in (nz, ny, nx)]
    return ax[0][:, None, None], ax[1][None, :, None], ax[2][None, None, :]


def _splash(case, seed, **params):
    """A developed dam break: a rough surface over about a fifth of the box,
    droplets of one to four cells' radius above it, velocities of a few hundredths."""
    dev, (nx, ny, nz) = _device(), (case["nx"], case["ny"], case["nz"])
    gen = torch.Generator(device=dev).manual_seed(seed)

    def uniform(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(shape, generator=gen, dtype=torch.float64, device=dev)

    zc, yc, xc = _grid(nx, ny, nz, dev)
    waves = torch.randint(1, 7, (6, 2), generator=gen, device=dev).to(torch.float64)
    amp, phase = uniform(0.01, 0.05, 6), uniform(0.0, 2 * math.pi, 6)
    h = torch.ones((1, ny, nx), dtype=torch.float64, device=dev)
    for k in range(6):
        h = h + amp[k] * torch.cos(2 * math.pi * (waves[k, 0] * xc / nx + waves[k, 1] * yc / ny) + phase[k])
    h = h * (0.19 * nz) + uniform(-0.5, 0.5, 1, ny, nx)
    phi = torch.clamp(h - (zc - 0.5), 0.0, 1.0)
    # droplets: each fills the cells of a 9 x 9 x 9 block around its centre
    count = max(2, nx * ny * nz // 40000)
    lo = torch.tensor([5.0, 5.0, 0.25 * nz], dtype=torch.float64, device=dev)
    hi = torch.tensor([nx - 5.0, ny - 5.0, nz - 5.0], dtype=torch.float64, device=dev)
    centre = lo + (hi - lo).clamp(min=0.0) * uniform(0.0, 1.0, count, 3)
    radius = uniform(1.0, 3.8, count)
    o = torch.arange(-4, 5, device=dev)
    block = torch.stack(torch.meshgrid(o, o, o, indexing="ij"), -1).reshape(1, -1, 3)
    cell = centre.floor().to(torch.int64)[:, None, :] + block
    size = torch.tensor([nx, ny, nz], device=dev)
    inside = ((cell >= 0) & (cell < size)).all(-1)
    r = (cell.to(torch.float64) + 0.5 - centre[:, None, :]).square().sum(-1).sqrt()
    fill = torch.where(inside, torch.clamp(radius[:, None] - r + 0.5, 0.0, 1.0), 0.0)
    at = torch.where(inside, cell[..., 0] + nx * (cell[..., 1] + ny * cell[..., 2]), 0)
    phi = phi.reshape(-1).scatter_reduce(0, at.reshape(-1), fill.reshape(-1), "amax").reshape(nz, ny, nx)
    phi = torch.where(phi > 0.0, phi.clamp(min=0.02), phi)
    phi = torch.where(phi > 0.0, phi + uniform(-1e-3, 1e-3, nz, ny, nx), phi)
    a, b = uniform(0.0, 2 * math.pi, 3), uniform(0.02, 0.04, 3)
    u = torch.stack([(b[0] * torch.sin(2 * math.pi * xc / nx + a[0]) + 0.0 * yc + 0.0 * zc),
                     (0.5 * b[1] * torch.sin(2 * math.pi * yc / ny + a[1]) + 0.0 * xc + 0.0 * zc),
                     (b[2] * torch.cos(2 * math.pi * xc / nx + 2 * math.pi * yc / ny + a[2]) + 0.0 * zc)], -1)
    p = dict(tau=0.53, magic=0.005, g=(0.0, 0.0, -1e-5), rule=case["rule"], bulk_loads=case.get("loads", "plain"))
    p.update(params)
    return _walled(phi, h, zc, 1e-5, cases.default_params(**p), u)


def _wave(case, seed):
    """The standing wave: surface at half height with a cosine of amplitude 2,
    fill noise 1e-4 on the interface, walls on every face, surface tension."""
    dev, (nx, ny, nz) = _device(), (case["nx"], case["ny"], case["nz"])
    gen = torch.Generator(device=dev).manual_seed(seed)
    zc, yc, xc = _grid(nx, ny, nz, dev)
    pt, wt = (torch.tensor(v, dtype=torch.float64, device=dev) for v in np.polynomial.legendre.leggauss(4))
    phi = torch.zeros((nz, ny, nx), dtype=torch.float64, device=dev)
    for i in range(4):
        for j in range(4):
            cosx = torch.cos(2 * math.pi * (xc + 0.5 * pt[i]) / nx)
            cosy = torch.cos(2 * math.pi * (yc + 0.5 * pt[j]) / ny)
            phi += 0.25 * wt[i] * wt[j] * torch.clamp(nz / 2 + 2.0 * cosx * cosy - (zc - 0.5), 0.0, 1.0)
    phi = torch.where(phi > 1.0 - 1e-12, 1.0, phi)
    noise = 1e-4 * (2.0 * torch.rand((nz, ny, nx), generator=gen, dtype=torch.float64, device=dev) - 1.0)
    phi = torch.where(phi > 0.0, (phi + noise).clamp(min=1e-3), phi)
    surface = nz / 2 + 2.0 * torch.cos(2 * math.pi * xc / nx) * torch.cos(2 * math.pi * yc / ny)
    p = cases.default_params(tau=0.55, g=(0.0, 0.0, -2e-5), sigma=1e-4, rule=case["rule"],
                             bulk_loads=case.get("loads", "plain"))
    return _walled(phi, surface, zc, 2e-5, p, torch.zeros((nz, ny, nx, 3), dtype=torch.float64, device=dev))


def _to_device(c):
    c = dict(c)
    for k in ("flags", "rho", "u", "phi", "noise", "wall_delta"):
        c[k] = None if c[k] is None else torch.as_tensor(c[k]).to(_device())
    return c


def _inputs(case, seed):
    kind = case["kind"]
    if kind in ("film", "adjoint_film"):
        g = 1e-6 if kind == "film" else 1e-4  # (the surface moves by a resolvable amount within the window)
        return _to_device(cases.film(nx=case["nx"], ny=case["ny"], nz=case["nz"], h=round(0.625 * case["nz"]), gx=g,
                                     rule=case["rule"], noise_amp=1e-8, seed=seed))
    if kind == "inclined":
        c = cases.inclined_film(h=case["h"], rule=case["rule"])
        c["noise"] = cases.uniform(seed, 19 * c.N, 1e-8)
        return _to_device(c)
    if kind == "wave":
        return _wave(case, seed)
    if kind == "adjoint_splash":
        return _splash(case, seed, tau=0.6, magic=3.0 / 16.0, adjoint_fp32=1)
    return _splash(case, seed)


# ---------------------------------------------------------------------------
# a pass
# ---------------------------------------------------------------------------
def prepare(case, seed):
    c = _inputs(case, seed)
    state = dict(case=case, inputs=c)
    if case["kind"] == "adjoint_film":
        dev = _device()
        state["leaves"] = [torch.tensor((c["params"]["tau"] - 0.5) / 3.0, dtype=torch.float64, requires_grad=True),
                           torch.tensor(c["params"]["g"], dtype=torch.float64, requires_grad=True),
                           c["phi"].to(dev).clone().requires_grad_(True)]
    else:
        extra = dict(keep_f0=1) if case["kind"] == "adjoint_splash" else {}
        state["lattice"] = fslbm.Lattice(c["dims"], dict(c["params"], **extra), precision=case["precision"])
    return state


def run(state):
    case, c = state["case"], state["inputs"]
    if case["kind"] == "adjoint_film":
        nu, g, phi0 = state["leaves"]
        for leaf in state["leaves"]:
            leaf.grad = None
        J = autograd.run(nu, g, phi0, c, case["steps"], K=case["K"], precision=case["precision"])
        J.backward()
        return dict(J=J.detach(), dnu=nu.grad, dg=g.grad, dphi0=phi0.grad)
    lat = state["lattice"]
    lat.init_equilibrium(c["flags"], c["rho"], c["u"], c["phi"], c["noise"], c["wall_delta"])
    if case["kind"] == "adjoint_splash":
        J = lat.adjoint_forward(case["steps"], case["K"])
        dnu, dg, dphi0 = lat.adjoint_backward(device=_device())
        return dict(J=J, dnu=dnu, dg=dg, dphi0=dphi0)
    lat.step(case["steps"])
    return lat.get(63, device=_device())


def work(case):
    """Bytes and operations a pass cannot do without: per step every fluid cell's
    19 populations read and written in the storage type and the cell kinds read
    once, the inputs read and the fields written in FP64; for a differentiation
    also the reverse steps, which read each state and read and write its adjoint
    in FP64.  (The fluid cells' share of a splash or a film is that of its generator.)"""
    kind, steps = case["kind"], case["steps"]
    n = 2 * case["h"] * (2 * case["h"] + 4) if kind == "inclined" else case["nx"] * case["ny"] * case["nz"]
    share = {"film": 0.625, "adjoint_film": 0.625, "inclined": 0.5, "wave": 0.5}.get(kind, 0.2)
    fluid = share * n
    s = {"f64": 8, "f32": 4, "f16": 2}[case["precision"]]
    step = fluid * 2 * 19 * s + n
    outer = n * (1 + 8 + 24 + 8)  # inputs: kinds, density, velocity, fill levels
    if kind.startswith("adjoint"):
        reverse = fluid * 19 * (s + 2 * 8) + n
        return {"bytes": 2 * steps * step + steps * reverse + outer + 8 * n, "flops": fluid * steps * (2 * 250 + 700)}
    noise = 19 * 8 * fluid if kind in ("film", "inclined") else 0
    return {"bytes": steps * step + outer + noise + n * (1 + 19 * 8 + 8 + 8 + 8 + 24), "flops": fluid * steps * 250}


# ---------------------------------------------------------------------------
# the method in 64-bit torch
# ---------------------------------------------------------------------------
C = cases.LINKS.tolist()
BAR = [0] + [q + 1 if q % 2 else q - 1 for q in range(1, 19)]
W = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12


def _dot(c, v):
    """c . v for a link c and three tensors (or numbers) v; None where c is 0."""
    out = None
    for a in range(3):
        if c[a]:
            term = v[a] if c[a] > 0 else -v[a]
            out = term if out is None else out + term
    return out


def _eplus(q, rho, u, usq):
    cu = _dot(C[q], u)
    return W[q] * (rho + 1.5 * ((0.0 if cu is None else 3.0 * cu * cu) - usq))


def _sq(u):
    return u[0] * u[0] + u[1] * u[1] + u[2] * u[2]


def _moments(f):
    j = [sum((C[q][a] * f[q] for q in range(19) if C[q][a])) for a in range(3)]
    return f.sum(0), j


class _Method:
    """One lattice in FP64: flags [N], f~ [19, N], m [N], phi [N]."""

    def __init__(self, c, lam=None, g=None):
        self.p = p = c["params"]
        self.nx, self.ny, self.nz = c["dims"]
        self.N = self.nx * self.ny * self.nz
        self.flags, self.wd = c["flags"], None if c["wall_delta"] is None else c["wall_delta"].reshape(19, -1)
        lp = -1.0 / p["tau"]
        self.lp, self.lm = lam if lam else (lp, -1.0 / (p["magic"] / (-(0.5 + 1.0 / lp)) + 0.5))
        self.g = g if g is not None else p["g"]
        self.frozen, self.sigma = bool(p["freeze"]), p["sigma"]

    def start(self, c, phi0):
        fluid = ((self.flags == LIQ) | (self.flags == IFC)).nonzero()[:, 0]
        rho, u = c["rho"][fluid], c["u"][fluid].T
        usq = _sq(u)
        f = torch.stack([_eplus(q, rho, u, usq) + (3.0 * W[q] * _dot(C[q], u) if q else 0.0) for q in range(19)])
        if c["noise"] is not None:
            f = f + c["noise"].reshape(19, -1)[:, fluid]
        rs = f.sum(0)
        zero = torch.zeros(self.N, dtype=torch.float64, device=f.device)
        ifc = self.flags[fluid] == IFC
        self.m = zero.index_copy(0, fluid, torch.where(ifc, phi0[fluid] * rs, zero[0]))
        keep = torch.where((self.flags == IFC) | ((self.flags == GAS) & self.frozen), phi0, zero)
        self.phi = keep.index_copy(0, fluid, torch.where(ifc, phi0[fluid] * rs / rs, zero[0]))
        self.f = f.new_zeros((19, self.N)).index_copy(1, fluid, self.collide(f)[0])

    def nbr(self, at, d):
        """Cells ``at`` + d, -1 past a face (the x wrap shifts z)."""
        px, py, pz = self.p["periodic"]
        x, y, z = at % self.nx + d[0], at // self.nx % self.ny + d[1], at // (self.nx * self.ny) + d[2]
        if px:
            z = z + self.p["zshift"] * ((x < 0).to(z.dtype) - (x >= self.nx).to(z.dtype))
            x = x % self.nx
        if py:
            y = y % self.ny
        if pz:
            z = z % self.nz
        ok = (x >= 0) & (x < self.nx) & (y >= 0) & (y < self.ny) & (z >= 0) & (z < self.nz)
        return torch.where(ok, x + self.nx * (y + self.ny * z), -1)

    def kind(self, j):
        return torch.where(j >= 0, self.flags[j.clamp(min=0)], WALL)

    def collide(self, f):
        rho, U = _moments(f)
        u = [U[a] + 0.5 * self.g[a] for a in range(3)]
        v = [U[a] - self.g[a] / self.lm for a in range(3)]
        usq = _sq(u)
        out = []
        for q in range(19):
            b = BAR[q]
            r = f[q] + self.lp * (0.5 * (f[q] + f[b]) - _eplus(q, rho, u, usq))
            if q:
                r = r + self.lm * (0.5 * (f[q] - f[b]) - 3.0 * W[q] * _dot(C[q], v))
            out.append(r)
        return torch.stack(out), rho

    def velocity(self, f):
        rho, j = _moments(f)
        return rho, [j[a] - 0.5 * self.g[a] for a in range(3)]

    # -- the interface plane --------------------------------------------------
    def level(self, at, d):
        """Fill level of cell at + d as the geometry sees it, and its kind."""
        j = self.nbr(at, d)
        k, raw = self.kind(j), self.phi[j.clamp(min=0)]
        stored = (k == IFC) | ((k == GAS) & self.frozen)
        return torch.where(k == LIQ, 1.0, torch.where(stored, raw, 0.0)), k

    def gradient(self, at, own):
        """The (negative) Parker-Youngs gradient."""
        n = [0.0, 0.0, 0.0]
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    if not (dx or dy or dz):
                        continue
                    v, k = self.level(at, (dx, dy, dz))
                    v = torch.where(k == WALL, own, v)
                    n[0] = n[0] - dx * (2 - abs(dy)) * (2 - abs(dz)) * v
                    n[1] = n[1] - dy * (2 - abs(dz)) * (2 - abs(dx)) * v
                    n[2] = n[2] - dz * (2 - abs(dx)) * (2 - abs(dy)) * v
        return torch.stack([v + 0.0 * own for v in n])

    def heights(self, at, a, s):
        """Column heights along axis a (gas side s) and whether every column is closed."""
        b = 1 if a == 0 else 0
        c = 3 - a - b
        H, closed = [], torch.ones_like(at, dtype=torch.bool)
        for ib in (-1, 0, 1):
            for ic in (-1, 0, 1):
                total = 0.0
                for k in range(-3, 4):
                    d = [0, 0, 0]
                    d[a], d[b], d[c] = k, ib, ic
                    v, kj = self.level(at, d)
                    closed = closed & (kj != WALL)
                    if abs(k) == 3:
                        closed = closed & (kj == torch.where(s * k < 0, LIQ, GAS))
                    total = total + v
                H.append(total)
        return torch.stack(H), closed, b, c

    @staticmethod
    def height_curvature(H):
        Hb, Hc = 0.5 * (H[7] - H[1]), 0.5 * (H[5] - H[3])
        Hbb, Hcc = H[7] - 2.0 * H[4] + H[1], H[5] - 2.0 * H[4] + H[3]
        Hbc = 0.25 * (H[8] - H[6] - H[2] + H[0])
        q2 = 1.0 + Hb * Hb + Hc * Hc
        return -(Hbb * (1.0 + Hc * Hc) + Hcc * (1.0 + Hb * Hb) - 2.0 * Hb * Hc * Hbc) / (q2 * torch.sqrt(q2))

    def open_curvature(self, at, n, a):
        """Heights along the two other axes, else the divergence of the unit gradient."""
        kap = torch.zeros_like(n[0])
        done = torch.zeros_like(at, dtype=torch.bool)
        mag = n.abs().scatter(0, a[None], -1.0)
        first = torch.where(mag.gather(0, ((a + 2) % 3)[None])[0] > mag.gather(0, ((a + 1) % 3)[None])[0],
                            (a + 2) % 3, (a + 1) % 3)
        for axes in (first, 3 - a - first):
            for ax in range(3):
                sub = (~done & (axes == ax)).nonzero()[:, 0]
                s = torch.where(n[ax][sub] > 0.0, 1, -1)
                H, closed, _, _ = self.heights(at[sub], ax, s)
                hit = sub[closed]
                kap[hit] = self.height_curvature(H[:, closed])
                done[hit] = True
        sub = (~done).nonzero()[:, 0]
        n0, div = n[:, sub], 0.0
        for d in range(3):
            side = []
            for sg in (-1, 1):
                step = [0, 0, 0]
                step[d] = sg
                j = self.nbr(at[sub], step)
                use = self.kind(j) != WALL
                jj = j.clamp(min=0)
                gj = self.gradient(jj, self.level(jj, (0, 0, 0))[0])
                use = use & (gj.norm(dim=0) > 1e-12)
                side.append(torch.where(use, gj[d] / gj.norm(dim=0).clamp(min=1e-300), n0[d] / n0.norm(dim=0)))
            div = div + 0.5 * (side[1] - side[0])
        kap[sub] = div
        return kap

    @staticmethod
    def volume(al, m1, m2, m3):
        """Volume below the plane m.x = al <= 1/2 in the unit cube (m sorted, sum 1) and its slope."""
        base, dbase, den = 3 * al * al - 3 * al * m1 + m1 * m1, 6 * al - 3 * m1, 6 * m2 * m3
        s, r, m12 = al - m2, al - m3, m1 + m2
        two, dtwo = base / den, dbase / den
        three, dthree = two - s * s * s / m1 / den, dtwo - 3 * s * s / m1 / den
        four, dfour = three - r * r * r / m1 / den, dthree - 3 * r * r / m1 / den
        late = torch.where(m3 >= m12, (al - 0.5 * m12) / m3, four)
        dlate = torch.where(m3 >= m12, 1.0 / m3, dfour)
        v = torch.where(al <= torch.minimum(m12, m3), three, late)
        dv = torch.where(al <= torch.minimum(m12, m3), dthree, dlate)
        v, dv = torch.where(al <= m2, two, v), torch.where(al <= m2, dtwo, dv)
        return (torch.where(al <= m1, al * al * al / (m1 * den), v),
                torch.where(al <= m1, 3 * al * al / (m1 * den), dv))

    def plane_offset(self, n, ph):
        """Offset of the plane with unit normal n that cuts the volume ph from the cell."""
        a = n.abs()
        L1 = a.sum(0)
        m1, m2, m3 = (a / L1).sort(0)[0].clamp(min=1e-13)
        ph = ph.clamp(1e-9, 1.0 - 1e-9)
        tv = torch.minimum(ph, 1.0 - ph)
        with torch.no_grad():
            lo, hi = torch.zeros_like(tv), torch.full_like(tv, 0.5)
            for _ in range(60):
                mid = 0.5 * (lo + hi)
                below = self.volume(mid, m1, m2, m3)[0] < tv
                lo, hi = torch.where(below, mid, lo), torch.where(below, hi, mid)
            root = 0.5 * (lo + hi)
        v, slope = self.volume(root, m1, m2, m3)
        al = root - (v - tv) / slope.detach()  # (the derivative of the implicit root)
        return L1 * (torch.where(ph > 0.5, 1.0 - al, al) - 0.5)

    def planes(self, at):
        """Unit normal, offset and curvature of the interface in the cells ``at``."""
        own = self.phi[at]
        py = self.gradient(at, own)
        flat = ~((py * py).sum(0) > 1e-24)
        a = torch.where(py[1].abs() > py[0].abs(), 1, 0)
        a = torch.where(py[2].abs() > torch.maximum(py[0].abs(), py[1].abs()), 2, a)
        n, d, kap = torch.zeros_like(py), torch.zeros_like(own), torch.zeros_like(own)
        for ax in range(3):
            sub = ((a == ax) & ~flat).nonzero()[:, 0]
            s = torch.where(py[ax][sub] > 0.0, 1, -1)
            H, closed, b, c = self.heights(at[sub], ax, s)
            hit, miss, H = sub[closed], sub[~closed], H[:, closed]
            v = [None] * 3
            v[ax], v[b], v[c] = s[closed] + 0.0 * H[0], -0.5 * (H[7] - H[1]), -0.5 * (H[5] - H[3])
            v = torch.stack(v)
            v = v / torch.sqrt((v * v).sum(0))
            n, d = n.index_copy(1, hit, v), d.index_copy(0, hit, v[ax].abs() * (H[4] - 3.5))
            g = py[:, miss]
            g = g / torch.sqrt((g * g).sum(0))
            n, d = n.index_copy(1, miss, g), d.index_copy(0, miss, self.plane_offset(g, own[miss]))
            if self.sigma:
                kap[hit] = self.height_curvature(H)
                kap[miss] = self.open_curvature(at[miss], py[:, miss], a[miss])
        return n, d, kap

    # -- one step --------------------------------------------------------------
    def step(self):
        p, flags = self.p, self.flags
        fluid = ((flags == LIQ) | (flags == IFC)).nonzero()[:, 0]
        on = (flags[fluid] == IFC).nonzero()[:, 0]  # the interface cells among them
        at = fluid[on]
        own = self.f[:, fluid]
        pulled, wall, gas, liquid, src = [own[0]], [None], [None], [None], [None]
        for q in range(1, 19):
            j = self.nbr(fluid, [-v for v in C[q]])
            k = self.kind(j)
            hit = (k == LIQ) | (k == IFC)
            pulled.append(torch.where(hit, self.f[q][j.clamp(min=0)], 0.0))
            wall.append(k == WALL)
            gas.append((k == GAS)[on])
            liquid.append((k == LIQ)[on])
            src.append(j[on])
        # mass exchange with the pulled values
        dm = torch.zeros_like(own[0][on])
        phi = self.phi[at]
        for q in range(1, 19):
            weight = torch.where(liquid[q], 1.0, 0.5 * (phi + self.phi[src[q].clamp(min=0)]))
            flux = weight * (pulled[q][on] - own[BAR[q]][on])
            dm = dm + torch.where(wall[q][on] | gas[q], 0.0, flux)
        # walls: half-way bounce-back, or the link-wise rule where a fraction is given
        f = list(pulled)
        for q in range(1, 19):
            b = BAR[q]
            back = own[b]
            if self.wd is not None:
                dw = self.wd[b][fluid]
                up = ~wall[b]
                up[on] = up[on] & ~gas[b]
                kap = (1.0 - 2.0 * dw) / (1.0 + 2.0 * dw)
                back = torch.where((dw >= 0.0) & up, back + kap * (pulled[b] - own[q]), back)
            f[q] = torch.where(wall[q], back, pulled[q])
        # gas links of the interface cells
        rt, ut = self.velocity(own[:, on])
        usq = _sq(ut)
        n, d, kap = self.planes(at)
        rb = p["rho_G"] + 3.0 * self.sigma * kap
        for q in range(1, 19):
            b = BAR[q]
            op, oq = own[b][on], own[q][on]
            eb = _eplus(b, rb, ut, usq)
            fsk = -op + 2.0 * eb
            new = fsk
            if p["rule"] == 1:
                cn = _dot(C[b], n)
                ahead = cn > 0.0
                dl = torch.where(ahead, (d / torch.where(ahead, cn, 1.0)).clamp(p["delta_min"], 1.0), 0.5)
                nplus = (0.5 * (op + oq) - _eplus(b, rt, ut, usq)) / (1.0 + self.lp)
                fsl = (0.5 - dl) * op + 0.5 * oq + (dl - 1.0) * f[b][on] + self.lp * (dl - 1.5) * nplus + eb
                new = torch.where(wall[b][on] | gas[b], fsk, fsl)
            f[q] = f[q].index_copy(0, on, torch.where(gas[q], new, f[q][on]))
        out, rho = self.collide(torch.stack(f))
        nxt = self.f.new_zeros((19, self.N)).index_copy(1, fluid, out)
        if self.frozen:
            self.f = nxt
            return
        rho, mm = rho[on], self.m[at] + dm
        no_gas = ~torch.stack(gas[1:]).any(0)
        alone = torch.stack([wall[q][on] | gas[q] for q in range(1, 19)]).all(0)
        fill = (mm > (1.0 + p["eps"]) * rho) | no_gas
        empty = ~fill & ((mm < -p["eps"] * rho) | alone)
        m, phi = self.m.index_copy(0, at, mm), self.phi.index_copy(0, at, mm / rho)
        self.convert(nxt, m, phi, at[fill], at[empty])

    def around(self, cells):
        return torch.stack([self.nbr(cells, C[q]) for q in range(1, 19)])

    def convert(self, f, m, phi, F, E):
        flags, N, dev = self.flags, self.N, f.device
        mark = torch.zeros(N, dtype=torch.bool, device=dev)
        mark[F] = True
        E = E[~(mark[self.around(E).clamp(min=0)] & (self.around(E) >= 0)).any(0)]

        def neighbours(cells, kind):
            j = self.around(cells).reshape(-1)
            j = j[j >= 0]
            return j[flags[j] == kind].unique()

        G, L = neighbours(F, GAS), neighbours(E, LIQ)
        if G.numel():  # equilibrium at the mean of the fluid neighbours
            j = self.around(G)
            k = self.kind(j)
            use = ((k == LIQ) | (k == IFC)).to(torch.float64)
            rho, u = self.velocity(f[:, j.clamp(min=0)])
            count = use.sum(0)
            rbar, ubar = (rho * use).sum(0) / count, [(v * use).sum(0) / count for v in u]
            usq = _sq(ubar)
            eq = torch.stack([_eplus(q, rbar, ubar, usq) + (3.0 * W[q] * _dot(C[q], ubar) if q else 0.0)
                              for q in range(19)])
            f = f.index_copy(1, G, self.collide(eq)[0])
            m, phi = m.index_fill(0, G, 0.0), phi.index_fill(0, G, 0.0)
        rho = f[:, L].sum(0)
        m, phi = m.index_copy(0, L, rho), phi.index_copy(0, L, rho / rho)
        conv = torch.cat([F, E])
        rho = f[:, conv].sum(0)
        filled = torch.arange(conv.numel(), device=dev) < F.numel()
        excess = torch.where(filled, m[conv] - rho, m[conv])
        m = m.index_copy(0, conv, torch.where(filled, rho, torch.zeros_like(rho)))
        takes = flags == IFC
        takes[conv] = False
        takes[G], takes[L] = True, True
        j = self.around(conv)
        give = (j >= 0) & takes[j.clamp(min=0)]
        count = give.sum(0)
        share = torch.where(count > 0, excess / count.clamp(min=1), 0.0)
        got = torch.zeros_like(m).index_add(0, j[give], share.expand(18, -1)[give])
        m = m + got
        R = j[give].unique()
        phi = phi.index_copy(0, R, m[R] / f[:, R].sum(0)).index_fill(0, E, 0.0)
        flags = flags.clone()
        flags[F], flags[E], flags[G], flags[L] = LIQ, GAS, IFC, IFC
        self.flags, self.f, self.m, self.phi = flags, f, m, phi

    def fields(self):
        liq, ifc = self.flags == LIQ, self.flags == IFC
        fluid = (liq | ifc).to(torch.float64)
        rho, u = self.velocity(self.f)
        zero = torch.zeros_like(rho)
        level = torch.where(liq, 1.0, torch.where(ifc | ((self.flags == GAS) & self.frozen), self.phi, zero))
        return dict(flags=None, f=self.f * fluid, m=torch.where(ifc, self.m, rho * liq), phi=level, rho=rho * fluid,
                    u=(torch.stack(u, -1) * fluid[:, None]))


def exact(case, seed):
    c = _inputs(case, seed)
    if not case["kind"].startswith("adjoint"):
        with torch.no_grad():
            sim = _Method(c)
            sim.start(c, c["phi"])
            for _ in range(case["steps"]):
                sim.step()
            return sim.fields()
    p, dev = c["params"], _device()
    nu = torch.tensor((p["tau"] - 0.5) / 3.0, dtype=torch.float64, device=dev, requires_grad=True)
    g = torch.tensor(p["g"], dtype=torch.float64, device=dev, requires_grad=True)
    phi0 = c["phi"].clone().requires_grad_(True)
    tau = 3.0 * nu + 0.5
    sim = _Method(c, (-1.0 / tau, -1.0 / (p["magic"] / (tau - 0.5) + 0.5)), g)
    sim.start(c, phi0)
    for _ in range(case["steps"]):
        sim.step()
    surface = (sim.flags == IFC).nonzero()[:, 0]
    J = sim.velocity(sim.f[:, surface])[1][0].mean()
    J.backward()
    if case["kind"] == "adjoint_splash":
        # (the slope in a fill level depends on which branch the plane of its cell takes, and at a
        # few cells the reduced forms' rounding decides that: no 64-bit value stands for them)
        return dict(J=J.detach(), dnu=float(nu.grad), dg=g.grad, dphi0=None)
    return dict(J=J.detach(), dnu=nu.grad, dg=g.grad, dphi0=torch.where(c["flags"] == IFC, phi0.grad, 0.0))
