"""Performance cases of the hyperbolic self-gravity framework: what a program that uses it has it do.

Four kinds of work, each through the public entry points (paper_1602_05700_gb300.Grid, Batch, Hydro, autograd):

  gravity   the gravity of one hydro step: set_density, wave sub-steps, -grad phi, phi (rho frozen over the sub-steps);
            with "restart" the potential starts from zero on every pass (a relaxation run)
  batch     many independent grids of uneven sides and both precisions advanced together (Batch.step)
  adjoint   forward sub-steps from phi = 0 and dL/drho of a probe loss, by autograd (FP64) or Grid.adjoint (float)
  hydro     a short coupled run of a star: primitive initial state, hydro steps (density hand-over, sub-steps,
            -grad phi, two Runge-Kutta stages), the characteristic speed the next step's Courant limit needs

Boxes are centred on the origin with their longest side 1; densities are seeded spheres, Gaussian blobs or a Plummer
star.  `exact` is a plain float64 torch evaluation of the same discrete scheme.
"""
from __future__ import annotations

import math
import random

import torch
import torch.nn.functional as F

import paper_1602_05700_gb300 as hg
from paper_1602_05700_gb300 import autograd

DEV = "cuda"
F64 = torch.float64


def listed():
    return [
        # the plain method: FP64, uniform sphere, analytic -GM/r boundary, relaxed from zero in many small sub-steps
        dict(name="relax_f64_32", kind="gravity", nx=32, ny=32, nz=32, prec="f64", bc="dirichlet", lmax=0, depth=1,
             substeps=200, shape="sphere", restart=True),
        # the smallest production step: one coarse grid (or one patch), bound by latency
        dict(name="step_f32k_64_robin", kind="gravity", nx=64, ny=64, nz=64, prec="f32k", bc="robin", lmax=0, depth=1,
             substeps=20, shape="blobs", restart=False),
        # the lag study's box: periodic, mean density removed
        dict(name="step_f32k_128_periodic", kind="gravity", nx=128, ny=128, nz=128, prec="f32k", bc="periodic", lmax=0,
             depth=1, substeps=20, shape="blobs", restart=False),
        # an ordinary box whose sides divide nothing
        dict(name="step_f32k_ragged", kind="gravity", nx=301, ny=259, nz=223, prec="f32k", bc="robin", lmax=0, depth=1,
             substeps=17, shape="blobs", restart=False),
        # the precision workload (multipole boundary data, l <= 4) in both precisions
        dict(name="step_f32k_256_multipole", kind="gravity", nx=256, ny=256, nz=256, prec="f32k", bc="multipole",
             lmax=4, depth=1, substeps=20, shape="blobs", restart=False),
        dict(name="step_f64_256_multipole", kind="gravity", nx=256, ny=256, nz=256, prec="f64", bc="multipole", lmax=4,
             depth=1, substeps=20, shape="blobs", restart=False),
        # the time-dependent workload: the largest grid, fused sub-steps
        dict(name="step_f32k_512_depth2", kind="gravity", nx=512, ny=512, nz=512, prec="f32k", bc="robin", lmax=0,
             depth=2, substeps=20, shape="blobs", restart=False),
        # the batching workload
        dict(name="batch_48_mixed", kind="batch", grids=48, side_seed=7, side_min=64, side_max=192, side_step=32,
             substeps=50),
        # the differentiation workload in both precisions
        dict(name="adjoint_f32k_128", kind="adjoint", n=128, prec="f32k", bc="robin", T=100, probes=64),
        dict(name="adjoint_f64_128", kind="adjoint", n=128, prec="f64", bc="robin", T=100, probes=64),
        # the virial workload: the paper's 3D star resolution in float, the reference precision on a smaller box
        dict(name="hydro_f32_280", kind="hydro", nx=280, ny=280, nz=280, dtype="f32", prec="f32k", bc="robin",
             steps=2, nsub=6),
        dict(name="hydro_f64_96", kind="hydro", nx=96, ny=96, nz=96, dtype="f64", prec="f64", bc="robin", steps=2,
             nsub=6),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _sides(rng, lo, hi):
    n = _log_int(rng, lo, hi)
    return [max(lo, min(hi, int(n * rng.uniform(0.7, 1.3)))) for _ in range(3)]


def draw(rng):
    kind = rng.choice(["gravity", "gravity", "gravity", "gravity", "batch", "adjoint", "hydro"])
    if kind == "gravity":
        prec = rng.choice(["f32k", "f32k", "f64"])
        bc = rng.choice(["robin", "robin", "multipole", "periodic", "dirichlet"])
        nx, ny, nz = _sides(rng, 24, 400 if prec == "f32k" else 224)
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, prec=prec, bc=bc, lmax=rng.randint(1, 4) if bc == "multipole" else 0,
                    depth=2 if prec == "f32k" and bc == "robin" and rng.random() < 0.5 else 1,
                    substeps=rng.randint(5, 20), shape=rng.choice(["blobs", "sphere"]), restart=rng.random() < 0.25)
    if kind == "batch":
        return dict(kind=kind, grids=rng.randint(3, 32), side_seed=rng.randint(0, 10 ** 6), side_min=rng.randint(33, 64),
                    side_max=rng.randint(96, 176), side_step=rng.choice([1, 7, 16]), substeps=rng.randint(22, 40))
    if kind == "adjoint":
        return dict(kind=kind, n=_log_int(rng, 40, 128), prec=rng.choice(["f32k", "f64"]),
                    bc=rng.choice(["robin", "periodic", "dirichlet"]), T=rng.randint(20, 100), probes=rng.randint(16, 128))
    dtype = rng.choice(["f32", "f32", "f64"])
    nx, ny, nz = _sides(rng, 32, 240 if dtype == "f32" else 96)
    return dict(kind=kind, nx=nx, ny=ny, nz=nz, dtype=dtype, prec="f64" if dtype == "f64" else "f32k", bc="robin",
                steps=rng.randint(1, 3), nsub=rng.randint(4, 9))


# ---- inputs ---------------------------------------------------------------------------------------------------------

def _box(nx, ny, nz):
    """(h, origin, nu): longest side 1, centred; nu = 0.5 / sqrt 3 or what the Robin boundary of a flat box allows."""
    h = 1.0 / max(nx, ny, nz)
    half = [0.5 * (n + 1) for n in (nx, ny, nz)]
    mu = min(half) / math.sqrt(sum(v * v for v in half))
    return h, (-0.5 * nx * h, -0.5 * ny * h, -0.5 * nz * h), min(0.5 / math.sqrt(3.0), 0.9 * mu)


def _axes(nx, ny, nz, h, ghost=0):
    """Cell-centre coordinates as broadcastable x, y, z (FP64); ghost = 1 adds one cell on each side."""
    def ax(n):
        return (torch.arange(-ghost, n + ghost, dtype=F64, device=DEV) + 0.5) * h - 0.5 * n * h
    return ax(nx)[None, None, :], ax(ny)[None, :, None], ax(nz)[:, None, None]


def _bodies(case, seed):
    """Seeded compact sources inside the box: (centre, width, peak) of 4 Gaussian blobs, or one sphere."""
    r = random.Random(seed * 7919 + 13)
    if case.get("shape") == "sphere":
        return [((0.0, 0.0, 0.0), r.uniform(0.2, 0.28), r.uniform(0.8, 1.2))]
    out = []
    for _ in range(4):
        out.append(([r.uniform(-0.17, 0.17) for _ in range(3)], r.uniform(0.02, 0.08), r.uniform(0.1, 2.0)))
    return out


def _density(shape, bodies, nx, ny, nz, h):
    x, y, z = _axes(nx, ny, nz, h)
    lim = [0.5 * n * h for n in (nx, ny, nz)]
    rho = torch.zeros(nz, ny, nx, dtype=F64, device=DEV)
    for c, w, a in bodies:
        c = [2 * v * m for v, m in zip(c, lim)]  # centres scale with the box
        if shape == "sphere":
            rho += a * ((x * x + y * y + z * z) < (2 * w * min(lim)) ** 2)
        else:
            e = [torch.exp(-(q - v) ** 2 / (2 * w * w)) for q, v in zip((x, y, z), c)]
            rho += a * (e[2] * e[1]) * e[0]
    return rho


def _potential(shape, bodies, rho, bc, nx, ny, nz, h):
    """The Poisson potential of the bodies, to start the wave solution from."""
    if bc == "periodic":
        k = [4.0 / h ** 2 * torch.sin(math.pi * torch.fft.fftfreq(n, dtype=F64, device=DEV)) ** 2 for n in (nx, ny, nz)]
        lam = k[2][:, None, None] + k[1][None, :, None] + k[0][None, None, :]
        lam[0, 0, 0] = 1.0
        f = torch.fft.fftn(4 * math.pi * (rho - rho.mean())) / -lam
        f[0, 0, 0] = 0.0
        return torch.fft.ifftn(f).real.contiguous()
    x, y, z = _axes(nx, ny, nz, h)
    lim = [0.5 * n * h for n in (nx, ny, nz)]
    phi = torch.zeros(nz, ny, nx, dtype=F64, device=DEV)
    for c, w, a in bodies:
        c = [2 * v * m for v, m in zip(c, lim)]
        r = torch.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2).clamp_(min=1e-9)
        if shape == "sphere":
            R = 2 * w * min(lim)
            phi -= torch.where(r < R, 2 * math.pi * a * (R * R - r * r / 3), 4 * math.pi / 3 * a * R ** 3 / r)
        else:
            phi -= a * (2 * math.pi) ** 1.5 * w ** 3 * torch.erf(r / (math.sqrt(2.0) * w)) / r
    return phi


def _gravity_inputs(case, seed):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    h, origin, nu = _box(nx, ny, nz)
    bodies = _bodies(case, seed)
    rho = _density(case["shape"], bodies, nx, ny, nz, h)
    phi = torch.zeros_like(rho) if case["restart"] else _potential(case["shape"], bodies, rho, case["bc"], nx, ny, nz, h)
    return rho.to(F64 if case["prec"] == "f64" else torch.float32), phi, h, origin, nu


def _batch_inputs(case, seed):
    r = random.Random(case["side_seed"])
    sides = list(range(case["side_min"], case["side_max"] + 1, case["side_step"]))
    out = []
    for i in range(case["grids"]):
        n, prec = r.choice(sides), ("f32k", "f64")[i % 2]
        rho = _density("blobs", _bodies({}, seed * 101 + i), n, n, n, 1.0 / n)
        out.append((n, prec, rho.to(F64 if prec == "f64" else torch.float32)))
    return out


def _adjoint_inputs(case, seed):
    n, dt = case["n"], F64 if case["prec"] == "f64" else torch.float32
    h, origin, nu = _box(n, n, n)
    rho = _density("blobs", _bodies({}, seed), n, n, n, h).to(dt)
    r = random.Random(seed * 31 + 5)
    dL = torch.zeros(n, n, n, dtype=F64)  # d/dphi of a squared misfit at probe points: their trilinear cells
    for _ in range(case["probes"]):
        u = [(0.5 + r.uniform(-0.4, 0.4)) * n - 0.5 for _ in range(3)]
        i0, g = [int(v) for v in u], r.gauss(0.0, 1.0)
        for b in range(8):
            w, at = g, []
            for a in range(3):
                hi = b >> a & 1
                f = u[a] - i0[a]
                w *= f if hi else 1.0 - f
                at.append(min(i0[a] + hi, n - 1))
            dL[at[2], at[1], at[0]] += w
    return rho, dL.to(DEV).to(dt), h, origin, nu


GAMMA, K_G, STAR = 5.0 / 3.0, 5.0, 0.1


def _hydro_inputs(case, seed):
    """A perturbed Plummer star (closed-form hydrostatic pressure and potential) with a slow rotation."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    h, origin, nu = _box(nx, ny, nz)
    x, y, z = _axes(nx, ny, nz, h)
    s2 = x * x + y * y + z * z + STAR * STAR
    phi = -1.0 / torch.sqrt(s2)
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    rho = 3.0 * STAR ** 2 / (4.0 * math.pi) * s2 ** -2.5
    P = -rho * phi / 6.0
    rho = rho * (1.0 + 0.01 * (2.0 * torch.rand(nz, ny, nx, dtype=F64, device=DEV, generator=gen) - 1.0))
    spin = random.Random(seed).uniform(0.2, 0.6)
    W = torch.stack([rho, -spin * y * torch.exp(-s2 / 0.02) + 0 * rho, spin * x * torch.exp(-s2 / 0.02) + 0 * rho,
                     0.01 * torch.sin(40.0 * z) + 0 * rho, P]).to(F64 if case["dtype"] == "f64" else torch.float32)
    Wd = W.double()
    speed = (torch.sqrt(Wd[1] ** 2 + Wd[2] ** 2 + Wd[3] ** 2) + torch.sqrt(GAMMA * Wd[4] / Wd[0])).max().item()
    c = K_G * speed
    dtg = 0.6 * nu * h / c  # Courant number 0.3 (0.5 is nu = 0.5 / sqrt 3)
    return W, phi, h, origin, c, dtg


# ---- the passes -----------------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "gravity":
        rho, phi, h, origin, nu = _gravity_inputs(case, seed)
        g = hg.Grid(case["nx"], case["ny"], case["nz"], h, origin, 1.0, 1.0, nu * h, case["prec"], case["bc"], case["lmax"])
        if case["depth"] > 1:
            g.set_temporal_depth(case["depth"])
        g.set_density(rho)
        g.set_phi(phi)
        return dict(case=case, g=g, rho=rho, phi=phi if case["restart"] else None)
    if kind == "batch":
        grids = []
        for n, prec, rho in _batch_inputs(case, seed):
            g = hg.Grid.unit_cube(n, precision=prec, bc="robin")
            g.set_density(rho)
            grids.append(g)
        return dict(case=case, grids=grids, batch=hg.Batch(grids))
    if kind == "adjoint":
        rho, dL, h, origin, nu = _adjoint_inputs(case, seed)
        n = case["n"]
        g = hg.Grid(n, n, n, h, origin, 1.0, 1.0, nu * h, case["prec"], case["bc"])
        return dict(case=case, g=g, rho=rho, dL=dL, zero=torch.zeros_like(rho))
    W, phi, h, origin, c, dtg = _hydro_inputs(case, seed)
    g = hg.Grid(case["nx"], case["ny"], case["nz"], h, origin, c, 1.0, dtg, case["prec"], case["bc"])
    H = hg.Hydro(case["nx"], case["ny"], case["nz"], h, GAMMA, 1e-12, 1e-14, case["dtype"])
    return dict(case=case, g=g, H=H, W=W, phi=phi, dt=case["nsub"] * dtg)


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "gravity":
        g = state["g"]
        g.set_density(state["rho"])
        if state["phi"] is not None:
            g.set_phi(state["phi"])
        g.step(case["substeps"])
        return {"accel": g.accel(), "phi": g.phi(state["rho"].dtype)}
    if kind == "batch":
        state["batch"].step(case["substeps"])
        return [g.phi(F64 if g.precision == hg.PREC["f64"] else torch.float32) for g in state["grids"]]
    if kind == "adjoint":
        g = state["g"]
        if case["prec"] == "f64":
            rho = state["rho"].detach().requires_grad_(True)
            phi = autograd.potential(rho, g, case["T"])
            (grad,) = torch.autograd.grad(phi, rho, state["dL"])
            return {"phi": phi.detach(), "grad": grad}
        g.set_density(state["rho"])
        g.set_phi(state["zero"])
        g.step(case["T"])
        return {"phi": g.phi(torch.float32), "grad": g.adjoint(state["dL"], case["T"])}
    g, H = state["g"], state["H"]
    H.set_primitive(state["W"])
    g.set_phi(state["phi"])
    for _ in range(case["steps"]):
        H.step(state["dt"], g, case["nsub"])
        speed = H.max_speed()
    return {"state": H.state(), "phi": g.phi(F64 if case["dtype"] == "f64" else torch.float32), "speed": speed}


def work(case):
    """Each input (density, carried state) read once, each output and the new state written once; the arithmetic of
    every sub-step (15 FP64 operations of the written order, about 30 float ones) and hydro stage."""
    kind = case["kind"]
    if kind == "batch":
        b = f = 0
        r = random.Random(case["side_seed"])
        sides = list(range(case["side_min"], case["side_max"] + 1, case["side_step"]))
        for i in range(case["grids"]):
            n = r.choice(sides)
            e = (14 + 10 + 4, 30) if i % 2 == 0 else (24 + 16 + 8, 15)
            b += n ** 3 * e[0]
            f += n ** 3 * case["substeps"] * e[1]
        return {"bytes": b, "flops": f}
    if kind == "gravity":
        n = case["nx"] * case["ny"] * case["nz"]
        f64 = case["prec"] == "f64"
        nq = (case["lmax"] + 1) ** 2 if case["bc"] == "multipole" else 0
        return {"bytes": n * (8 + 16 + 16 + 32 if f64 else 4 + 10 + 10 + 16),
                "flops": n * (case["substeps"] * (15 if f64 else 30) + 9 + 2 * nq)}
    if kind == "adjoint":
        n, f64 = case["n"] ** 3, case["prec"] == "f64"
        return {"bytes": n * (32 if f64 else 16), "flops": n * case["T"] * 2 * (15 if f64 else 30)}
    n, f64 = case["nx"] * case["ny"] * case["nz"], case["dtype"] == "f64"
    return {"bytes": n * ((5 + 1 + 5 + 1) * 8 if f64 else 5 * 4 + 8 + 5 * 4 + 4),
            "flops": n * case["steps"] * (case["nsub"] * (15 if f64 else 30) + 2 * 700)}


# ---- the same discrete scheme in plain float64 torch ------------------------------------------------------------------

def _faces(p):
    """(ghost, interior neighbour, opposite interior) views of the six faces of a padded field."""
    c = slice(1, -1)
    return [(p[c, c, 0], p[c, c, 1], p[c, c, -2]), (p[c, c, -1], p[c, c, -2], p[c, c, 1]),
            (p[c, 0, c], p[c, 1, c], p[c, -2, c]), (p[c, -1, c], p[c, -2, c], p[c, 1, c]),
            (p[0, c, c], p[1, c, c], p[-2, c, c]), (p[-1, c, c], p[-2, c, c], p[1, c, c])]


class _Wave:
    """phi^{n+1} = 2 phi^n - phi^{n-1} + nu^2 sum(phi_nb - phi) - s on a centred box, fields padded by one ghost."""

    def __init__(self, nx, ny, nz, h, nu, bc, lmax=0):
        self.nx, self.ny, self.nz, self.h, self.nu, self.bc, self.lmax = nx, ny, nz, h, nu, bc, lmax
        x, y, z = _axes(nx, ny, nz, h, 1)
        self.xyz = [t.expand(nz + 2, ny + 2, nx + 2) for t in (x, y, z)]
        self.data = None
        if bc == "robin":
            r = torch.sqrt(x * x + y * y + z * z)
            self.r = [(g.clone(), i.clone()) for g, i, _ in _faces(r)]
            self.a = []
            for f, (rg, _) in enumerate(self.r):
                xg = _faces(self.xyz[f // 2])[f][0]
                self.a.append(nu * rg / xg.abs())

    def solid(self, l, m, x, y, z):
        """r^l Y_lm, real orthonormal."""
        am, r2 = abs(m), x * x + y * y + z * z
        C, S = torch.ones_like(r2), torch.zeros_like(r2)
        for _ in range(am):
            C, S = x * C - y * S, x * S + y * C
        q0, q1 = torch.zeros_like(r2), torch.full_like(r2, math.prod(-(2.0 * k - 1) for k in range(1, am + 1)))
        for k in range(am + 1, l + 1):
            q0, q1 = q1, ((2 * k - 1) * z * q1 - (k + am - 1) * r2 * q0) / (k - am)
        norm = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - am) / math.factorial(l + am))
        return norm * q1 if m == 0 else math.sqrt(2.0) * norm * q1 * (C if m > 0 else S)

    def set_density(self, rho, src):
        """Source s; for the Dirichlet modes the boundary data of the moments of rho."""
        rho = rho.double()
        self.s = src * (rho - (rho.mean() if self.bc == "periodic" else 0.0))
        if self.bc in ("dirichlet", "multipole"):
            c = (slice(1, -1),) * 3
            inner = [t[c] for t in self.xyz]
            self.data = [torch.zeros_like(g) for g, _, _ in _faces(self.xyz[0])]
            for l in range((self.lmax if self.bc == "multipole" else 0) + 1):
                for m in range(-l, l + 1):
                    Q = (rho * self.solid(l, m, *inner)).sum() * self.h ** 3
                    for f, d in enumerate(self.data):
                        p = [_faces(t)[f][0] for t in self.xyz]
                        r = torch.sqrt(p[0] ** 2 + p[1] ** 2 + p[2] ** 2)
                        d -= 4 * math.pi / (2 * l + 1) * Q * self.solid(l, m, *p) / r ** (2 * l + 1)

    def seed(self, phi):
        p = F.pad(phi.double(), (1,) * 6)
        self.fill(p)
        if self.bc == "robin":
            for (g, i, _), (rg, ri) in zip(_faces(p), self.r):
                g.copy_(i * ri / rg)
        return p, p.clone()

    def fill(self, p):
        for f, (g, _, o) in enumerate(_faces(p)):
            if self.bc == "periodic":
                g.copy_(o)
            elif self.data is not None:
                g.copy_(self.data[f])

    def step(self, p, q):
        """(phi^n, phi^{n-1}) -> (phi^{n+1}, phi^n)"""
        c = p[1:-1, 1:-1, 1:-1]
        L = p[1:-1, 1:-1, :-2] - c
        for nb in (p[1:-1, 1:-1, 2:], p[1:-1, :-2, 1:-1], p[1:-1, 2:, 1:-1], p[:-2, 1:-1, 1:-1], p[2:, 1:-1, 1:-1]):
            L += nb - c
        qi = q[1:-1, 1:-1, 1:-1]
        qi.copy_(2 * c - qi + self.nu ** 2 * L - self.s)
        if self.bc == "robin":
            for (g, _, _), (g0, i0, _), (rg, ri), a in zip(_faces(q), _faces(p), self.r, self.a):
                g.copy_((rg * g0 - a * (rg * g0 - ri * i0)) / rg)
        else:
            self.fill(q)
        return q, p

    def accel(self, p):
        s = -0.5 / self.h
        return ((p[1:-1, 1:-1, 2:] - p[1:-1, 1:-1, :-2]) * s, (p[1:-1, 2:, 1:-1] - p[1:-1, :-2, 1:-1]) * s,
                (p[2:, 1:-1, 1:-1] - p[:-2, 1:-1, 1:-1]) * s)


def _inner(p):
    return p[1:-1, 1:-1, 1:-1].contiguous()


def _mc_half(a, b):
    """Half the monotonized-central slope."""
    m = torch.minimum(torch.minimum(a.abs(), b.abs()), 0.25 * (a + b).abs())
    return torch.where(a * b > 0, torch.sign(a) * m, torch.zeros_like(m))


def _prim(U):
    v = U[1:4] / U[0]
    return torch.cat([U[:1], v, ((GAMMA - 1.0) * (U[4] - 0.5 * (U[1:4] * v).sum(0)))[None]])


def _hllc(wl, wr, d):
    al, ar = torch.sqrt(GAMMA * wl[4] / wl[0]), torch.sqrt(GAMMA * wr[4] / wr[0])
    ul, ur = wl[1 + d], wr[1 + d]
    sl, sr = torch.minimum(ul - al, ur - ar), torch.maximum(ul + al, ur + ar)
    dl, dr = wl[0] * (sl - ul), wr[0] * (sr - ur)
    ss = ((wr[4] - wl[4]) + (ul * dl - ur * dr)) / (dl - dr)
    up, left = (sl >= 0) | (sr <= 0), (sl >= 0) | ((sr > 0) & (ss >= 0))
    w, sk, dk = torch.where(left, wl, wr), torch.where(left, sl, sr), torch.where(left, dl, dr)
    un = w[1 + d]
    E = w[4] / (GAMMA - 1.0) + 0.5 * w[0] * (w[1:4] ** 2).sum(0)
    u = torch.cat([w[:1], w[0] * w[1:4], E[None]])
    f = u * un
    f[1 + d] += w[4]
    f[4] += w[4] * un
    fac = dk / (sk - ss)
    us = torch.stack([fac, fac * w[1], fac * w[2], fac * w[3], fac * (E / w[0] + (ss - un) * (ss + w[4] / dk))])
    us[1 + d] = fac * ss
    return torch.where(up, f, f + sk * (us - u))


def _rhs(U, A, h):
    W, R = _prim(U), torch.zeros_like(U)
    for d, ax in ((0, 3), (1, 2), (2, 1)):
        n = W.shape[ax]
        i = torch.arange(-2, n + 2, device=DEV).clamp(0, n - 1)
        P = W.index_select(ax, i)
        s = _mc_half(P.narrow(ax, 1, n + 2) - P.narrow(ax, 0, n + 2), P.narrow(ax, 2, n + 2) - P.narrow(ax, 1, n + 2))
        fl = _hllc(P.narrow(ax, 1, n + 1) + s.narrow(ax, 0, n + 1), P.narrow(ax, 2, n + 1) - s.narrow(ax, 1, n + 1), d)
        R += (fl.narrow(ax, 0, n) - fl.narrow(ax, 1, n)) / h
    R[1:4] += U[0] * A
    R[4] += (U[1:4] * A).sum(0)
    return R


def _floors(U):
    U[0].clamp_(min=1e-12)
    ke = 0.5 * (U[1:4] ** 2).sum(0) / U[0]
    U[4] = torch.where((GAMMA - 1.0) * (U[4] - ke) < 1e-14, 1e-14 / (GAMMA - 1.0) + ke, U[4])
    return U


def exact(case, seed):
    kind = case["kind"]
    if kind == "gravity":
        rho, phi, h, _, nu = _gravity_inputs(case, seed)
        w = _Wave(case["nx"], case["ny"], case["nz"], h, nu, case["bc"], case["lmax"])
        w.set_density(rho, (nu * h) ** 2 * 4 * math.pi)
        p, q = w.seed(phi)
        for _ in range(case["substeps"]):
            p, q = w.step(p, q)
        return {"accel": w.accel(p), "phi": _inner(p)}
    if kind == "batch":
        out = []
        for n, _, rho in _batch_inputs(case, seed):
            nu = 0.5 / math.sqrt(3.0)
            w = _Wave(n, n, n, 1.0 / n, nu, "robin")
            w.set_density(rho, (nu / n) ** 2 * 4 * math.pi)
            p, q = w.seed(torch.zeros_like(rho))
            for _ in range(case["substeps"]):
                p, q = w.step(p, q)
            out.append(_inner(p))
        return out
    if kind == "adjoint":
        rho, dL, h, _, nu = _adjoint_inputs(case, seed)
        n, src = case["n"], (nu * h) ** 2 * 4 * math.pi
        w = _Wave(n, n, n, h, nu, case["bc"])
        w.set_density(rho, src)
        p, q = w.seed(torch.zeros_like(rho))
        for _ in range(case["T"]):
            p, q = w.step(p, q)
        # the transpose: the same sub-step with zero source and zero boundary data, run on lambda
        w.s, w.data = torch.zeros_like(w.s), None
        lam, old = F.pad(dL.double(), (1,) * 6), torch.zeros_like(p)
        w.fill(lam)
        acc = torch.zeros_like(w.s)
        for _ in range(case["T"]):
            acc += lam[1:-1, 1:-1, 1:-1]
            lam, old = w.step(lam, old)
        grad = -src * acc
        return {"phi": _inner(p), "grad": grad - grad.mean() if case["bc"] == "periodic" else grad}
    W, phi, h, _, c, dtg = _hydro_inputs(case, seed)
    W = W.double()
    dt, v = case["nsub"] * dtg, W[1:4]
    U = torch.cat([W[:1], W[0] * v, (W[4] / (GAMMA - 1.0) + 0.5 * W[0] * (v * v).sum(0))[None]])
    w = _Wave(case["nx"], case["ny"], case["nz"], h, c * dtg / h, case["bc"])
    p, q = w.seed(phi)
    for _ in range(case["steps"]):
        w.set_density(U[0], (c * dtg) ** 2 * 4 * math.pi)
        for _ in range(case["nsub"]):
            p, q = w.step(p, q)
        A = torch.stack(w.accel(p))
        U1 = _floors(U + dt * _rhs(U, A, h))
        U = _floors(0.5 * (U + (U1 + dt * _rhs(U1, A, h))))
    W = _prim(U)
    speed = (torch.sqrt((W[1:4] ** 2).sum(0)) + torch.sqrt(GAMMA * W[4] / W[0])).max().item()
    return {"state": U, "phi": _inner(p), "speed": speed}
