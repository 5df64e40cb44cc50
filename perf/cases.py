"""Timed workloads of the library: what a program that uses it has it do, through its public
entry points (Context.step_io, Context.set_state / step_async / get_state, SnapSteps).

listed() names the cases, draw(rng) gives more of the same ranges, prepare / run make and do
one pass, work counts the bytes and operations a pass cannot do without, and exact gives the
result of the pass in 64 bits from a plain torch statement of the method (whole-array
operations, none of the library's code).

Families (field "kind"):
  dry2    dry gas in the x-z plane: warm bubbles and the viscous density current
  dry3    dry gas in three dimensions, periodic in x and y
  moist2  one vapour with cloud and rain in the x-z plane (saturation adjustment every stage)
  bryan   the same layout in a saturated environment: cloud in every cell
  jovian  two vapours with cloud and precipitation each, three dimensions
  rce     the same with Kessler microphysics, falling precipitation, cooling, sponge and a
          no-slip floor at a fixed temperature
  members many moist x-z domains of four sizes in one context
  adjoint forward and adjoint of the dry x-z plane through torch.autograd
"""
import dataclasses
import functools
import math

import numpy as np
import torch

import workloads as W
from paper_1901_02955_gb300 import Context
from paper_1901_02955_gb300.autograd import SnapSteps, dry_state_from_theta, kinetic_energy


def listed():
    return [
        # the paper-sized warm bubble in double precision, a few steps at a time as a program
        # that looks at the state between outputs calls it: one small grid, latency counts
        dict(name="bubble_f64_small", kind="dry2", dtype="f64", nx=128, ny=1, nz=128, nu=0.0,
             steps=5, host=False),
        # one small moist member on its own: every launch and every dependent load is visible
        dict(name="moist_f32_small", kind="moist2", dtype="f32", nx=61, ny=1, nz=47, nu=0.0,
             steps=10, host=False),
        # the density current the library is quoted on, single precision
        dict(name="current_f32", kind="dry2", dtype="f32", nx=1024, ny=1, nz=256, nu=75.0,
             steps=20, host=False),
        # the same in double precision
        dict(name="current_f64", kind="dry2", dtype="f64", nx=1024, ny=1, nz=256, nu=75.0,
             steps=2, host=False),
        # the same through pinned host memory, one step per call (coupling to a host program)
        dict(name="current_f32_host", kind="dry2", dtype="f32", nx=1024, ny=1, nz=256, nu=75.0,
             steps=1, host=True),
        # three-dimensional dry convection on a ragged grid
        dict(name="dry3_f32_ragged", kind="dry3", dtype="f32", nx=190, ny=131, nz=85, nu=0.0,
             steps=4, host=False),
        # moist Jovian column, the largest grid of the configurations
        dict(name="jovian_f32", kind="jovian", dtype="f32", nx=256, ny=256, nz=128, nu=0.0,
             steps=2, host=False),
        # its radiative-convective setup (all the microphysics and forcing) on a crop
        dict(name="rce_f32", kind="rce", dtype="f32", nx=128, ny=96, nz=128, nu=0.0,
             steps=2, host=False),
        # the ensemble of 96 uneven moist bubbles
        dict(name="members_f32", kind="members", dtype="f32", n0=64, per_size=24, steps=8),
        # the Bryan moist bubble in double precision (cloud in every cell)
        dict(name="bryan_f64", kind="bryan", dtype="f64", nx=200, ny=1, nz=100, nu=0.0,
             steps=3, host=False),
        # gradient of the final kinetic energy with respect to the initial potential
        # temperature: checkpointed in single precision, every stage kept in double
        dict(name="adjoint_f32", kind="adjoint", dtype="f32", nx=256, ny=1, nz=256, nu=0.0,
             steps=40, ckpt=20),
        dict(name="adjoint_f64", kind="adjoint", dtype="f64", nx=256, ny=1, nz=256, nu=0.0,
             steps=10, ckpt=5),
    ]


def _size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dry2", "dry2", "dry3", "moist2", "bryan", "jovian", "rce", "members",
                       "adjoint"])
    dtype = rng.choice(["f32", "f32", "f64"])
    if kind == "members":
        return dict(kind=kind, dtype="f32", n0=_size(rng, 16, 64), per_size=rng.randint(3, 24),
                    steps=rng.randint(1, 8))
    if kind == "adjoint":
        steps = rng.randint(4, 20) if dtype == "f32" else rng.randint(2, 10)
        return dict(kind=kind, dtype=dtype, nx=_size(rng, 48, 256), ny=1, nz=_size(rng, 48, 256),
                    nu=0.0, steps=steps, ckpt=rng.choice([0, 2, max(1, steps // 2)]))
    case = dict(kind=kind, dtype=dtype, nu=0.0, steps=rng.randint(1, 8 if dtype == "f32" else 2),
                host=False)
    if kind == "dry2":
        case.update(nx=_size(rng, 40, 1024), ny=1, nz=_size(rng, 40, 512),
                    nu=rng.choice([0.0, 75.0]), host=rng.random() < 0.25)
    elif kind in ("moist2", "bryan"):
        case.update(nx=_size(rng, 40, 512), ny=1, nz=_size(rng, 40, 512 if kind == "moist2" else 200),
                    host=kind == "moist2" and rng.random() < 0.25)
    elif kind == "dry3":
        top = 190 if dtype == "f32" else 96
        case.update(nx=_size(rng, 16, top), ny=_size(rng, 16, top), nz=_size(rng, 16, 85),
                    steps=rng.randint(1, 4) if dtype == "f32" else 1)
    else:
        case.update(dtype="f32", nx=_size(rng, 16, 160), ny=_size(rng, 16, 160),
                    nz=_size(rng, 48, 128), steps=rng.randint(1, 2))
    return case


# ------------------------------------------------------------------------------------------
# inputs
# ------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _column(kind, nz):
    """The family's background at rest on a few columns: its reference profile, species and
    scheme options (a pure function of the family and the number of levels)."""
    if kind == "current":
        return W.density_current(nx=4, nz=nz)
    if kind == "bubble":
        return W.warm_bubble(n=nz, A=0.0)
    if kind == "dry3":
        return W.dry_bubble_3d(nx=4, ny=4, nz=nz, L=4 * 1000.0 / 96, A=0.0)
    if kind == "moist2":
        return W.moist_bubble(nx=4, nz=nz, A=0.0)
    if kind == "bryan":
        return W.bryan_moist_bubble(nx=4, nz=nz, A=0.0)
    make = W.jovian if kind == "jovian" else W.jovian_rce
    return make(nx=4, ny=4, nz=nz, noise_K=0.0)


def _domain(case, nx, ny, nz):
    """The domain of one case: the family's column widened to nx x ny at the family's spacing."""
    kind = case["kind"]
    if kind == "adjoint":
        kind = "bubble"
    if kind == "members":
        kind = "moist2"
    if kind == "dry2":
        kind = "current" if case["nu"] > 0 else "bubble"
    w = _column(kind, nz)
    dx = {"current": 25.0, "bubble": 1000.0 / nz, "dry3": w.dz, "moist2": 1000.0 / nz,
          "bryan": 100.0, "jovian": 100e3 / 256, "rce": 100e3 / 256}[kind]
    nu = case.get("nu", 0.0)
    return dataclasses.replace(w, name=kind, nx=nx, ny=ny, nz=nz, dx=dx, dy=dx, nu=nu)


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _modes(g, w, amp, n):
    """n seeded smooth fields (nz, ny, nx): a few Fourier modes of wavelengths from the domain
    down to about eight cells, so that the flow has structure on the grid's own scale."""
    dev = _device()
    x = (torch.arange(w.nx, device=dev, dtype=torch.float64) + 0.5) / w.nx
    y = (torch.arange(w.ny, device=dev, dtype=torch.float64) + 0.5) / w.ny
    z = (torch.arange(w.nz, device=dev, dtype=torch.float64) + 0.5) / w.nz
    out = []
    for _ in range(n):
        f = torch.zeros((w.nz, w.ny, w.nx), device=dev, dtype=torch.float64)
        for m in range(4):
            kx = int(g.integers(1, max(2, w.nx // 8))) if m else 1
            ky = int(g.integers(0, max(1, w.ny // 8))) if w.ny > 1 else 0
            kz = int(g.integers(1, max(2, w.nz // 8))) if m else 1
            a, p, q, r = g.uniform(0.3, 1.0), *g.uniform(0.0, 2 * math.pi, 3)
            f += (0.5 * amp * a) * (torch.sin(math.pi * kz * z + r)[:, None, None] *
                                    torch.sin(2 * math.pi * ky * y + q)[None, :, None] *
                                    torch.sin(2 * math.pi * kx * x + p)[None, None, :]
                                    if w.ny > 1 else
                                    torch.sin(math.pi * kz * z + r)[:, None, None] *
                                    torch.sin(2 * math.pi * kx * x + p)[None, None, :])
        out.append(f)
    return out


def _heating(g, w, kind):
    """Relative temperature perturbation (nz, ny, nx) at fixed pressure: the family's bubble at
    a seeded place and strength, and white noise."""
    dev = _device()
    Tref = {"current": 300.0, "bubble": 300.0, "dry3": 300.0, "moist2": 300.0, "bryan": 290.0,
            "jovian": 250.0, "rce": 300.0}[kind]
    A, r = {"current": (-15.0, 0.3), "bubble": (0.5, 0.25), "dry3": (0.5, 0.25),
            "moist2": (1.0, 0.25), "bryan": (2.0, 0.2), "jovian": (1.0, 0.15),
            "rce": (1.0, 0.15)}[kind]
    A *= g.uniform(0.5, 1.5)
    x = (torch.arange(w.nx, device=dev, dtype=torch.float64) + 0.5) * w.dx
    y = (torch.arange(w.ny, device=dev, dtype=torch.float64) + 0.5) * w.dx
    z = (torch.arange(w.nz, device=dev, dtype=torch.float64) + 0.5) * w.dz
    X, Y, Z = w.nx * w.dx, w.ny * w.dx, w.nz * w.dz
    d = ((x - g.uniform(0.3, 0.7) * X) / (r * X))[None, None, :] ** 2
    d = d + ((z - g.uniform(0.3, 0.6) * Z) / (r * Z))[:, None, None] ** 2
    if w.ny > 1:
        d = d + ((y - g.uniform(0.3, 0.7) * Y) / (r * Y))[None, :, None] ** 2
    d = d.expand(w.nz, w.ny, w.nx).clamp(max=1.0).sqrt()
    dT = A * torch.cos(0.5 * math.pi * d) ** 2
    tg = torch.Generator(device=dev)
    tg.manual_seed(int(g.integers(1 << 40)))
    noise = torch.randn(dT.shape, generator=tg, device=dev, dtype=torch.float64)
    return (dT + 0.1 * noise) / Tref


def _state(case, w, seed):
    """Conserved state (nv, nz, ny, nx) in 64 bits on the device."""
    g = np.random.default_rng([190102955, seed])
    base = torch.from_numpy(np.ascontiguousarray(_column(w.name, w.nz).Y[:, :, 0, 0])).to(_device())
    Y = base[:, :, None, None].expand(-1, -1, w.ny, w.nx).clone()
    ns = 1 + w.nvapor * (1 + w.ncond)
    Y[:ns] /= 1.0 + _heating(g, w, w.name)
    if w.name == "rce":  # rain already falling
        for i in range(w.nvapor):
            Y[1 + w.nvapor + 2 * i + 1] = Y[1 + i] * (0.02 * float(g.uniform(0.5, 1.5)))
    rho = Y[:ns].sum(0)
    amp = {"jovian": 8.0, "rce": 8.0, "current": 4.0, "bryan": 4.0}.get(w.name, 2.0)
    for m, u in enumerate(_modes(g, w, amp, w.nmom)):
        Y[ns + m] = rho * u
        Y[-1] += 0.5 * rho * u * u
    return Y


def _members(case):
    return [n for f in (1, 2, 4, 8) for n in [case["n0"] * f] * case["per_size"]]


def _domains(case):
    if case["kind"] == "members":
        return [_domain(case, n, 1, n) for n in _members(case)]
    return [_domain(case, case["nx"], case["ny"], case["nz"])]


def _inputs(case, seed):
    """The conserved states of a case's domains as the program holds them (its own type)."""
    dt = torch.float32 if case["dtype"] == "f32" else torch.float64
    return [_state(case, w, seed * 1000 + d).to(dt) for d, w in enumerate(_domains(case))]


def _theta(case, seed):
    """Initial potential temperature and velocity of an adjoint case."""
    w = _domains(case)[0]
    dt = torch.float32 if case["dtype"] == "f32" else torch.float64
    g = np.random.default_rng([190102955, seed])
    theta = (300.0 * (1.0 + _heating(g, w, w.name))).to(dt)
    vel = torch.stack(_modes(g, w, 2.0, 2)).to(dt)
    pc = torch.from_numpy(0.5 * (w.p_bar_face[:-1] + w.p_bar_face[1:])).to(_device())
    return w, theta, vel, pc


def prepare(case, seed):
    if case["kind"] == "adjoint":
        w, theta, vel, pc = _theta(case, seed)
        ctx = Context(w, dtype=case["dtype"])
        ctx.set_stream(torch.cuda.current_stream())
        return dict(case=case, w=w, ctx=ctx, theta=theta, vel=vel, pc=pc)
    ws = _domains(case)
    Y = _inputs(case, seed)
    ctx = Context(ws, dtype=case["dtype"])
    ctx.set_stream(torch.cuda.current_stream())
    if case["kind"] == "members":  # the results of one size in one array
        out = [torch.empty((case["per_size"],) + tuple(y.shape), dtype=y.dtype, device=y.device)
               for y in Y[::case["per_size"]]]
    elif case.get("host"):
        Y = [y.cpu().pin_memory() for y in Y]
        out = [torch.empty_like(y, pin_memory=True) for y in Y]
    else:
        out = [torch.empty_like(y) for y in Y]
    return dict(case=case, ctx=ctx, Y=Y, out=out)


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "adjoint":
        w = state["w"]
        theta = state["theta"].detach().requires_grad_(True)
        Y0 = dry_state_from_theta(theta, state["pc"], velocity=state["vel"])
        YN = SnapSteps.apply(Y0, ctx, case["steps"], case["ckpt"])
        kinetic_energy(YN, w.dx * w.dz).backward()
        return [YN.detach(), theta.grad]
    if case["kind"] == "members":
        for d, y in enumerate(state["Y"]):
            ctx.set_state(y, domain=d)
        ctx.step_async(case["steps"])
        for d, o in enumerate(o for size in state["out"] for o in size):
            ctx.get_state(domain=d, out=o)
        return state["out"]
    ctx.step_io(state["Y"][0], state["out"][0], nsteps=case["steps"])
    return state["out"]


def work(case):
    """Each input and output once; the method's operations (per cell and stage: WENO 65 per face
    side and variable, LMARS, primitives, divergence, gravity, stage combine, viscosity). An
    adjoint pass is counted as the forward steps, their transpose at twice a forward step and,
    with checkpoints, the forward steps once more."""
    word = 4 if case["dtype"] == "f32" else 8
    cells = (sum(n * n for n in _members(case)) if case["kind"] == "members"
             else case["nx"] * case["ny"] * case["nz"])
    three_d = case["kind"] in ("dry3", "jovian", "rce")
    ntr = {"dry2": 0, "dry3": 0, "adjoint": 0, "moist2": 3, "bryan": 3, "members": 3}.get(
        case["kind"], 6)
    D, nmom = (3, 3) if three_d else (2, 2)
    nv = 2 + ntr + nmom
    per = (D * nv * 130 + D * (31 + 3 * nmom + 10 * ntr) + 3 * nmom + 3 + 8 * ntr +
           3 * D * nv + 7 + 4 * nv)
    if case.get("nu", 0.0) > 0.0:
        per += D * (6 * nmom + 12) + 5
    flops = 3.0 * per * cells * case["steps"]
    nbytes = 2.0 * nv * cells * word
    if case["kind"] == "adjoint":
        flops *= 4.0 if case["ckpt"] else 3.0
        nbytes = (2 + nmom + nv) * cells * word
    return {"bytes": nbytes, "flops": flops}


# ------------------------------------------------------------------------------------------
# the method in 64 bits, plain torch: SSP-RK3 of WENO5 + LMARS with gravity against the
# hydrostatic reference, viscosity, saturation adjustment, Kessler scheme and forcing
# ------------------------------------------------------------------------------------------
class _Method:
    """The domains are stacked along y when they do not use it (x-z plane), each with its own
    time step: fields (nv, nz, ny, nx), time step (ny or 1, 1)."""

    def __init__(self, w, stacked=False):
        dev = _device()
        t = functools.partial(torch.tensor, dtype=torch.float64, device=dev)
        self.w, self.stacked = w, stacked
        self.three_d = w.nmom == 3
        self.ns = 1 + w.nvapor * (1 + w.ncond)
        self.cvd = w.R_d / (w.gamma_d - 1.0)
        col = lambda a: t(np.asarray(a))[:, None, None]
        pc = 0.5 * (w.p_bar_face[:-1] + w.p_bar_face[1:])
        self.rb, self.pc, self.pf = col(w.rho_bar), col(pc), col(w.p_bar_face)
        self.heat, self.gas, self.mu = [1.0], [1.0], [0.0]  # per density: c_v/c_vd, R/R_d, mu
        for v in w.vapors:
            self.heat.append(v.sigma_v), self.gas.append(1.0 / v.eps), self.mu.append(0.0)
        for v in w.vapors:
            cp = v.sigma_v * self.cvd + w.R_d / v.eps
            for c in v.cond:
                self.heat.append(c.sigma_v), self.gas.append(0.0)
                self.mu.append(-(c.L_ref + (c.sigma_v * self.cvd - cp) * v.T_ref))

    def mom(self, d):
        return self.ns + (d if self.three_d else (0, None, 1)[d])

    def cond(self, i, j):
        return 1 + self.w.nvapor + i * self.w.ncond + j

    def mix(self, q, coef):
        return sum(c * f for c, f in zip(coef, q))

    def kinetic(self, Y):
        return 0.5 * (Y[self.ns:-1] ** 2).sum(0) / Y[:self.ns].sum(0)

    def temperature(self, Y):
        r = Y[:self.ns]
        return ((Y[-1] - self.kinetic(Y) - self.mix(r, self.mu)) /
                (self.cvd * self.mix(r, self.heat)))

    def primitives(self, Y):
        r = Y[:self.ns]
        rho = r.sum(0)
        p = self.w.R_d * self.mix(r, self.gas) * self.temperature(Y)
        return torch.stack([rho] + [r[s] / rho for s in range(1, self.ns)] +
                           [Y[m] / rho for m in range(self.ns, Y.shape[0] - 1)] + [p - self.pc])

    def fractions(self, X):
        return [1.0 - X[1:self.ns].sum(0)] + list(X[1:self.ns])

    def gamma(self, q):
        return 1.0 + (self.w.gamma_d - 1.0) * self.mix(q, self.gas) / self.mix(q, self.heat)

    def time_step(self, Y):
        X, w = self.primitives(Y), self.w
        c = torch.sqrt(self.gamma(self.fractions(X)) * (X[-1] + self.pc) / X[0])
        rate = sum((X[self.mom(d)].abs() + c) / h for d, h in
                   ((0, w.dx), (1, w.dy), (2, w.dz)) if d != 1 or self.three_d)
        if self.stacked:
            return w.cfl / rate.amax(dim=(0, 2))[:, None]
        return w.cfl / rate.max()

    def pad(self, X, d, ghost_T=True):
        """Three ghost cells on both sides along direction d."""
        w, dim = self.w, 3 - d
        if w.bc[2 * d] == W.PERIODIC:
            return torch.cat([X.narrow(dim, X.shape[dim] - 3, 3), X, X.narrow(dim, 0, 3)], dim)
        sides = []
        for s, start in ((2 * d, 0), (2 * d + 1, X.shape[dim] - 3)):
            sign = torch.ones(X.shape[0], dtype=X.dtype, device=X.device)
            for m in range(self.ns, X.shape[0] - 1):
                if w.bc[s] == W.NOSLIP or m == self.mom(d):
                    sign[m] = -1.0
            G = X.narrow(dim, start, 3).flip(dim) * sign.view(-1, 1, 1, 1)
            if s == 4 and w.T_bottom > 0.0:
                p = G[-1] + self.pc[:3].flip(0)
                rho = p / (w.R_d * self.mix(self.fractions(G), self.gas) * w.T_bottom)
                G = torch.cat([rho[None], G[1:]])
            sides.append(G)
        return torch.cat([sides[0], X, sides[1]], dim)

    def weno(self, a, b, c, d, e):
        """Value at the face beyond c (towards d) from the five cells a .. e."""
        eps = self.w.weno_eps
        b0 = 13 / 12 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2
        b1 = 13 / 12 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2
        b2 = 13 / 12 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2
        a0, a1, a2 = 0.1 / (eps + b0) ** 2, 0.6 / (eps + b1) ** 2, 0.3 / (eps + b2) ** 2
        q0 = (2 * a - 7 * b + 11 * c) / 6
        q1 = (-b + 5 * c + 2 * d) / 6
        q2 = (2 * c + 5 * d - e) / 6
        return (a0 * q0 + a1 * q1 + a2 * q2) / (a0 + a1 + a2)

    def flux(self, X, d):
        w, dim = self.w, 3 - d
        P = self.pad(X, d)
        n = X.shape[dim]
        cell = lambda k: P.narrow(dim, k, n + 1)  # cell k - 3 + face number
        L = self.weno(cell(0), cell(1), cell(2), cell(3), cell(4))
        R = self.weno(cell(5), cell(4), cell(3), cell(2), cell(1))
        pref = self.pf if d == 2 else self.pc
        m, g1 = self.mom(d), w.gamma_d - 1.0
        qL, qR = self.fractions(L), self.fractions(R)
        cL = torch.sqrt(self.gamma(qL) * (pref + L[-1]) / L[0])
        cR = torch.sqrt(self.gamma(qR) * (pref + R[-1]) / R[0])
        rc = 0.25 * (L[0] + R[0]) * (cL + cR)
        ps = 0.5 * (L[-1] + R[-1]) - 0.5 * rc * (R[m] - L[m])
        us = 0.5 * (L[m] + R[m]) - 0.5 * (R[-1] - L[-1]) / rc
        S = torch.where(us > 0, L, R)
        q, rho, p = self.fractions(S), S[0], S[-1] + pref
        vel = S[self.ns:-1]
        rhoe = (p * self.mix(q, self.heat) / self.mix(q, self.gas) / g1 +
                0.5 * rho * (vel ** 2).sum(0) + rho * self.mix(q, self.mu))
        F = [us * rho * f for f in q] + [us * rho * v for v in vel] + [us * (rhoe + p)]
        F[m] = F[m] + ps
        if d == 2 and any(w.w_term):
            self.sediment(F, L, R, pref)
        if w.nu > 0.0:
            h = (w.dx, w.dy, w.dz)[d]
            lo, hi = P.narrow(dim, 2, n + 1), P.narrow(dim, 3, n + 1)
            k = torch.arange(-1, n + 1, device=X.device)
            prof = self.pc[k.clamp(0, n - 1)] if d == 2 else self.pc
            Q = P.narrow(dim, 2, n + 2)
            Pi = ((Q[-1] + prof) / 1e5) ** (g1 / w.gamma_d)
            th = (Q[-1] + prof) / (Q[0] * Pi * w.R_d)
            cut = lambda f, k: f.narrow(dim - 1, k, n + 1)
            rf, work = 0.5 * (lo[0] + hi[0]), 0.0
            for mm in range(self.ns, X.shape[0] - 1):
                grad = (hi[mm] - lo[mm]) / h
                F[mm] = F[mm] - rf * w.nu * grad
                work = work + 0.5 * (lo[mm] + hi[mm]) * grad
            heat = 0.5 * (cut(Pi, 0) + cut(Pi, 1)) * (cut(th, 1) - cut(th, 0)) / h
            F[-1] = F[-1] - rf * w.nu * (work + w.gamma_d * self.cvd * heat)
        return torch.stack(F)

    def sediment(self, F, L, R, pref):
        w = self.w
        for j, wt in enumerate(w.w_term):
            if wt == 0.0:
                continue
            S = R if wt < 0 else L
            T = (pref + S[-1]) / (S[0] * w.R_d * self.mix(self.fractions(S), self.gas))
            u2 = (S[self.ns:-1] ** 2).sum(0)
            for i in range(w.nvapor):
                c = self.cond(i, j)
                ms = wt * S[0] * S[c]
                ms[0], ms[-1] = 0.0, 0.0  # nothing passes the walls
                F[c] = F[c] + ms
                for m in range(self.ns, L.shape[0] - 1):
                    F[m] = F[m] + ms * S[m]
                F[-1] = F[-1] + ms * (self.heat[c] * self.cvd * T + 0.5 * u2 + self.mu[c])

    def tendency(self, Y):
        w = self.w
        X = self.primitives(Y)
        out = 0.0
        for d, h in ((0, w.dx), (1, w.dy), (2, w.dz)):
            if d == 1 and not self.three_d:
                continue
            F, dim = self.flux(X, d), 3 - d
            n = X.shape[dim]
            out = out - (F.narrow(dim, 1, n) - F.narrow(dim, 0, n)) / h
        mass = F[:self.ns].sum(0)  # the z fluxes
        src = [torch.zeros_like(X[0]) for _ in range(Y.shape[0])]
        src[self.mom(2)] = -(X[0] - self.rb) * w.grav
        src[-1] = -w.grav * 0.5 * (mass[:-1] + mass[1:])
        if w.cooling:
            rate, lo, hi = w.cooling
            band = ((self.pc >= lo) & (self.pc <= hi)).double()
            src[-1] = src[-1] - band * rate * self.cvd * self.mix(Y[:self.ns], self.heat)
        if w.sponge:
            tau, p0 = w.sponge
            damp = (self.pc < p0).double() / (tau * (self.pc / p0) ** 2)
            for d in (0, 1):
                if d == 0 or self.three_d:
                    src[self.mom(d)] = -damp * Y[self.mom(d)]
        return out + torch.stack(src)

    def saturation(self, i, T):
        """Saturation pressure of vapour i and its logarithmic derivative times T."""
        v = self.w.vapors[i]
        Rv = self.w.R_d / v.eps
        dc = v.cond[0].sigma_v * self.cvd - (v.sigma_v * self.cvd + Rv)
        beta, delta = v.cond[0].L_ref / (Rv * v.T_ref) + dc / Rv, dc / Rv
        t = T / v.T_ref
        return v.p_ref * torch.exp(beta * (1 - 1 / t) - delta * torch.log(t)), beta / t - delta

    def adjust(self, Y, sweeps=40):
        """Saturation adjustment of every cell at fixed energy and momenta."""
        w = self.w
        if w.nvapor == 0:
            return Y
        Y = Y.clone()
        for _ in range(sweeps):
            worst = 0.0
            for i, v in enumerate(w.vapors):
                T = self.temperature(Y)
                p = w.R_d * self.mix(Y[:self.ns], self.gas) * T
                N, gas, heat = Y[0], Y[0], 0.0
                for k, vk in enumerate(w.vapors):
                    tot = Y[1 + k] + sum(Y[self.cond(k, j)] for j in range(w.ncond))
                    N = N + tot / vk.eps
                    gas = gas + Y[1 + k] / vk.eps
                    heat = heat + tot / vk.eps * (vk.sigma_v * vk.eps - 1.0)
                vap, cl = 1 + i, self.cond(i, 0)
                qv, qc = Y[vap] / v.eps / N, Y[cl] / v.eps / N
                rest = gas / N - qv
                ps, slope = self.saturation(i, T)
                s = ps / p
                alpha = (w.gamma_d - 1.0) * (slope - 1.0) / (1.0 + heat / N)
                om = torch.where(s < 1.0, 1.0 - s, torch.ones_like(s))
                dq = (qv - s / om * rest) / (1.0 + s / om ** 2 * slope * alpha * rest)
                dq = torch.where(s < 1.0, dq, -qc)
                move = torch.where(dq >= qv, Y[vap],
                                   torch.where(dq <= -qc, -Y[cl], dq * v.eps * N))
                Y[vap] -= move
                Y[cl] += move
                rel = (move.abs() / (Y[vap].abs() + Y[cl].abs() + 1e-300)).max()
                worst = max(worst, float(rel))
            if worst < 1e-14:
                break
        return Y

    def kessler(self, Y, dt):
        """Backward Euler of the Kessler scheme in every cell (both forms of the rates by
        Newton, then the one consistent with its own side of saturation)."""
        w = self.w
        if not w.kessler_k:
            return Y
        k1, k2, k3, k4 = w.kessler_k
        Y = Y.clone()
        rho = Y[:self.ns].sum(0)
        for i, v in enumerate(w.vapors):
            iv, ic, ir = 1 + i, self.cond(i, 0), self.cond(i, 1)
            yn = [Y[iv].clone(), Y[ic].clone(), Y[ir].clone()]
            tot = yn[0] + yn[1] + yn[2]

            def excess(a, b):
                """rho_v - rho*(T) and its derivatives by the three densities."""
                Y[iv], Y[ic], Y[ir] = a, b, tot - a - b
                T = self.temperature(Y)
                Cv = self.cvd * self.mix(Y[:self.ns], self.heat)
                ps, slope = self.saturation(i, T)
                rs = ps / (w.R_d / v.eps * T)
                drs = rs * (slope - 1.0) / T
                ds = [(k == iv) * 1.0 + drs * (self.mu[k] + self.heat[k] * self.cvd * T) / Cv
                      for k in (iv, ic, ir)]
                return a - rs, ds

            def solve(sat):
                a, b = yn[0].clone(), yn[1].clone()
                for _ in range(w.kessler_max_iter):
                    s, ds = excess(a, b)
                    r = tot - a - b
                    acc = k3 * b * r / rho
                    if sat:
                        Fv, Ft = -k1 * s, -acc - k2 * b
                        Jv, Jt = [-k1 * q for q in ds], [0.0, 0.0, 0.0]
                    else:
                        e = k4 * r / rho
                        Fv, Ft = -e * s, -e * s - acc - k2 * b
                        Jv = [-e * ds[0], -e * ds[1], -e * ds[2] - k4 * s / rho]
                        Jt = list(Jv)
                    Jt = [Jt[0], Jt[1] - k3 * r / rho - k2, Jt[2] - k3 * b / rho]
                    G0 = Fv - (a - yn[0]) / dt
                    G1 = Ft - (a - yn[0] + b - yn[1]) / dt
                    A00, A01 = Jv[0] - Jv[2] - 1 / dt, Jv[1] - Jv[2]
                    A10, A11 = Jt[0] - Jt[2] - 1 / dt, Jt[1] - Jt[2] - 1 / dt
                    det = A00 * A11 - A01 * A10
                    da, db = (-G0 * A11 + G1 * A01) / det, (-G1 * A00 + G0 * A10) / det
                    a, b = a + da, b + db
                    if float(((da.abs() + db.abs()) / (tot.abs() + 1e-300)).max()) < 1e-15:
                        break
                return a, b, excess(a, b)[0]

            s0 = excess(yn[0], yn[1])[0]
            aw, bw, sw = solve(True)
            ad, bd, sd = solve(False)
            wet = torch.where(s0 > 0, (sw > 0) | ~(sd <= 0), ~(sd <= 0))
            a, b = torch.where(wet, aw, ad), torch.where(wet, bw, bd)
            Y[iv], Y[ic], Y[ir] = a, b, tot - a - b
        return Y

    def step(self, Y, dt, stage=lambda f, Y: f(Y)):
        for weight in (1.0, 0.25, 2.0 / 3.0):
            if weight == 1.0:
                Yn = Y
            Z = Y + dt * stage(self.tendency, Y)
            Y = self.adjust(Yn + weight * (Z - Yn))
        return self.kessler(Y, dt)


def exact(case, seed):
    if case["kind"] == "adjoint":
        from torch.utils.checkpoint import checkpoint
        w, theta, vel, pc = _theta(case, seed)
        M = _Method(w)
        theta = theta.double().requires_grad_(True)
        vel, g1 = vel.double(), w.gamma_d - 1.0
        kappa = g1 / w.gamma_d
        rho = M.pc / (w.R_d * theta * (M.pc / 1e5) ** kappa)
        Y = torch.stack([rho, rho * vel[0], rho * vel[1],
                         M.pc / g1 + 0.5 * rho * (vel ** 2).sum(0)])
        for _ in range(case["steps"]):
            with torch.no_grad():
                dt = M.time_step(Y)
            Y = M.step(Y, dt, lambda f, Z: checkpoint(f, Z, use_reentrant=False))
        (0.5 * (Y[1:-1] ** 2).sum(0) / Y[0]).sum().mul(w.dx * w.dz).backward()
        return [Y.detach(), theta.grad]
    with torch.no_grad():
        Y, ws = [y.double() for y in _inputs(case, seed)], _domains(case)
        out = []
        for n in dict.fromkeys((w.nx, w.nz) for w in ws):
            same = [d for d, w in enumerate(ws) if (w.nx, w.nz) == n]
            M = _Method(ws[same[0]], stacked=case["kind"] == "members")
            Z = torch.cat([Y[d] for d in same], 2)  # x-z domains of one size side by side
            for _ in range(case["steps"]):
                Z = M.step(Z, M.time_step(Z))
            out.append(Z.permute(2, 0, 1, 3)[:, :, :, None].contiguous() if M.stacked else Z)
        return out
