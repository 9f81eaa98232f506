"""The work that users of the TRT-R library have it do, as cases that can be timed and checked.

Every case goes through the public entry points of ``paper_2312_10316_gb300`` (``Solver``,
``Batch``, ``autograd``) on inputs that are on the GPU, and ends with what the caller's program
goes on with: phi (or populations, or a gradient) as a tensor of the storage's own type.
``exact`` is the same scheme in plain FP64 torch: direction by direction equilibria, explicit
Hermite tensors and rolls.
"""
from __future__ import annotations

import dataclasses
import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_2312_10316_gb300 import autograd as A
from paper_2312_10316_gb300 import trtr as T
from paper_2312_10316_gb300 import workloads as W

DEV = "cuda"
OUT = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
PULSES = {"pulse64": W.C1_F64_64, "pulse1024": W.C2A_F32_1024, "pulse4096": W.C2B_F32_4096,
          "pulse8192": W.C3_HALF_8192}
KAPPA = 0.01


def listed():
    return [
        # the paper's rotating pulse on the smallest grid, FP64, a whole 500-step run: each step
        # is a few thousand nodes, so latency and launches are all of it
        {"name": "pulse64_f64", "kind": "pulse", "pulse": "pulse64", "precision": "f64", "steps": 500},
        # one entry of the paper's Table 2 (N = 100): Dirichlet edges and a source field that
        # change every step, so the program calls the library three times per step
        {"name": "paper101_f64", "kind": "paper", "precision": "f64", "N": 100, "steps": 100},
        # a small transport problem on the caller's own velocity and diffusivity, no source
        {"name": "flow256_f32", "kind": "flow", "precision": "f32", "nx": 256, "ny": 256, "steps": 500, "src": "none"},
        # the variable-D pulse with its manufactured source: the accuracy workload ...
        {"name": "pulse1024_f32", "kind": "pulse", "pulse": "pulse1024", "precision": "f32", "steps": 200},
        # ... the benchmark's default grid ...
        {"name": "pulse4096_f32", "kind": "pulse", "pulse": "pulse4096", "precision": "f32", "steps": 100},
        # ... and the half-precision storage at the largest grid
        {"name": "pulse8192_f16", "kind": "pulse", "pulse": "pulse8192", "precision": "f16", "steps": 40},
        # a stationary source field on a ragged grid (the parity tests' large ragged size)
        {"name": "source1101x700_f32", "kind": "flow", "precision": "f32", "nx": 1101, "ny": 700, "steps": 100,
         "src": "field"},
        # bfloat16 storage on an odd width
        {"name": "flow2049x1537_bf16", "kind": "flow", "precision": "bf16", "nx": 2049, "ny": 1537, "steps": 60,
         "src": "none"},
        # a supervised run: stability check, mass and error against a reference on the way
        {"name": "monitor2048_f32", "kind": "monitor", "precision": "f32", "nx": 2048, "ny": 2048, "steps": 60,
         "every": 20},
        # parameter estimation: misfit and its gradient with respect to D (forward and adjoint)
        {"name": "adjoint512_f32", "kind": "adjoint", "precision": "f32", "n": 512, "steps": 200},
        # many uneven problems advanced together
        {"name": "batch48_f32", "kind": "batch", "precision": "f32", "count": 48, "layout": 0, "steps": 32},
        # populations handed in and out: a restart, or coupling with another code
        {"name": "restart513x384_f64", "kind": "restart", "precision": "f64", "nx": 513, "ny": 384, "steps": 20},
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["flow", "flow", "flow", "pulse", "pulse", "monitor", "adjoint", "batch", "restart", "paper"])
    precision = rng.choice(["f64", "f32", "f32", "f16", "bf16"])
    if kind == "batch":
        return {"kind": kind, "precision": rng.choice(["f32", "f16"]), "count": rng.randint(12, 48),
                "layout": rng.randint(1, 10**6), "steps": rng.randint(6, 32)}
    if kind == "paper":
        return {"kind": kind, "precision": rng.choice(["f64", "f32"]), "N": rng.randint(20, 120), "steps": rng.randint(20, 100)}
    if kind == "adjoint":
        n = log(64, 700)
        return {"kind": kind, "precision": rng.choice(["f32", "f64"]), "n": n, "steps": min(200, max(8, 16_000_000 // (n * n)))}
    # node updates of a pass that cost no more than the largest listed case
    budget = 2e7 if precision == "f64" else 4e8
    nx = log(32, 3000)
    ny = max(3, min(3000, int(nx * math.exp(rng.uniform(-0.7, 0.7)))))
    steps = int(max(4, min(rng.randint(40, 400), budget / (nx * ny))))
    if precision == "f64" and nx * ny * steps > 4 * budget:
        nx, ny = nx // 2, max(3, ny // 2)
    if kind == "pulse":
        return {"kind": kind, "pulse": "scaled", "precision": precision, "nx": nx, "ny": ny, "steps": steps}
    if kind == "monitor":
        return {"kind": kind, "precision": precision, "nx": nx, "ny": ny, "steps": steps, "every": max(1, steps // 3)}
    if kind == "restart":
        return {"kind": kind, "precision": precision, "nx": nx, "ny": ny, "steps": min(steps, 40)}
    return {"kind": kind, "precision": precision, "nx": nx, "ny": ny, "steps": steps, "src": rng.choice(["none", "none", "field"])}


# ------------------------------------------------------------------------- inputs

def modes(rng, ny, nx, count=6, kmax=4):
    """A smooth periodic field of max |value| 1 and its stream-function velocity, FP64 on the GPU."""
    x = torch.arange(nx, dtype=torch.float64, device=DEV) * (2 * math.pi / nx)
    y = (torch.arange(ny, dtype=torch.float64, device=DEV) * (2 * math.pi / ny))[:, None]
    f, u, v = (torch.zeros(ny, nx, dtype=torch.float64, device=DEV) for _ in range(3))
    for _ in range(count):
        kx, ky = (int(k) for k in rng.integers(1, kmax + 1, size=2))
        ph = float(rng.uniform(0, 2 * math.pi))
        arg = kx * x + ky * y + ph
        f += torch.cos(arg)
        u += -ky * torch.sin(arg)
        v += kx * torch.sin(arg)
    speed = torch.sqrt(u * u + v * v).max()
    return f / f.abs().max(), u / speed, v / speed


def flow_inputs(nx, ny, seed):
    """Lattice spacing and step of 1 / max(nx, ny) (unit lattice speed), |u| <= 0.2, tau1 - 1/2
    from 0.1 to 0.5, a positive phi0 and a source that changes phi by a few per cent a run."""
    rng = np.random.default_rng(seed)
    h = 1.0 / max(nx, ny)
    _, u, v = modes(rng, ny, nx)
    d, _, _ = modes(rng, ny, nx)
    p, _, _ = modes(rng, ny, nx)
    s, _, _ = modes(rng, ny, nx)
    D = h * (0.1 + 0.0667 * d)
    return {"dx": h, "dt": h, "ux": 0.2 * u, "uy": 0.2 * v, "D": D, "phi0": 1.0 + 0.3 * p, "S": 0.2 * s}


def pulse_of(case, seed):
    """The case's pulse, its centre, width and speed from the seed, and the grid's sides."""
    rng = np.random.default_rng(seed)
    how = dict(xc=float(rng.uniform(-0.5, 0.5)), yc=float(rng.uniform(-0.5, 0.5)), sigma0=float(rng.uniform(0.08, 0.12)))
    if case["pulse"] != "scaled":
        p = dataclasses.replace(PULSES[case["pulse"]], **how)
        return p, p.n, p.n
    n = max(case["nx"], case["ny"])
    p = W.Pulse(n=n, D_amp=0.5, courant=0.4, **how)
    # the relaxation times of the 1024^2 workload: D dt / dx^2 = 0.0922
    return dataclasses.replace(p, D0=0.0922 * p.dx**2 / p.dt), case["nx"], case["ny"]


def pulse_params(case, p, nx, ny, **more):
    fixed = {} if p.tau2 is None else {"tau2_mode": T.TRTR_TAU2_FIXED, "tau2": p.tau2}
    return T.Params(nx=nx, ny=ny, dx=p.dx, dt=p.dt, x0=p.x0, y0=p.y0, precision=T.PRECISIONS[case["precision"]],
                    src_mode=T.TRTR_SRC_PULSE if p.D_amp else T.TRTR_SRC_NONE,
                    grad_mode=T.TRTR_GRAD_ONESIDED_EDGE, **fixed, **more)


def flow_params(case, f, **more):
    return T.Params(nx=case["nx"], ny=case["ny"], dx=f["dx"], dt=f["dt"], x0=0.0, y0=0.0,
                    precision=T.PRECISIONS[case["precision"]], phi_ref=1.0, grad_mode=T.TRTR_GRAD_PERIODIC, **more)


def paper_inputs(case, seed):
    """The Sec. 3 benchmark: phi = a exp(-(x^2 + 3 y^2 + 2 kappa t)), its source at t = -dt .. and
    its edge values, the amplitude and kappa from the seed."""
    rng = np.random.default_rng(seed)
    amp, kappa = float(rng.uniform(0.5, 2.0)), KAPPA * float(rng.uniform(0.5, 2.0))
    p = W.PaperPulse(N=case["N"], kappa=kappa)
    x = p.x0 + p.dx * torch.arange(p.nx, dtype=torch.float64, device=DEV)
    X, Y = x[None, :].expand(p.ny, p.nx), x[:, None].expand(p.ny, p.nx)
    space = amp * torch.exp(-(X * X + 3 * Y * Y))
    t = p.time_step * torch.arange(-1, case["steps"] + 1, dtype=torch.float64, device=DEV)
    fade = torch.exp(-2 * kappa * t)[:, None, None]
    S = ((6 * kappa - 4 * X * Y - 4 * kappa * (X * X + 9 * Y * Y)) * space)[None] * fade
    return p, {"dx": p.dx, "dt": p.time_step, "ux": (-Y).contiguous(), "uy": X.contiguous(),
               "D": torch.full_like(space, kappa), "S": S.contiguous(), "phi": (space[None] * fade).contiguous()}


def adjoint_inputs(case, seed):
    p = dataclasses.replace(W.C5_ADJ_512, n=case["n"])
    p = dataclasses.replace(p, D0=W.C5_ADJ_512.D0 * 512 / p.n)  # the same relaxation times on every grid
    rng = np.random.default_rng(seed)
    p = dataclasses.replace(p, xc=float(rng.uniform(-0.5, 0.5)), yc=float(rng.uniform(-0.5, 0.5)))
    d, _, _ = modes(rng, p.n, p.n)
    x = p.x0 + p.dx * torch.arange(p.n, dtype=torch.float64, device=DEV)
    X, Y = x[None, :].expand(p.n, p.n), x[:, None].expand(p.n, p.n)
    phi0 = torch.exp(-((X - p.xc) ** 2 + (Y - p.yc) ** 2) / (2 * p.sigma0**2))
    f = {"dx": p.dx, "dt": p.dt, "ux": (-p.omega * Y).contiguous(), "uy": (p.omega * X).contiguous(),
         "D": p.D0 * (1 + 0.3 * d), "phi0": phi0}
    t = p.dt * case["steps"]
    c, s = math.cos(p.omega * t), math.sin(p.omega * t)
    s2 = p.sigma0**2 + 2 * p.D0 * t
    f["obs"] = (p.sigma0**2 / s2) * torch.exp(-((X - (p.xc * c - p.yc * s)) ** 2 + (Y - (p.xc * s + p.yc * c)) ** 2) / (2 * s2))
    return p, f


def batch_pulses(case, seed):
    """Uneven grids fixed by the case's layout; omega, sigma0 and D0 of each instance by the seed."""
    sizes = [b.pulse for b in W.batch_instances(seed=case["layout"], count=case["count"])]
    rng = np.random.default_rng(seed)
    return [dataclasses.replace(p, omega=float(rng.uniform(0.5 * math.pi, 2 * math.pi)), sigma0=float(rng.uniform(0.05, 0.15)),
                                D0=float(rng.uniform(1e-4, 1e-2))) for p in sizes]


def populations(nx, ny, f, seed):
    """Equilibria of phi0 plus one per cent of noise: a state that another code hands over."""
    g = equilibrium(f["phi0"], f["ux"] * f["dt"] / f["dx"], f["uy"] * f["dt"] / f["dx"])
    gen = torch.Generator(device=DEV).manual_seed(seed)
    return (g * (1 + 0.01 * (2 * torch.rand(g.shape, generator=gen, dtype=torch.float64, device=DEV) - 1))).contiguous()


# ------------------------------------------------------------------------- the cases

def prepare(case, seed):
    kind = case["kind"]
    out = OUT[case["precision"]]
    state = {"case": case, "out": out}
    if kind == "pulse":
        p, nx, ny = pulse_of(case, seed)
        s = T.Solver(pulse_params(case, p, nx, ny))
        s.set_pulse(p.omega, p.xc, p.yc, p.sigma0, p.D0, p.D_amp)
    elif kind in ("flow", "monitor", "restart"):
        nx, ny = case["nx"], case["ny"]
        f = flow_inputs(nx, ny, seed)
        field = case.get("src") == "field"
        s = T.Solver(flow_params(case, f, src_mode=T.TRTR_SRC_FIELD if field else T.TRTR_SRC_NONE,
                                 check_every=case.get("every", 0)))
        s.set_fields(f["ux"], f["uy"], f["D"], f["S"] if field else None)
        state["phi0"] = f["phi0"]
        if kind == "restart":
            state["g"] = populations(nx, ny, f, seed)
            state["pops"] = torch.empty_like(state["g"])
    elif kind == "paper":
        p, f = paper_inputs(case, seed)
        nx, ny = p.nx, p.ny
        s = T.Solver(T.Params(nx=nx, ny=ny, x0=p.x0, y0=p.y0, dx=p.dx, dt=p.time_step,
                              precision=T.PRECISIONS[case["precision"]], grad_mode=T.TRTR_GRAD_ONESIDED_EDGE,
                              src_mode=T.TRTR_SRC_FIELD, bc_mode=T.TRTR_BC_DIRICHLET_NEE))
        s.set_fields(f["ux"], f["uy"], f["D"], f["S"][1])
        state["f"] = f
    elif kind == "adjoint":
        p, f = adjoint_inputs(case, seed)
        nx = ny = p.n
        s = T.Solver(T.Params(nx=nx, ny=ny, dx=p.dx, dt=p.dt, precision=T.PRECISIONS[case["precision"]]))
        state["f"] = f
    else:
        pulses = batch_pulses(case, seed)
        b = T.Batch([T.pulse_instance(p, T.PRECISIONS[case["precision"]]) for p in pulses])
        state["batch"] = b
        state["views"] = [b.instance(k) for k in range(len(pulses))]
        state["phis"] = [torch.empty(p.n, p.n, dtype=torch.float64, device=DEV) for p in pulses]
        return state
    state["solver"] = s
    state["phi"] = torch.empty(ny, nx, dtype=torch.float64, device=DEV)
    return state


def run(state):
    case, out = state["case"], state["out"]
    kind, steps = case["kind"], case["steps"]
    if kind == "batch":  # the batch goes on from where it is
        state["batch"].step(steps)
        return [v.moments(phi).to(out) for v, phi in zip(state["views"], state["phis"])]
    s = state["solver"]
    if kind == "pulse":
        s.init_equilibrium(None)
        s.step(steps)
    elif kind == "flow":
        s.init_equilibrium(state["phi0"])
        s.step(steps)
    elif kind == "monitor":
        s.init_equilibrium(state["phi0"])
        seen = []
        for n in range(0, steps, case["every"]):
            s.step(min(case["every"], steps - n))
            seen += [s.mass(), s.error_vs(state["phi0"])[1]]
        return {"phi": s.moments(state["phi"]).to(out), "seen": torch.tensor(seen, dtype=torch.float32)}
    elif kind == "restart":
        s.set_populations(state["g"])
        s.step(steps)
        return s.get_populations(state["pops"]).to(out)
    elif kind == "paper":
        f = state["f"]
        s.set_source(f["S"][1])
        s.init_equilibrium(f["phi"][1])
        s.set_source_prev(f["S"][0])
        for n in range(steps):
            s.set_dirichlet(f["phi"][n + 2])
            s.step(1)
            if n + 1 < steps:
                s.set_source(f["S"][n + 2])
    else:
        f = state["f"]
        J, grad = A.misfit_and_gradient(s, f["ux"], f["uy"], f["D"], f["phi0"], f["obs"], steps)
        return {"J": J.to(out), "grad": grad.to(out)}
    return s.moments(state["phi"]).to(out)


def size_of(case):
    if case["kind"] == "batch":
        return sum(p.n * p.n for p in batch_pulses(case, 0))
    if case["kind"] == "paper":
        return (case["N"] + 1) ** 2
    if case["kind"] == "adjoint":
        return case["n"] ** 2
    if "nx" in case:
        return case["nx"] * case["ny"]
    return PULSES[case["pulse"]].n ** 2


def work(case):
    """Bytes: every input field, population and result once, in the type it is handed over or kept in.
    Flops: about 150 a node and step (moments, relaxation, rebuild), 30 more for the pulse's source,
    four times as many for a gradient (forward, recomputation, adjoint)."""
    n, steps, kind = size_of(case), case["steps"], case["kind"]
    c = 8 if case["precision"] == "f64" else 4
    per = 3 * c + 16  # u, D; phi0 and phi
    flops = 150 + (30 if kind == "pulse" and case["pulse"] != "pulse64" else 0)
    if kind == "restart":
        per = 3 * c + 2 * 72
    if kind == "paper":
        per += 8 * steps
    if kind == "monitor":
        per += 8 * -(-steps // case["every"])
    if kind == "adjoint":
        per, flops = 6 * 8, 4 * flops
    if case.get("src") == "field":
        per += c
    return {"bytes": float(n * per), "flops": float(n * steps * flops)}


# ------------------------------------------------------------------------- the scheme in FP64 torch

EX = (0, 1, -1, 0, 0, 1, -1, 1, -1)
EY = (0, 0, 0, 1, -1, 1, -1, -1, 1)
WT = (4 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 36, 1 / 36, 1 / 36, 1 / 36)


def equilibrium_of(q, phi, u, v):
    eu, uu = EX[q] * u + EY[q] * v, u * u + v * v
    return WT[q] * phi * (1 + 3 * eu + 4.5 * (eu * eu - uu / 3) + 4.5 * (eu**3 - eu * uu))


def equilibrium(phi, u, v):
    return torch.stack([equilibrium_of(q, phi, u, v) for q in range(9)])


def slope(f, axis, periodic):
    if periodic:
        return 0.5 * (torch.roll(f, -1, axis) - torch.roll(f, 1, axis))
    return torch.gradient(f, dim=axis, edge_order=1)[0]


class Exact:
    """The step of Eq. (14) in lattice units on [9, ny, nx] populations."""

    def __init__(self, dx, dt, ux, uy, D, periodic, tau2=None):
        self.u, self.v, self.dt = ux * dt / dx, uy * dt / dx, dt
        self.ax = self.u * slope(self.u, 1, periodic) + self.v * slope(self.u, 0, periodic)
        self.ay = self.u * slope(self.v, 1, periodic) + self.v * slope(self.v, 0, periodic)
        self.set_D(D * dt / dx**2, tau2)

    def set_D(self, Dh, tau2=None):
        self.w1 = 1 / (0.5 + 3 * Dh)
        self.w2 = 1 / (0.5 + (1 / 12) / (3 * Dh)) if tau2 is None else torch.full_like(Dh, 1 / tau2)

    def collide(self, g, Sn=None, Sp=None):
        u, v = self.u, self.v
        phi = g.sum(0)
        jx = sum(EX[q] * g[q] for q in range(9) if EX[q]) - phi * u
        jy = sum(EY[q] * g[q] for q in range(9) if EY[q]) - phi * v
        bxx = sum((EX[q] ** 2 - 1 / 3) * g[q] for q in range(9)) - phi * u * u
        byy = sum((EY[q] ** 2 - 1 / 3) * g[q] for q in range(9)) - phi * v * v
        bxy = sum(EX[q] * EY[q] * g[q] for q in range(5, 9)) - phi * u * v
        k1, k2, kh = 1 - self.w1, 1 - self.w2, 1 - 0.5 * self.w1
        mx, my = k1 * jx + kh * phi * self.ax, k1 * jy + kh * phi * self.ay
        s = 0.0
        if Sn is not None:
            s = self.dt * (1.5 * Sn - 0.5 * Sp)
            mx, my = mx + kh * u * s, my + kh * v * s
        out = []
        for q in range(9):
            ex, ey = EX[q], EY[q]
            second = (ex * ex - 1 / 3) * bxx + (ey * ey - 1 / 3) * byy + 2 * ex * ey * bxy
            out.append(equilibrium_of(q, phi, u, v) + WT[q] * (s + 3 * (ex * mx + ey * my) + 4.5 * k2 * second))
        return out

    def step(self, g, Sn=None, Sp=None):
        post = self.collide(g, Sn, Sp)
        return torch.stack([torch.roll(p, (EY[q], EX[q]), (0, 1)) for q, p in enumerate(post)])

    def hold_edges(self, g, phi_b):
        """Non-equilibrium extrapolation: edge nodes from their inward neighbours."""
        ny, nx = phi_b.shape
        edge = torch.ones(ny, nx, dtype=torch.bool, device=DEV)
        edge[1:-1, 1:-1] = False
        j, i = torch.nonzero(edge, as_tuple=True)
        fj, fi = j.clamp(1, ny - 2), i.clamp(1, nx - 2)
        gf = g[:, fj, fi]
        geq = lambda phi, jj, ii: equilibrium(phi, self.u[jj, ii], self.v[jj, ii])  # noqa: E731
        g[:, j, i] = geq(phi_b[j, i], j, i) + gf - geq(gf.sum(0), fj, fi)
        return g


def pulse_fields(p, nx, ny):
    x = p.x0 + p.dx * torch.arange(nx, dtype=torch.float64, device=DEV)
    y = p.y0 + p.dx * torch.arange(ny, dtype=torch.float64, device=DEV)
    X, Y = x[None, :].expand(ny, nx), y[:, None].expand(ny, nx)
    sx, cx, sy, cy = torch.sin(math.pi * X), torch.cos(math.pi * X), torch.sin(math.pi * Y), torch.cos(math.pi * Y)
    a = p.D0 * p.D_amp

    def phi(t):
        s2 = p.sigma0**2 + 2 * p.D0 * t
        cx_, cy_ = W.centre(p, t)
        return (p.sigma0**2 / s2) * torch.exp(-((X - cx_) ** 2 + (Y - cy_) ** 2) / (2 * s2))

    def source(t):
        s2 = p.sigma0**2 + 2 * p.D0 * t
        cx_, cy_ = W.centre(p, t)
        rx, ry = X - cx_, Y - cy_
        grad = a * math.pi * (cx * sy * rx + sx * cy * ry)
        return phi(t) / s2 * (grad - a * sx * sy * ((rx * rx + ry * ry) / s2 - 2))

    return -p.omega * Y, p.omega * X, p.D0 * (1 + p.D_amp * sx * sy), phi, source


def exact(case, seed):
    kind, steps = case["kind"], case["steps"]
    with torch.no_grad():
        if kind == "pulse":
            p, nx, ny = pulse_of(case, seed)
            ux, uy, D, phi, source = pulse_fields(p, nx, ny)
            m = Exact(p.dx, p.dt, ux, uy, D, False, p.tau2)
            g = equilibrium(phi(0.0), m.u, m.v)
            Sp = source(-p.dt) if p.D_amp else None
            for n in range(steps):
                Sn = source(n * p.dt) if p.D_amp else None
                g, Sp = m.step(g, Sn, Sp), Sn
            return g.sum(0)
        if kind in ("flow", "monitor", "restart"):
            f = flow_inputs(case["nx"], case["ny"], seed)
            m = Exact(f["dx"], f["dt"], f["ux"], f["uy"], f["D"], True)
            S = f["S"] if case.get("src") == "field" else None
            g = populations(case["nx"], case["ny"], f, seed) if kind == "restart" else equilibrium(f["phi0"], m.u, m.v)
            seen = []
            for n in range(1, steps + 1):
                g = m.step(g, S, S)
                if kind == "monitor" and (n % case["every"] == 0 or n == steps):
                    phi = g.sum(0)
                    seen += [float(phi.sum()), float((phi - f["phi0"]).norm() / f["phi0"].norm())]
            if kind == "monitor":
                return {"phi": g.sum(0), "seen": torch.tensor(seen, dtype=torch.float64)}
            return g if kind == "restart" else g.sum(0)
        if kind == "paper":
            p, f = paper_inputs(case, seed)
            m = Exact(f["dx"], f["dt"], f["ux"], f["uy"], f["D"], False)
            g = equilibrium(f["phi"][1], m.u, m.v)
            for n in range(steps):
                g = m.hold_edges(m.step(g, f["S"][n + 1], f["S"][n]), f["phi"][n + 2])
            return g.sum(0)
        if kind == "batch":
            phis = []
            for p in batch_pulses(case, seed):
                ux, uy, D, phi, _ = pulse_fields(p, p.n, p.n)
                m = Exact(p.dx, p.dt, ux, uy, D, False)
                g = equilibrium(phi(0.0), m.u, m.v)
                for _ in range(steps):
                    g = m.step(g)
                phis.append(g.sum(0))
            return phis
    p, f = adjoint_inputs(case, seed)
    D = f["D"].clone().requires_grad_(True)
    m = Exact(f["dx"], f["dt"], f["ux"], f["uy"], D.detach(), False)

    def some(g, D, count):
        m.set_D(D * f["dt"] / f["dx"] ** 2)
        for _ in range(count):
            g = m.step(g)
        return g

    g = equilibrium(f["phi0"], m.u, m.v)
    for n in range(0, steps, 10):
        g = checkpoint(some, g, D, min(10, steps - n), use_reentrant=False)
    J = 0.5 * torch.sum((g.sum(0) - f["obs"]) ** 2)
    J.backward()
    return {"J": J.detach(), "grad": D.grad}
