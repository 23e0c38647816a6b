"""Cases that stand for what a user of the two-phase DUGKS library runs.

A case names a problem of the paper's tests (Sec. 3), its mesh, the precision
and the calls made on it.  One pass is what a program does between two looks at
its results: bring a field (or a saved state) to the library, advance it, and
read the fields, the state, the diagnostics or the gradients back.  The library
takes and returns host arrays, so the host copies are part of a pass.

An FP32 simulation computes in FP32; the fields that a program reads back from
one are kept as float32 snapshots, except for the ensemble, which lands in
page-locked float64 buffers as the benchmark does it.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1802_02868_gb300 import autograd as A
from paper_1802_02868_gb300 import dugks
from paper_1802_02868_gb300 import inputs as I

FIELDS = ("phi", "rho", "ux", "uy", "p")


def listed():
    return [
        # the smallest call: a solver coupled step by step reloads a small saved
        # state, takes a step and saves it again; launches and copies count
        {"name": "restart_48x40_fp64", "call": "restart", "problem": "drop", "nx": 48, "ny": 40, "fp32": False, "steps": 1},
        # the stationary drop of the plain FP64 workload, between two outputs
        {"name": "drop_64_fp64", "call": "fields", "problem": "drop", "nx": 64, "ny": 64, "fp32": False, "steps": 100},
        # the same mesh in FP32: a step is a few microseconds of latency
        {"name": "drop_64_fp32", "call": "fields", "problem": "drop", "nx": 64, "ny": 64, "fp32": True, "steps": 400},
        # layered Poiseuille, 4 cells wide, tanh-stretched between walls
        {"name": "channel_4x256_fp64", "call": "fields", "problem": "channel", "nx": 4, "ny": 256, "fp32": False, "steps": 100},
        # the viscosity-ratio sweep as one batch in FP32
        {"name": "channel_sweep_fp32", "call": "fields", "problem": "channel_sweep", "nx": 4, "ny": 256, "fp32": True, "steps": 200},
        # the CFL sweep, odd sizes, each instance with its own step count
        {"name": "cfl_sweep_100_fp64", "call": "each", "problem": "cfl_sweep", "nx": 100, "ny": 100, "fp32": False, "steps": 24},
        # Rayleigh-Taylor between walls, FP32 and FP64
        {"name": "rt_256x1024_fp32", "call": "fields", "problem": "rt", "nx": 256, "ny": 1024, "fp32": True, "steps": 200},
        {"name": "rt_256x1024_fp64", "call": "fields", "problem": "rt", "nx": 256, "ny": 1024, "fp32": False, "steps": 20},
        # a large drop watched while it runs: sums, diagnostics, Laplace pressure
        {"name": "monitor_2048_fp32", "call": "monitor", "problem": "drop", "nx": 2048, "ny": 2048, "fp32": True, "steps": 40},
        # the batched ensemble of uneven squares, the flagship workload
        {"name": "ensemble_512_fp32", "call": "ensemble", "problem": "ensemble", "count": 512, "fp32": True, "steps": 60},
        # the gradient of the Rayleigh-Taylor loss, FP32 with checkpoints
        {"name": "grad_rt_256x512_fp32", "call": "grad", "problem": "rt", "nx": 256, "ny": 512, "fp32": True, "steps": 120, "every": 40},
        # a small FP64 gradient, as in a calibration loop
        {"name": "grad_rt_48x96_fp64", "call": "grad", "problem": "rt", "nx": 48, "ny": 96, "fp32": False, "steps": 40, "every": 10},
    ]


def draw(rng):
    def log_int(a, b):
        return int(round(math.exp(rng.uniform(math.log(a), math.log(b)))))

    kind = rng.choice(["restart", "drop", "drop", "channel", "channel_sweep", "cfl_sweep", "rt", "rt", "monitor",
                       "ensemble", "grad", "grad"])
    fp32 = rng.random() < 0.5
    if kind == "restart":
        return {"call": "restart", "problem": "drop", "nx": log_int(20, 300), "ny": log_int(20, 300), "fp32": fp32,
                "steps": rng.randint(1, 4)}
    if kind == "drop":
        return {"call": "fields", "problem": "drop", "nx": log_int(32, 640), "ny": log_int(32, 640), "fp32": fp32,
                "steps": rng.randint(60, 200) if fp32 else rng.randint(20, 80)}
    if kind == "channel":
        return {"call": "fields", "problem": "channel", "nx": rng.randint(3, 12), "ny": 2 * log_int(32, 256), "fp32": fp32,
                "steps": rng.randint(60, 200)}
    if kind == "channel_sweep":
        return {"call": "fields", "problem": "channel_sweep", "nx": rng.randint(3, 12), "ny": 2 * log_int(32, 192),
                "fp32": fp32, "steps": rng.randint(60, 200)}
    if kind == "cfl_sweep":
        n = rng.randint(60, 140)
        return {"call": "each", "problem": "cfl_sweep", "nx": n, "ny": n, "fp32": fp32, "steps": rng.randint(10, 40)}
    if kind == "rt":
        return {"call": "fields", "problem": "rt", "nx": log_int(48, 256), "ny": log_int(96, 1024), "fp32": fp32,
                "steps": rng.randint(50, 200) if fp32 else rng.randint(5, 20)}
    if kind == "monitor":
        return {"call": "monitor", "problem": "drop", "nx": log_int(200, 2048), "ny": log_int(200, 2048), "fp32": True,
                "steps": 10 * rng.randint(1, 4)}
    if kind == "ensemble":
        return {"call": "ensemble", "problem": "ensemble", "count": log_int(8, 256), "fp32": True, "steps": rng.randint(20, 60)}
    every = rng.randint(5, 30)
    return {"call": "grad", "problem": "rt", "nx": log_int(32, 256) if fp32 else log_int(24, 64),
            "ny": log_int(64, 512) if fp32 else log_int(48, 128), "fp32": fp32, "steps": rng.randint(20, 120) if fp32 else rng.randint(10, 40),
            "every": every}


# ---------------------------------------------------------------------------
# Inputs, from the seed alone
# ---------------------------------------------------------------------------
def _drop(case, rng):
    """A drop of the stationary-drop workload, off centre and slightly off its
    equilibrium width."""
    nx, ny = case["nx"], case["ny"]
    c = I.stationary_drop(n=8, radius=2.0, density_ratio=rng.uniform(4.0, 12.0))
    mesh = I.uniform_mesh(nx, ny)
    r = rng.uniform(0.2, 0.28) * min(nx, ny)
    phi = I.drop_field(mesh, r, (rng.uniform(0.45, 0.55) * nx, rng.uniform(0.45, 0.55) * ny), rng.uniform(3.6, 4.4))
    return [I.Case("drop", mesh, c.params, phi, steps=case["steps"])]


def _channel(case, rng, ratio):
    c = I.layered_poiseuille(nx=case["nx"], ny=case["ny"], height=float(case["ny"]), nu_ratio=ratio,
                             force=1e-6 * rng.uniform(0.8, 1.2))
    # released from an interface somewhat wider than its equilibrium width
    c.phi0 = np.ascontiguousarray(I.layered_field(c.mesh, 0.5 * case["ny"], rng.uniform(4.6, 5.4)))
    return c


def _cases(case, seed):
    rng = np.random.default_rng([seed, 77])
    kind = case["problem"]
    if kind == "drop":
        return _drop(case, rng)
    if kind == "channel":
        return [_channel(case, rng, 10.0)]
    if kind == "channel_sweep":
        return [_channel(case, rng, r) for r in (3.0, 10.0, 100.0, 1000.0)]
    if kind == "cfl_sweep":
        return I.cfl_sweep(n=case["nx"], radius=0.25 * case["nx"] * rng.uniform(0.9, 1.1), width=rng.uniform(3.8, 4.2))
    if kind == "rt":
        L = float(case["nx"])
        amp = [0.1 * L] + list(0.01 * L * rng.standard_normal(7))
        c = I.rayleigh_taylor(nx=case["nx"], ny=case["ny"], amplitudes=amp)
        return [c]
    raise ValueError(kind)


def _ensemble(case, seed):
    """Meshes and parameters of the batched ensemble; its fields are formed on
    the device (inputs.batched_ensemble forms them one numpy field at a time)."""
    rng = np.random.default_rng([seed, 78])
    sides = np.random.default_rng(1802).choice(np.asarray(I.BATCH_SIDES), case["count"])   # sizes are the case's, not the seed's
    beta, kappa = I.params_from_sigma_width(1e-3, 4.0)
    meshes, params, drops = [], [], []
    for side in map(int, sides):
        radius = float(rng.uniform(0.1, 0.25)) * side
        rhoA = 1.0 / float(np.exp(rng.uniform(math.log(2.0), math.log(20.0))))
        nu_ratio = float(rng.uniform(1.0, 100.0))
        bubble = bool(rng.integers(0, 2))
        gy = -10.0 * 1e-3 / ((1.0 - rhoA) * (2.0 * radius) ** 2) if bubble else 0.0
        meshes.append(I.uniform_mesh(side, side))
        params.append(I.Params(rhoA=rhoA, rhoB=1.0, nuA=0.1 * nu_ratio, nuB=0.1, mobility=0.1, beta=beta, kappa=kappa,
                               gy=gy, rho_ref=1.0 if bubble else 0.0, cfl=0.5))
        drops.append((side, radius, side / 3.0 if bubble else 0.5 * side))
    return meshes, params, drops


def prepare(case, seed):
    prec = dugks.FP32 if case["fp32"] else dugks.FP64
    if case["call"] == "ensemble":
        meshes, params, drops = _ensemble(case, seed)
        total = sum(s * s for s, _, _ in drops)
        phi = torch.empty(total, dtype=torch.float64).pin_memory()
        o = 0
        for s, r, yc in drops:
            x = torch.arange(s, dtype=torch.float64, device="cuda") + 0.5
            d = torch.sqrt((x[None, :] - 0.5 * s) ** 2 + (x[:, None] - yc) ** 2)
            phi[o:o + s * s].copy_((0.5 + 0.5 * torch.tanh(0.5 * (r - d))).reshape(-1))
            o += s * s
        out = [torch.empty(total, dtype=torch.float64).pin_memory() for _ in range(5)]
        return {"case": case, "sim": dugks.Sim(meshes, params, prec), "phi": phi.numpy(), "keep": (phi, out),
                "out": [t.numpy() for t in out]}
    cs = _cases(case, seed)
    one = len(cs) == 1
    if case["call"] == "grad":
        c = cs[0]
        target = _target(c, case, seed)
        typ = torch.float32 if case["fp32"] else torch.float64
        return {"case": case, "phi0": torch.tensor(c.phi0, dtype=typ).requires_grad_(),
                "kappa": torch.tensor(c.params.kappa, dtype=typ).requires_grad_(),
                "mobility": torch.tensor(c.params.mobility, dtype=typ).requires_grad_(),
                "problem": A.Problem(c.mesh, c.params, target, case["steps"], case["every"], prec)}
    state = {"case": case, "sim": dugks.Sim(cs[0].mesh if one else [c.mesh for c in cs], cs[0].params if one else [c.params for c in cs], prec),
             "phi": cs[0].phi0 if one else [c.phi0 for c in cs]}
    if case["call"] == "restart":
        state["f"], state["g"] = _saved(case, cs[0])
    if case["call"] == "each":
        state["counts"] = _counts(cs, case)
    return state


def _saved(case, c):
    """The saved state of a restart: step 1 of the procedure, in the precision of the run."""
    f, g = _Ref(c.mesh, c.params, "cpu").init(torch.as_tensor(c.phi0))
    dt = np.float32 if case["fp32"] else np.float64
    return tuple(a.numpy().astype(dt).astype(np.float64) for a in (f, g))


def _target(c, case, seed):
    """The field that the gradient's loss aims at: another interface."""
    rng = np.random.default_rng([seed, 79])
    L = float(case["nx"])
    return np.ascontiguousarray(I.rt_field(c.mesh, L, 0.5 * case["ny"], [0.12 * L] + list(0.01 * L * rng.standard_normal(7)), 4.0))


def _counts(cs, case):
    """Step counts that bring the sweep to one time, the fastest taking `steps`."""
    t = case["steps"] * max(c.params.cfl for c in cs)
    return [int(round(t / c.params.cfl)) for c in cs]


def _kept(case, d):
    """A snapshot as a program keeps it: in the precision of the run."""
    if not case["fp32"]:
        return d
    return {k: [a.astype(np.float32) for a in v] if isinstance(v, list) else v.astype(np.float32) for k, v in d.items()}


def run(state):
    case = state["case"]
    call = case["call"]
    if call == "grad":
        t = (state["phi0"], state["kappa"], state["mobility"])
        for x in t:
            x.grad = None
        loss = A.DugksLoss.apply(*t, state["problem"])
        loss.backward()
        return {"loss": loss.detach(), "phi0": t[0].grad, "kappa": t[1].grad, "mobility": t[2].grad}
    sim = state["sim"]
    if call == "restart":
        sim.set_state(state["f"], state["g"])
        sim.step(case["steps"])
        f, g = sim.state()
        return _kept(case, {"f": f, "g": g})
    sim.init(state["phi"])
    if call == "ensemble":
        sim.step(case["steps"])
        sums = sim.conservation()
        sim.moments(out=state["out"])
        return {"fields": dict(zip(FIELDS, state["out"])), "sum_phi": sums[0], "sum_rho": sums[1]}
    if call == "each":
        sim.step_each(state["counts"])
        return _kept(case, sim.moments())
    if call == "monitor":
        sums = []
        for _ in range(case["steps"] // 10):
            sim.step(10)
            sums.append(sim.conservation())
        return {"sums": np.asarray(sums), "diagnostics": sim.diagnostics_array(),
                "laplace": sim.laplace_pressure().astype(np.float32)}
    sim.step(case["steps"])
    return _kept(case, sim.moments())


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
FLOP = 2127          # of one cell update (Sec. 2.2, steps 2-7), FMA = 2, division = 1


def work(case):
    w = 4 if case["fp32"] else 8
    if case["call"] == "ensemble":
        cells = case["count"] * sum(s * s for s in I.BATCH_SIDES) // len(I.BATCH_SIDES)
    else:
        cells = case["nx"] * case["ny"]
    if case["problem"] in ("channel_sweep", "cfl_sweep"):
        cells *= 4
    steps = case["steps"]
    if case["call"] == "each":
        steps = steps * (1 + 2 + 4 + 8) / 4            # CFL 0.8, 0.4, 0.2, 0.1
    flops = float(FLOP) * cells * steps
    # the state is read and written once a step; the field in, the fields out
    size = cells * steps * (36 * w + 16) + cells * 8
    if case["call"] == "restart":
        size += cells * 35 * 8
    elif case["call"] == "monitor":
        size += cells * (9 * w + 8 + 4) + cells * 8 * (case["steps"] // 10)
    elif case["call"] == "grad":
        # forward, forward again from the checkpoints, and the reverse step (about three forward steps of arithmetic)
        flops *= 5
        size = cells * steps * 3 * (36 * w + 16) + cells * 8 * 2
    else:
        size += cells * 5 * 8
    return {"bytes": float(size), "flops": flops}


# ---------------------------------------------------------------------------
# The scheme in 64 bits with plain torch (Sec. 2.2), for `exact`
# ---------------------------------------------------------------------------
class _Axis:
    def __init__(self, d, wall, device):
        d = np.asarray(d, dtype=np.float64)
        n = d.size
        k = np.arange(n)
        km, kp = (k - 1) % n, (k + 1) % n
        dl, dr = 0.5 * (d + d[km]), 0.5 * (d + d[kp])
        has_m, has_p = np.ones(n, bool), np.ones(n, bool)
        if wall:
            km[0], kp[-1], dl[0], dr[-1] = 0, n - 1, d[0], d[-1]
            has_m[0] = has_p[-1] = False
        c1 = np.stack([-dr / (dl * (dl + dr)), (dr - dl) / (dl * dr), dl / (dr * (dl + dr))])
        c2 = np.stack([2 / (dl * (dl + dr)), -2 / (dl * dr), 2 / (dr * (dl + dr))])
        e1 = c1.copy()                                   # distributions: one-sided next to a wall
        only_p, only_m = has_p & ~has_m, has_m & ~has_p
        e1[:, only_p] = np.stack([0 * dr, -1 / dr, 1 / dr])[:, only_p]
        e1[:, only_m] = np.stack([-1 / dl, 1 / dl, 0 * dl])[:, only_m]

        def t(a):
            return torch.as_tensor(a, device=device)
        self.n, self.wall, self.d = n, wall, t(d)
        self.km, self.kp = t(km), t(kp)
        self.c1, self.c2, self.e1 = t(c1), t(c2), t(e1)
        lo = k[:-1] if wall else k                       # interior faces: between lo and its kp
        self.lo, self.hi = t(lo), t(kp[lo])
        s = d[lo] + d[kp[lo]]
        self.wL, self.wR, self.invd = t(d[kp[lo]] / s), t(d[lo] / s), t(2 / s)


class _Ref:
    """One instance; fields are [ny, nx], distributions [9, ny, nx]."""

    def __init__(self, mesh, prm, device):
        self.prm, self.dev = prm, device
        self.ax = (_Axis(mesh.dx, mesh.bc_x == I.WALL, device), _Axis(mesh.dy, mesh.bc_y == I.WALL, device))
        self.dt = prm.cfl * min(float(np.min(mesh.dx)), float(np.min(mesh.dy))) / math.sqrt(2.0)
        self.xi = torch.tensor([[0, 1, 0, -1, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1]], dtype=torch.float64, device=device)
        self.w = torch.tensor([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, dtype=torch.float64, device=device)[:, None, None]
        self.opp = torch.tensor([0, 3, 4, 1, 2, 7, 8, 5, 6], device=device)
        self.kappa = torch.tensor(prm.kappa, dtype=torch.float64, device=device)
        self.lam = torch.tensor(prm.mobility, dtype=torch.float64, device=device)

    def _x(self, v, a):
        """A per-position vector of axis a, against [ny, nx]."""
        return v if a == 0 else v[:, None]

    def _tri(self, F, c, a):
        x, dim = self.ax[a], -1 if a == 0 else -2
        return self._x(c[0], a) * F.index_select(dim, x.km) + self._x(c[1], a) * F + self._x(c[2], a) * F.index_select(dim, x.kp)

    def grad(self, F):
        return self._tri(F, self.ax[0].c1, 0), self._tri(F, self.ax[1].c1, 1)

    def lap(self, F):
        return self._tri(F, self.ax[0].c2, 0) + self._tri(F, self.ax[1].c2, 1)

    def mu(self, phi):
        p = self.prm
        return 4 * p.beta * (phi - p.phiA) * (phi - p.phiB) * (phi - 0.5 * (p.phiA + p.phiB)) - self.kappa * self.lap(phi)

    def rho(self, phi):
        p = self.prm
        return p.rhoB + (p.rhoA - p.rhoB) * (phi - p.phiB) / (p.phiA - p.phiB)

    def consts(self):
        p = self.prm
        rr = p.rhoA / p.rhoB
        return (p.rhoA - p.rhoB) / (p.phiA - p.phiB), (rr - 1) / (p.phiA - p.phiB * rr), 3 * self.lam / p.tau_g

    def tauf(self, phi, rho):
        p = self.prm
        ma, mb = p.rhoA * p.nuA, p.rhoB * p.nuB
        return 3 * ma * mb * (p.phiA - p.phiB) / ((phi - p.phiB) * mb + (p.phiA - phi) * ma) / rho

    def force(self, phi, rho, gm):
        p = self.prm
        return -phi * gm[0] + (rho - p.rho_ref) * p.gx, -phi * gm[1] + (rho - p.rho_ref) * p.gy

    def velocity_pressure(self, f, rho, F, gphi, lmu, tau, rest=False):
        """Eqs. u and P with half a step `tau` of the force."""
        drho, gam, _ = self.consts()
        if rest:
            ux = uy = torch.zeros_like(rho)
        else:
            m = torch.einsum("aq,qyx->ayx", self.xi, f)
            ux, uy = (m[0] + 0.5 * tau * F[0] / 3) * 3 / rho, (m[1] + 0.5 * tau * F[1] / 3) * 3 / rho
        p = f.sum(0) + 0.5 * tau / 3 * (drho * (ux * gphi[0] + uy * gphi[1]) - gam * rho * self.lam * lmu)
        return ux, uy, p

    def eq_src(self, phi, rho, ux, uy, p, mu, lmu, F, gphi, gp):
        drho, gam, eta = self.consts()
        cx, cy = self.xi[0][:, None, None], self.xi[1][:, None, None]
        w = self.w
        xu = cx * ux + cy * uy
        s = w * (3 * xu + 4.5 * xu * xu - 1.5 * (ux * ux + uy * uy))
        feq = w * p + rho / 3 * s
        H = w * eta * mu
        H = torch.cat([(phi - (1 - w[0]) * eta * mu)[None], H[1:]])
        geq = H + phi * s
        ex, ey = cx - ux, cy - uy
        Ff = (w + s) * (ex * F[0] + ey * F[1]) + s * (ex * gphi[0] + ey * gphi[1]) * drho / 3 - w * rho / 3 * gam * self.lam * lmu
        Fg = 3 * phi / rho * (w + s) * (ex * (F[0] - gp[0]) + ey * (F[1] - gp[1]))
        return feq, geq, Ff, Fg

    def init(self, phi):
        mu, rho = self.mu(phi), self.rho(phi)
        gm, gphi, zero = self.grad(mu), self.grad(phi), torch.zeros_like(phi)
        feq, geq, Ff, Fg = self.eq_src(phi, rho, zero, zero, zero, mu, self.lap(mu), self.force(phi, rho, gm), gphi, (zero, zero))
        return feq - 0.5 * self.dt * Ff, geq - 0.5 * self.dt * Fg

    def macros(self, f, g):
        phi = g.sum(0)
        mu, rho = self.mu(phi), self.rho(phi)
        gm, gphi, lmu = self.grad(mu), self.grad(phi), self.lap(mu)
        F = self.force(phi, rho, gm)
        ux, uy, p = self.velocity_pressure(f, rho, F, gphi, lmu, self.dt)
        return phi, rho, ux, uy, p, mu, gm, gphi, lmu, F

    def face(self, B, aux, A, wall_side=0):
        """Originals of both distributions at faces from their bar values B and
        the aux fields (mu, lap mu, grad mu, grad phi, grad p)."""
        h = 0.5 * self.dt
        fb, gb = B
        mu, lmu, gm, gphi, gp = aux
        phi = gb.sum(0)
        rho = self.rho(phi)
        F = self.force(phi, rho, gm)
        ux, uy, p = self.velocity_pressure(fb, rho, F, gphi, lmu, h, rest=bool(wall_side))
        feq, geq, Ff, Fg = self.eq_src(phi, rho, ux, uy, p, mu, lmu, F, gphi, gp)
        tf, tg = self.tauf(phi, rho), self.prm.tau_g
        return (2 * tf * fb + h * feq + tf * h * Ff) / (2 * tf + h), (2 * tg * gb + h * geq + tg * h * Fg) / (2 * tg + h)

    def step(self, f, g):
        dt, h, tg = self.dt, 0.5 * self.dt, self.prm.tau_g
        phi, rho, ux, uy, p, mu, gm, gphi, lmu, F = self.macros(f, g)
        gp = self.grad(p)
        feq, geq, Ff, Fg = self.eq_src(phi, rho, ux, uy, p, mu, lmu, F, gphi, gp)
        tf = self.tauf(phi, rho)
        bp = (((2 * tf - h) * f + 3 * h * feq + 3 * tf * h * Ff) / (2 * tf + dt),
              ((2 * tg - h) * g + 3 * h * geq + 3 * tg * h * Fg) / (2 * tg + dt))
        J = [torch.zeros_like(f), torch.zeros_like(g)]
        vol = self.ax[1].d[:, None] * self.ax[0].d
        for A in (0, 1):
            x, dim = self.ax[A], -1 if A == 0 else -2
            area = self._x(self.ax[1 - A].d, 1 - A)
            xn, xt = self.xi[A][:, None, None], self.xi[1 - A][:, None, None]
            wL, wR, invd = (self._x(v, A) for v in (x.wL, x.wR, x.invd))

            def at(F):
                return wL * F.index_select(dim, x.lo) + wR * F.index_select(dim, x.hi)
            B = [at(b) - h * (xn * (b.index_select(dim, x.hi) - b.index_select(dim, x.lo)) * invd
                              + xt * at(self._tri(b, self.ax[1 - A].e1, 1 - A))) for b in bp]
            aux = (at(mu), at(lmu), tuple(map(at, gm)), tuple(map(at, gphi)), tuple(map(at, gp)))
            for k, o in enumerate(self.face(B, aux, A)):
                fl = xn * area * o
                J[k] = J[k].index_add(f.dim() + dim, x.lo, fl).index_add(f.dim() + dim, x.hi, -fl)
            if not x.wall:
                continue
            for side, c in ((-1, 0), (1, x.n - 1)):
                i = torch.tensor([c], device=self.dev)
                inc = self.xi[A] * side < 0               # incoming: bounce-back
                off = (side * 0.5 * x.d[c] - h * self.xi[A])[:, None, None]
                B = []
                for b in bp:
                    v = (b.index_select(dim, i) + off * self._tri(b, x.e1, A).index_select(dim, i)
                         - h * xt * self._tri(b, self.ax[1 - A].e1, 1 - A).index_select(dim, i))
                    B.append(torch.where(inc[:, None, None], v[self.opp], v))

                def one(F):
                    return F.index_select(dim, i)

                def pair(G):
                    return tuple(torch.zeros_like(one(v)) if a == A else one(v) for a, v in enumerate(G))
                aux = (one(mu), one(lmu), pair(gm), pair(gphi), pair(gp))
                for k, o in enumerate(self.face(B, aux, A, side)):
                    o = torch.where(inc[:, None, None], o[self.opp], o)
                    J[k] = J[k].index_add(f.dim() + dim, i, side * xn * area * o)
        return tuple(4 / 3 * b - 1 / 3 * t - dt / vol * j for b, t, j in zip(bp, (f, g), J))

    def laplace(self, f, g):
        """The Laplace pressure field of Sec. 3.1."""
        phi, _, _, _, p, _, _, gphi, _, _ = self.macros(f, g)
        q = self.prm
        a, b = phi - q.phiA, phi - q.phiB
        psi, dpsi = q.beta * a * a * b * b, 2 * q.beta * a * b * (a + b)
        return phi * dpsi - psi - self.kappa * phi * self.lap(phi) + 0.5 * self.kappa * (gphi[0] ** 2 + gphi[1] ** 2) + p


def _fields(ref, f, g):
    return dict(zip(FIELDS, (v.cpu().numpy() for v in ref.macros(f, g)[:5])))


def exact(case, seed):
    call = case["call"]
    if call == "ensemble":
        return None                                       # minutes of 64-bit work
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    cs = _cases(case, seed)
    refs = [_Ref(c.mesh, c.params, dev) for c in cs]
    if call == "grad":
        c, r = cs[0], refs[0]
        typ = np.float32 if case["fp32"] else np.float64
        phi0 = torch.as_tensor(c.phi0.astype(typ).astype(np.float64), device=dev).requires_grad_()
        r.kappa = torch.tensor(float(typ(c.params.kappa)), dtype=torch.float64, device=dev).requires_grad_()
        r.lam = torch.tensor(float(typ(c.params.mobility)), dtype=torch.float64, device=dev).requires_grad_()
        f, g = r.init(phi0)
        for _ in range(case["steps"]):
            f, g = checkpoint(r.step, f, g, use_reentrant=False)
        loss = ((g.sum(0) - torch.as_tensor(_target(c, case, seed), device=dev)) ** 2).sum()
        loss.backward()
        return {"loss": loss.detach(), "phi0": phi0.grad, "kappa": r.kappa.grad, "mobility": r.lam.grad}
    counts = _counts(cs, case) if call == "each" else [case["steps"]] * len(cs)
    with torch.no_grad():
        state = [r.init(torch.as_tensor(c.phi0, device=dev)) for r, c in zip(refs, cs)]
        if call == "restart":
            st = _saved(case, cs[0])
            state = [tuple(torch.as_tensor(a, device=dev) for a in st)]
        sums = []
        for k, r in enumerate(refs):
            f, g = state[k]
            vol = r.ax[1].d[:, None] * r.ax[0].d
            for n in range(counts[k]):
                f, g = r.step(f, g)
                if call == "monitor" and (n + 1) % 10 == 0:
                    phi = g.sum(0)
                    sums.append((float((vol * phi).sum()), float((vol * r.rho(phi)).sum())))
            state[k] = (f, g)
        if call == "restart":
            return {"f": state[0][0].cpu().numpy(), "g": state[0][1].cpu().numpy()}
        if call == "monitor":
            return {"sums": np.asarray(sums), "diagnostics": None, "laplace": refs[0].laplace(*state[0]).cpu().numpy()}
        every = [_fields(r, *s) for r, s in zip(refs, state)]
        return every[0] if len(every) == 1 else {k: [e[k] for e in every] for k in FIELDS}

