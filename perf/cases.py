"""Timed cases of the porosity-wave solvers: what a program that uses this package has it do.

Kinds of case (one pass of `run` each):

  step    one physical time step of a `PTSolver` with a fixed number of PT iterations (FP64-lean or
          double-float form), as the time loop of a forward run takes it
  corr    one physical time step of the FP32 form with a fixed number of defect-correction rounds
          (`step_begin`, `iterate` per round, `step_end`), plain PT or multigrid correction solves
  batch   one physical time step of an ensemble of uneven instances (`PTBatch`)
  evolve  the porosity after a few steps and the gradient of its misfit w.r.t. the log-permeability
          field (`adjoint.evolve` and its backward)
  rx      one physical time step of the reactive solver with a fixed number of PT iterations
  rxmg    the same step by a fixed number of multigrid V-cycles

Inputs are seeded: one to three Gaussian porosity anomalies at random places (the ellipsoid setup
under background shear) on a background that varies smoothly by a few per cent, as rock does (over
an exactly uniform one the far pressures are rounding noise, and with them the weakening switch at
Pf = Pt), and a smooth random log-permeability field where the case has one. The single-precision
forms hand their iterate on in single precision; they and the ensembles solve the step from the
given state at every pass, the others go on in time.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import pt_inputs as I
from paper_2207_08716_gb300 import adjoint as A
from paper_2207_08716_gb300 import native as N
from paper_2207_08716_gb300.solver import PTBatch, PTSolver, RXSolver

FIELDS = N.FIELD_NAMES
ITERATE = ("Vx", "Vy", "Vz", "Pt", "Pf", "phi", "mu", "eta")
# of a single-precision iterate: eta jumps by the weakening factor where Pf - Pt changes sign, so
# that next to those surfaces it is a matter of rounding; the stresses follow from V and mu
HANDED_ON = ITERATE[:-1]
PRECISION = {"fp64": N.PT_FP64, "fp32": N.PT_FP32, "df64": N.PT_DF64}


def listed() -> list:
    return [
        # the 32^3 single-step workload: the smallest grid in use, where launches and latency count
        dict(name="fp64 c1 32", kind="step", form="fp64", nx=32, ny=32, nz=32, iters=300, shear=False, logk=False),
        # the background-shear setup (30 x 30 x 60 box, wall edges carry stress), native FP64
        dict(name="fp64 shear 127x127x254", kind="step", form="fp64", nx=127, ny=127, nz=254, iters=30, shear=True,
             logk=False),
        # an ordinary double-float run with a heterogeneous permeability
        dict(name="df64 127 logk", kind="step", form="df64", nx=127, ny=127, nz=127, iters=60, shear=False,
             logk=True),
        # the headline form at the thesis's production size (382^3 there, an odd grid here)
        dict(name="df64 383", kind="step", form="df64", nx=383, ny=383, nz=383, iters=30, shear=False, logk=False),
        # plain FP32 correction solves on a small grid, four rounds of a step
        dict(name="fp32 96", kind="corr", nx=96, ny=96, nz=96, rounds=4, iters=60, mg=0, logk=False),
        # the FP32 iteration at the benchmark grid
        dict(name="fp32 511", kind="corr", nx=511, ny=511, nz=511, rounds=1, iters=60, mg=0, logk=False),
        # rounds of a multigrid step on an odd grid: most of a converged step takes one V-cycle a round
        dict(name="fp32 mg 255", kind="corr", nx=255, ny=255, nz=255, rounds=4, iters=5, mg=5, logk=False),
        # ensembles of the batched workload's sizes, both precisions
        dict(name="batch fp64 24", kind="batch", form="fp64", members=24, iters=60),
        dict(name="batch fp32 24", kind="batch", form="fp32", members=24, iters=60),
        # gradient of a final-porosity misfit, power law on: forward, checkpoints and reverse sweep
        dict(name="evolve 63", kind="evolve", nx=63, ny=63, nz=63, steps=2, iters=150),
        # the reactive solver as the thesis ran it (FP32, n x n x 4n)
        dict(name="rx fp32 255x255x1020", kind="rx", form="fp32", nx=255, ny=255, nz=1020, iters=100),
        # its multigrid form
        dict(name="rx mg fp32 128x128x512", kind="rxmg", form="fp32", nx=128, ny=128, nz=512, levels=6, cycles=5),
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random) -> dict:
    kind = rng.choice(("step", "step", "step", "corr", "corr", "corr", "batch", "evolve", "rx", "rxmg"))
    if kind == "step":
        form = rng.choice(("df64", "df64", "fp64"))
        n = _log_int(rng, 24, 320 if form == "df64" else 200)
        nx, ny, nz = (max(16, int(n * rng.uniform(0.8, 1.2))) for _ in range(3))
        shear = rng.random() < 0.25
        cells = nx * ny * nz
        iters = 300 if cells < 1e5 else 60 if cells < 4e6 else 30
        return dict(kind=kind, form=form, nx=nx, ny=ny, nz=nz, iters=iters, shear=shear, logk=rng.random() < 0.3)
    if kind == "corr":
        n = _log_int(rng, 24, 400)
        nx, ny, nz = (max(16, int(n * rng.uniform(0.8, 1.2))) for _ in range(3))
        mg = 0 if rng.random() < 0.5 else max(2, min(6, int(math.log2(min(nx, ny, nz))) - 2))
        big = nx * ny * nz > 2e7
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, rounds=1 if big else 4, iters=5 if mg else 60, mg=mg,
                    logk=rng.random() < 0.3)
    if kind == "batch":
        return dict(kind=kind, form=rng.choice(("fp64", "fp32")), members=rng.randint(4, 24), iters=60)
    if kind == "evolve":
        n = _log_int(rng, 24, 80)
        nx, ny, nz = (max(16, int(n * rng.uniform(0.8, 1.2))) for _ in range(3))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, steps=rng.randint(1, 3), iters=90)
    if kind == "rx":
        form = rng.choice(("fp32", "fp64"))
        nx = _log_int(rng, 16, 255 if form == "fp32" else 128)
        ny = max(12, int(nx * rng.uniform(0.8, 1.0)))
        return dict(kind=kind, form=form, nx=nx, ny=ny, nz=4 * nx, iters=100)
    levels = rng.randint(2, 5)
    m = 1 << (levels - 1)
    nx = max(2, int(_log_int(rng, 16, 200) / m)) * m
    ny = max(2, int(nx * rng.uniform(0.8, 1.0) / m)) * m
    return dict(kind=kind, form="fp32" if rng.random() < 0.7 else "fp64", nx=nx, ny=ny, nz=4 * nx, levels=levels,
                cycles=5)


# ------------------------------------------------------------------------------------ inputs
def _background(p: dict, rs: np.random.Generator) -> torch.Tensor:
    """phi0 (1 + a few waves of random direction, length and phase, 4 % in all)."""
    ax = [(torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n for n in (p["nx"], p["ny"], p["nz"])]
    f = torch.ones((p["nz"], p["ny"], p["nx"]), dtype=torch.float64, device="cuda")
    for _ in range(4):
        k = rs.uniform(5.0, 30.0, size=3) * rs.choice([-1.0, 1.0], size=3)
        f += 0.01 * torch.sin((ax[2] * float(k[2]))[:, None, None] + (ax[1] * float(k[1]))[None, :, None]
                              + (ax[0] * float(k[0]) + float(rs.uniform(0.0, 6.28)))[None, None, :])
    return f * p["phi0"]


def _anomalies(p: dict, rs: np.random.Generator) -> torch.Tensor:
    """The background + 2 phi0 exp(-(r / 0.1)^2) around one to three seeded places, (nz, ny, nx)."""
    ax = [(torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n for n in (p["nx"], p["ny"], p["nz"])]
    phi = _background(p, rs)
    for _ in range(int(rs.integers(1, 4))):
        c = rs.uniform(0.2, 0.8, size=3)
        g = [torch.exp(-((x - float(v)) / 0.1) ** 2) for x, v in zip(ax, c)]
        phi += 2.0 * p["phi0"] * g[2][:, None, None] * g[1][None, :, None] * g[0][None, None, :]
    return phi


def _ellipsoid(p: dict, rs: np.random.Generator) -> torch.Tensor:
    """The background doubled in a flat ellipsoid in the lower part of the sheared box."""
    c = (0.5 + rs.uniform(-0.05, 0.05), 0.5 + rs.uniform(-0.05, 0.05), 0.2 + rs.uniform(-0.02, 0.02))
    ax = [((torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n - float(v)) * l / (0.5 * a)
          for n, v, l, a in zip((p["nx"], p["ny"], p["nz"]), c, (p["lx"], p["ly"], p["lz"]), (14.0, 14.0, 3.5))]
    r2 = ax[2][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[0][None, None, :] ** 2
    return torch.where(r2 <= 1.0, 2.0, 1.0) * _background(p, rs)


def _logk(p: dict, seed: int) -> torch.Tensor:
    """Smooth random field of correlation length 0.1 and standard deviation 0.5."""
    shape = (p["nz"], p["ny"], p["nx"])
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    w = torch.fft.rfftn(torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen))
    ks = [torch.fft.fftfreq(n, d=1.0 / n, dtype=torch.float64, device="cuda") for n in shape[:2]]
    ks.append(torch.fft.rfftfreq(shape[2], d=1.0 / shape[2], dtype=torch.float64, device="cuda"))
    for d, k in enumerate(ks):
        w *= torch.exp(-0.5 * (2 * math.pi * 0.1 * k) ** 2).reshape([-1 if e == d else 1 for e in range(3)])
    f = torch.fft.irfftn(w, s=shape)
    f -= f.mean()
    return f * (0.5 / f.std())


def _params(case: dict) -> dict:
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    p = I.shear_params(nx, ny, nz) if case.get("shear") else I.c1_params(nx, ny, nz)
    p.update(tol=0.0, max_iter=case["iters"])
    return p


def _pt_inputs(case: dict, seed: int) -> tuple:
    p = _params(case)
    rs = np.random.default_rng(seed)
    phi = _ellipsoid(p, rs) if case.get("shear") else _anomalies(p, rs)
    return p, phi, (_logk(p, seed) if case.get("logk") else None)


def _members(case: dict, seed: int) -> list:
    """The batched workload's ensemble (uneven grids, weakening, porosity and anomalies per member)."""
    sizes = np.random.default_rng(0).choice([32, 48, 64, 96, 127], size=case["members"])  # the same work for every seed
    rs = np.random.default_rng(seed)
    out = []
    for n in sizes:
        p = I.c1_params(int(n))
        p.update(R_weak=float(rs.uniform(0.01, 0.2)), phi0=float(rs.uniform(0.005, 0.02)), tol=0.0,
                 max_iter=case["iters"])
        out.append((p, _anomalies(p, rs)))
    return out


def _rx_inputs(case: dict, seed: int) -> tuple:
    p = I.rx_params(case["nx"], case["ny"], case["nz"])
    p.update(tol=0.0, max_iter=case.get("iters", 20000), precision=PRECISION[case["form"]])
    rs = np.random.default_rng(seed)
    ax = [(torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) / n for n in (p["nx"], p["ny"], p["nz"])]
    phi = torch.full((p["nz"], p["ny"], p["nx"]), p["phi0"], dtype=torch.float64, device="cuda")
    for zc, amp in ((0.1, 1.5), (0.23, 0.75)):
        c = (0.5 + rs.uniform(-0.05, 0.05), 0.5 + rs.uniform(-0.05, 0.05), zc + rs.uniform(-0.01, 0.01))
        g = [torch.exp(-((x - float(v)) / r) ** 2) for x, v, r in zip(ax, c, (0.12, 0.12, 0.03))]
        phi += amp * p["phi0"] * g[2][:, None, None] * g[1][None, :, None] * g[0][None, None, :]
    return p, torch.zeros_like(phi), phi, torch.full_like(phi, 0.5 * p["xs_max"])


def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    if kind in ("step", "corr"):
        p, phi, logk = _pt_inputs(case, seed)
        p["precision"] = PRECISION[case.get("form", "fp32")]
        p["mg_levels"] = case.get("mg", 0)
        s = PTSolver(p, phi, logk=logk)
        return dict(case=case, solver=s, start=_saved([s.f]) if kind == "corr" else None)
    if kind == "batch":
        s = PTBatch(_members(case, seed), precision=PRECISION[case["form"]])
        return dict(case=case, solver=s, start=_saved(s.f))
    if kind == "evolve":
        p, phi, _ = _pt_inputs(case, seed)
        logk = _logk(p, seed)
        return dict(case=case, params=p, phi=phi, logk=logk, target=phi * (1.0 + 0.05 * _logk(p, seed + 1)))
    p, Pf, phi, Xs = _rx_inputs(case, seed)
    mg = dict(levels=case["levels"], nu_pre=2, nu_post=2, nu_coarse=30, max_cycles=50,
              omega=6.0 / 7.0) if kind == "rxmg" else None
    return dict(case=case, solver=RXSolver(p, Pf, phi, Xs, mg=mg))


# -------------------------------------------------------------------------------------- passes
def _saved(fields: list) -> tuple:
    """The given state: porosity and viscosities; velocities, pressures and stresses are zero."""
    own = [f[k] for f in fields for k in ("phi", "mu", "eta")]
    rest = [f[k] for f in fields for k in FIELDS if k not in ("phi", "mu", "eta")]
    return own, [t.clone() for t in own], rest


def _restore(start: tuple) -> None:
    torch._foreach_copy_(start[0], start[1])
    torch._foreach_zero_(start[2])


def _natural(s: PTSolver, name: str) -> torch.Tensor:
    dz, dy, dx = {"Vx": (0, 0, 1), "Vy": (0, 1, 0), "Vz": (1, 0, 0), "txy": (0, 1, 1), "txz": (1, 0, 1),
                  "tyz": (1, 1, 0)}.get(name, (0, 0, 0))
    return s.f[name][: s.nz + dz, : s.ny + dy, : s.nx + dx]


def run(state: dict):
    case = state["case"]
    kind = case["kind"]
    if kind == "evolve":
        logk = state["logk"].detach().requires_grad_(True)
        phi = A.evolve(logk, state["params"], state["phi"], case["steps"])
        ((phi - state["target"]) ** 2).sum().backward()
        return dict(phi=phi.detach(), grad=logk.grad)
    s = state["solver"]
    if kind == "step":
        s.step()
        return {k: _natural(s, k) for k in FIELDS}
    if kind == "corr":
        _restore(state["start"])
        s.step_begin()
        for _ in range(case["rounds"]):
            s.iterate(0, case["iters"])
        s.step_end()
        return {k: _natural(s, k).float() for k in HANDED_ON}
    if kind == "batch":
        _restore(state["start"])
        s.step()
        dtype, names = (torch.float32, HANDED_ON) if case["form"] == "fp32" else (torch.float64, ITERATE)
        return {k: torch.cat([f[k][:n[2], :n[1], :n[0]].reshape(-1) for f, n in zip(s.f, s.shape)]).to(dtype)
                for k in names}
    if kind == "rx":
        s.step()
    else:
        s.mg_cycles(case["cycles"])
    out = {k: s.f[k][: s.nz, : s.ny, : s.nx] for k in ("Pf", "phi", "Xs")}
    return {k: v.float() for k, v in out.items()} if case["form"] == "fp32" else out


# ------------------------------------------------------------------------------------- its work
def work(case: dict) -> dict:
    """Bytes: the effective access A_eff of the thesis per iteration (unknown fields read and
    written, known ones read: 25 values per cell, 7 for the reactive solver) at the form's width;
    operations counted from the equations."""
    kind = case["kind"]
    width = 4 if case.get("form") == "fp32" or kind == "corr" else 8
    if kind == "batch":
        cells = sum(p["nx"] ** 3 for p in ({"nx": int(n)} for n in np.random.default_rng(0).choice(
            [32, 48, 64, 96, 127], size=case["members"])))
        return dict(bytes=25.0 * cells * width * case["iters"], flops=200.0 * cells * case["iters"])
    cells = float(case["nx"] * case["ny"] * case["nz"])
    if kind == "rx":
        return dict(bytes=7.0 * cells * width * case["iters"], flops=90.0 * cells * case["iters"])
    if kind == "rxmg":   # four finest sweeps, a restriction and a prolongation a cycle, coarse grids an eighth each
        n = cells * 8.0 / 7.0 * case["cycles"]
        return dict(bytes=6 * 7.0 * n * width, flops=5 * 90.0 * n)
    if kind == "evolve":   # as many adjoint iterations as forward ones
        n = cells * case["steps"] * case["iters"]
        return dict(bytes=2 * 25.0 * n * 8, flops=400.0 * n)
    if kind == "corr":     # the FP64 state is read and written once a round besides
        sweeps = case["iters"] * (8.0 / 7.0 if case["mg"] else 1.0)
        return dict(bytes=cells * case["rounds"] * (25.0 * 4 * sweeps + 25.0 * 8),
                    flops=cells * case["rounds"] * (180.0 * sweeps + 400.0))
    return dict(bytes=25.0 * cells * width * case["iters"], flops=200.0 * cells * case["iters"])


# ----------------------------------------------------------------------------- 64-bit references
def _diff(a: torch.Tensor, d: int) -> torch.Tensor:
    n = a.shape[d] - 1
    return a.narrow(d, 1, n) - a.narrow(d, 0, n)


def _mean(a: torch.Tensor, d: int) -> torch.Tensor:
    n = a.shape[d] - 1
    return 0.5 * (a.narrow(d, 1, n) + a.narrow(d, 0, n))


def _pad(a: torch.Tensor, *dims: int) -> torch.Tensor:
    pads = [0, 0, 0, 0, 0, 0]
    for d in dims:
        pads[2 * (2 - d)] = pads[2 * (2 - d) + 1] = 1
    return torch.nn.functional.pad(a, pads)


def _edge_mu(mu: torch.Tensor, d: int, e: int) -> torch.Tensor:
    """Mean over the centres next to each edge (in the d, e plane) that lie inside the grid."""
    one = torch.ones_like(mu)
    s, n = _pad(mu, d, e), _pad(one, d, e)
    return (_mean(_mean(s, d), e)) / (_mean(_mean(n, d), e))


def _neighbour_max(k: torch.Tensor) -> torch.Tensor:
    m = k.clone()
    for d in range(3):
        n = k.shape[d] - 1
        hi, lo = k.narrow(d, 1, n), k.narrow(d, 0, n)
        m.narrow(d, 0, n).copy_(torch.maximum(m.narrow(d, 0, n), hi))
        m.narrow(d, 1, n).copy_(torch.maximum(m.narrow(d, 1, n), lo))
    return m


class _Exact:
    """The implicit step's PT iteration (thesis Art. 1, Eqs. 17-27) on whole arrays in 64 bits;
    axes (z, y, x), velocities on faces, shear stresses on edges."""

    def __init__(self, p: dict, phi: torch.Tensor, logk):
        self.p = p
        nz, ny, nx = phi.shape
        z = lambda *s: torch.zeros(s, dtype=torch.float64, device=phi.device)  # noqa: E731
        self.r = (p["nz"] / p["lz"], p["ny"] / p["ly"], p["nx"] / p["lx"])
        h = min(1.0 / v for v in self.r)
        self.h2 = h * h
        self.V = [z(nz + 1, ny, nx), z(nz, ny + 1, nx), z(nz, ny, nx + 1)]
        self.R = [torch.zeros_like(v) for v in self.V]
        self.Pt, self.Pf, self.phi = z(nz, ny, nx), z(nz, ny, nx), phi.clone()
        self.mu = torch.full_like(phi, p["mu0"])
        self.eta = p["eta0"] * p["mu0"] / phi
        self.K0 = p["k0"] * torch.exp(logk) if logk is not None else p["k0"]
        self.tau = [z(nz, ny, nx) for _ in range(3)]                       # zz, yy, xx
        self.tas = {(1, 2): z(nz, ny + 1, nx + 1), (0, 2): z(nz + 1, ny, nx + 1), (0, 1): z(nz + 1, ny + 1, nx)}
        self.dt_cum, self.steps = 0.0, 0
        self.damp = (p["damp_z"], p["damp_y"], p["damp_x"])
        self.dtauv = p["cfl_v"] * self.h2 * p["rho_i"] / (1.0 + p["beta_n"])
        self.dtaupt = p["dtpt_scale"] * (1.0 + p["beta_n"]) / p["nz"]
        self.ifac = 1.0 / (p["cfl_pf"] * self.h2 * (1.0 + p["beta_d"] * p["B"] / p["alpha"]))
        self.buoy = p["rhof_g"] - (p["phi0"] * p["rhof_g"] + (1.0 - p["phi0"]) * p["rhos_g"])

    def begin(self):
        p = self.p
        self.Pto, self.Pfo, self.Lo = self.Pt.clone(), self.Pf.clone(), torch.log(1.0 - self.phi)
        self.Gdt = float(self.mu.max()) / p["xsi_w"]
        if self.steps == 0 or self.dt_cum >= self.Gdt / p["G"]:
            self.tauo = [t.clone() for t in self.tau]
            self.taso = {k: t.clone() for k, t in self.tas.items()}
            self.dt_cum = 0.0
        self.steps += 1

    def stresses(self, V, mu, old, olds, extra, bg):
        """Maxwell stresses of the velocities V (Eq. 21); `extra` joins the normal strain rates."""
        g = [_diff(v, d) * self.r[d] for d, v in enumerate(V)]
        div = g[0] + g[1] + g[2]
        xi = mu / self.Gdt
        tau = [(o * xi + 2.0 * mu * (e - div / 3.0 + extra)) / (1.0 + xi) for o, e in zip(old, g)]
        tas = {}
        for (d, e) in ((1, 2), (0, 2), (0, 1)):
            rate = 0.5 * (_pad(_diff(V[e], d), d) * self.r[d] + _pad(_diff(V[d], e), e) * self.r[e])
            inner = torch.zeros_like(rate)
            inner.narrow(d, 1, rate.shape[d] - 2).narrow(e, 1, rate.shape[e] - 2).fill_(1.0)
            m = _edge_mu(mu, d, e)
            on = 1.0 if (bg and (d, e) == (1, 2)) else inner
            rate = rate * inner + (0.5 * self.p["tau_bg"] / self.p["mu0"] if (bg and (d, e) == (1, 2)) else 0.0)
            x = m / self.Gdt
            tas[(d, e)] = on * (olds[(d, e)] * x + 2.0 * m * rate) / (1.0 + x)
        return div, tau, tas

    def perm(self):
        return self.K0 * (self.phi / self.p["phi0"]) ** 3

    def darcy(self, k, Pf, buoy):
        div = 0.0
        for d in range(3):
            q = -_mean(k, d) * (_diff(Pf, d) * self.r[d] + (buoy if d == 0 else 0.0))
            div = div + _diff(_pad(q, d), d) * self.r[d]
        return div

    def momentum(self, tau, tas, P, phi=None):
        """Momentum residual on the inner faces (Eq. 19), zero on the walls."""
        F = []
        for d in range(3):
            f = _diff(tau[d], d) * self.r[d] - _diff(P, d) * self.r[d]
            for e in range(3):
                if e != d:
                    t = _diff(tas[(min(d, e), max(d, e))], e) * self.r[e]
                    f = f + t.narrow(d, 1, t.shape[d] - 2)
            if d == 0 and phi is not None:
                f = f - (_mean(phi, 0) - self.p["phi0"]) * (self.p["rhof_g"] - self.p["rhos_g"])
            F.append(_pad(f, d))
        return F

    def residuals(self, cc, k):
        p = self.p
        div = sum(_diff(v, d) * self.r[d] for d, v in enumerate(self.V))
        a, b = p["beta_d"] / p["dt"], p["beta_d"] * p["alpha"] / p["dt"]
        dPt, dPf = self.Pt - self.Pto, self.Pf - self.Pfo
        rpt = div + a * dPt - b * dPf + (self.Pt - self.Pf) * cc
        rpf = self.darcy(k, self.Pf, self.buoy) + b * (dPf / p["B"] - dPt) + (self.Pf - self.Pt) * cc
        return rpt, rpf

    def porosity(self, phi, Pt1, Pf1):
        p = self.p
        om = 1.0 - phi
        adv = 0.0
        for d in range(3):
            v = self.V[d].narrow(d, 1, om.shape[d] - 1)
            f = v * _diff(om, d) * self.r[d]
            adv = adv + 2.0 * _mean(_pad(f, d), d)
        adv = 0.5 * adv / om
        comp = (Pf1 - Pt1) / self.eta if p["compaction_on"] else 0.0
        L = self.Lo - p["dt"] * (p["beta_phi"] * ((Pf1 - self.Pfo) - (Pt1 - self.Pto)) / p["dt"] + comp + adv)
        return 1.0 - torch.exp(L)

    def picard(self, tau, tas):
        p = self.p
        t2 = 0.5 * sum(t * t for t in tau) + sum(_mean(_mean(t, d), e) ** 2 for (d, e), t in tas.items())
        mus = p["mu0"] / (1.0 + (torch.sqrt(t2) / p["tau0"]) ** (p["n_pow"] - 1.0) if p["powerlaw_on"] else 1.0)
        r = torch.log(mus / self.mu)
        self.mu = self.mu * torch.exp(p["rel_mu"] * r)
        R = 1.0 + (p["R_weak"] - 1.0) * (self.Pf > self.Pt).double()
        e = torch.log(p["eta0"] * self.mu * R / (self.phi * self.eta))
        self.eta = self.eta * torch.exp(p["rel_eta"] * e)
        return max(float(r.abs().max()), float(e.abs().max()))

    def compaction(self):
        return 1.0 / (self.eta * (1.0 - self.phi)) if self.p["compaction_on"] else torch.zeros_like(self.phi)

    def iterate(self, n: int):
        p = self.p
        a, b = p["beta_d"] / p["dt"], p["beta_d"] * p["alpha"] / p["dt"]
        for it in range(1, n + 1):
            k, cc = self.perm(), self.compaction()
            rpt, rpf = self.residuals(cc, k)
            Pt1 = self.Pt - rpt / (1.0 / (self.dtaupt * self.mu) + a + cc)
            Pf1 = self.Pf - rpf / (_neighbour_max(k) * self.ifac + b / p["B"] + cc)
            _, tau, tas = self.stresses(self.V, self.mu, self.tauo, self.taso, p["beta_n"] * rpt, p["tau_bg"] != 0.0)
            phi1 = self.porosity(self.phi, Pt1, Pf1)
            F = self.momentum(tau, tas, Pt1, self.phi)
            self.relax(self.V, self.R, F, self.mu)
            self.Pt, self.Pf, self.phi = Pt1, Pf1, phi1
            if it % p["nup"] == 0:
                self.picard(tau, tas)

    def relax(self, V, R, F, mu):
        for d in range(3):
            R[d] = F[d] / self.p["rho_i"] + self.damp[d] * R[d]
            V[d] = V[d] + _pad(_mean(self.dtauv / mu, d), d) * R[d]

    def correct(self, rounds: int, n: int):
        """Rounds of the defect correction: 64-bit residuals, Picard update, n PT iterations on the
        correction of the linearised system, update, porosity."""
        p = self.p
        a, b = p["beta_d"] / p["dt"], p["beta_d"] * p["alpha"] / p["dt"]
        omega, before = 1.0, 0.0
        for _ in range(rounds):
            k, cc = self.perm(), self.compaction()
            rpt, rpf = self.residuals(cc, k)
            idtp = 1.0 / (self.dtaupt * self.mu)
            _, tau, tas = self.stresses(self.V, self.mu, self.tauo, self.taso, p["beta_n"] * rpt, p["tau_bg"] != 0.0)
            rF = self.momentum(tau, tas, self.Pt, self.phi)
            r = max(float(x.abs().max()) for x in (rpt, rpf, *rF))
            r = max(r, self.picard(tau, tas))
            if before > 0.0:
                omega = max(0.5 * omega, 0.0625) if r > 2.0 * before else min(1.25 * omega, 1.0) if r < before else omega
            before = r
            dV, R = [torch.zeros_like(v) for v in self.V], [torch.zeros_like(v) for v in self.V]
            dPt, dPf = torch.zeros_like(self.Pt), torch.zeros_like(self.Pf)
            kf, cpl = _neighbour_max(k) * self.ifac, b + cc
            zero, zeros = [0.0] * 3, {e: 0.0 for e in self.tas}
            for _ in range(n):
                div = sum(_diff(v, d) * self.r[d] for d, v in enumerate(dV))
                rho = rpt + div + (a + cc) * dPt - cpl * dPf
                rhf = rpf + self.darcy(k, dPf, 0.0) + (b / p["B"] + cc) * dPf - cpl * dPt
                _, tau, tas = self.stresses(dV, self.mu, zero, zeros, p["beta_n"] * (rho - rpt), False)
                dPt1 = dPt - rho / (idtp + a + cc)
                dPf = dPf - rhf / (kf + b / p["B"] + cc)
                dPt = dPt1
                F = [f + g for f, g in zip(rF, self.momentum(tau, tas, dPt))]
                self.relax(dV, R, F, self.mu)
            self.V = [v + omega * w for v, w in zip(self.V, dV)]
            self.Pt, self.Pf = self.Pt + omega * dPt, self.Pf + omega * dPf
            self.phi = self.porosity(self.phi, self.Pt, self.Pf)

    def end(self):
        rpt, _ = self.residuals(self.compaction(), self.perm())
        _, self.tau, self.tas = self.stresses(self.V, self.mu, self.tauo, self.taso, self.p["beta_n"] * rpt,
                                              self.p["tau_bg"] != 0.0)
        self.dt_cum += self.p["dt"]

    def fields(self) -> dict:
        return dict(Vx=self.V[2], Vy=self.V[1], Vz=self.V[0], Pt=self.Pt, Pf=self.Pf, phi=self.phi, mu=self.mu,
                    eta=self.eta, txx=self.tau[2], tyy=self.tau[1], tzz=self.tau[0], txy=self.tas[(1, 2)],
                    txz=self.tas[(0, 2)], tyz=self.tas[(0, 1)])


def _rx_exact(p: dict, Pf, phi, Xs) -> dict:
    """The reactive PT iteration (thesis Art. 3, Eqs. 8-10) on whole arrays in 64 bits."""
    r = (p["nz"] / p["lz"], p["ny"] / p["ly"], p["nx"] / p["lx"])
    h2 = min(1.0 / v for v in r) ** 2
    dt, tau = p["dt"], p["tau"]
    s = (1.0 - p["rhos"] / (p["rhof"] * (1.0 + p["dX"]))) * (1.0 + p["dX"])
    Pfo, phio, Xso = Pf, phi, Xs
    bp_of = lambda f: f * p["beta_f"] + p["beta_d"] - (1.0 + f) * p["beta_s"]  # noqa: E731
    k_of = lambda f: p["k0"] * (f / p["phi0"]) ** 3                            # noqa: E731
    dtau = h2 / float((k_of(phi) / bp_of(phi)).max()) / p["cfl_div"]
    for it in range(1, p["max_iter"] + 1):
        k, bp, w = k_of(phi), bp_of(phi), 1.0 / (1.0 - phi)
        div = 0.0
        for d in range(3):
            q = -_mean(k, d) * (_diff(Pf, d) * r[d] - (p["rhof"] * p["g"] if d == 0 else 0.0))
            div = div + _diff(_pad(q, d), d) * r[d]
        xr = p["beta_x"] * Pf + 0.5 * p["xs_max"]
        xeq = xr.clamp(0.0, p["xs_max"])
        dXs = (xeq - Xs) / tau
        src = s * (1.0 - phi) / (1.0 - Xs)
        comp = Pf * w / p["eta"]
        R = (-div - comp + src * dXs) / bp
        slope = p["beta_x"] * ((xr > 0) & (xr < p["xs_max"])).double()
        a = (w / p["eta"] - src * slope / tau) / bp
        Pf1 = Pf + dtau * (R - (Pf - Pfo) / dt) / (1.0 + dtau * (1.0 / dt + a))
        rate = (1.0 - phi) * ((p["beta_d"] - p["beta_s"] * w) * R + comp - (1.0 + p["dX"]) / (1.0 - Xs) * dXs)
        phi = (phio + dt * rate).clamp(1e-4, 1.0)
        Xs = (Xso + dt / tau * xeq) / (1.0 + dt / tau)
        Pf = Pf1
        if it % p["nup"] == 0:
            dtau = h2 / float((k_of(phi) / bp_of(phi)).max()) / p["cfl_div"]
    return dict(Pf=Pf, phi=phi, Xs=Xs)


def exact(case: dict, seed: int):
    kind = case["kind"]
    if kind == "rxmg" or case.get("mg") or (kind == "batch" and case["form"] == "fp32"):
        return None   # V-cycle hierarchies and data-dependent inner stops: their whole arrays take too long here
    if kind == "rx":
        return _rx_exact(*_rx_inputs(case, seed))
    if kind == "batch":
        out = {k: [] for k in ITERATE}
        for p, phi in _members(case, seed):
            e = _Exact(p, phi, None)
            e.begin()
            e.iterate(p["max_iter"])
            f = e.fields()
            for k in ITERATE:   # the cells' part of the staggered arrays, as run() hands them on
                out[k].append(f[k][: p["nz"], : p["ny"], : p["nx"]].reshape(-1))
        return {k: torch.cat(v) for k, v in out.items()}
    p, phi, logk = _pt_inputs(case, seed)
    if kind == "evolve":
        p, logk = A.adjoint_scope(p), _logk(p, seed)
    e = _Exact(p, phi, logk)
    for _ in range(case.get("steps", 1)):
        e.begin()
        if kind == "corr":
            e.correct(case["rounds"], case["iters"])
        else:
            e.iterate(case["iters"])
        e.end()
    # the gradient's 64-bit value is a transposed solve on whole arrays of its own: not given
    if kind == "evolve":
        return dict(phi=e.phi, grad=None)
    return {k: v for k, v in e.fields().items() if kind == "step" or k in HANDED_ON}
