"""Timed cases of the lattice Boltzmann library: what a user's program has it do.

A time-stepping case holds a `Lattice` (parameters and populations on the GPU) and one pass
advances it by `steps` time steps and takes the snapshot such a program takes: the macroscopic
fields (rho, u, T) on the device, and the Nusselt number where the program samples it. The
snapshot is kept in the precision of the form (FP64 fields of the FP64 form, FP32 of the FP32
form, FP16 of the 16-bit forms). Every pass goes on from the state the last one left.

The cells are those of `paper_1111_0905_gb300.config` (boiling cell at the paper's geometry,
single-phase convection cell, adjoint cell), with the relaxation times that hold over long runs,
at the sizes of its tests and its benchmark (32 to 512 nodes a side) and at ragged sizes between.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1111_0905_gb300 import config, lb
from paper_1111_0905_gb300.autograd import nusselt_objective

Q = 19
SNAPSHOT = {"f64": torch.float64, "f32": torch.float32, "fp16loc": torch.float16,
            "fp16dev": torch.float16, "bf16dev": torch.float16}


def _case(name, kind, prec, cell, nx, ny, nz, steps, nu_every=0, forcing="shift", psi="exp"):
    c = {"kind": kind, "prec": prec, "cell": cell, "nx": nx, "ny": ny, "nz": nz, "steps": steps,
         "nu_every": nu_every, "forcing": forcing, "psi": psi}
    return c if name is None else {"name": name, **c}


def listed():
    return [
        # the plain FP64 boiling cell of the parity runs: tiny launches, latency counts; the
        # whole updated state (populations) comes back
        _case("fp64_boiling_32", "restart", "f64", "boiling", 32, 32, 32, 10),
        # a monitoring loop on a small cell: a few steps, then the Nusselt number on the host
        _case("fp32_monitor_64", "monitor", "f32", "boiling", 64, 64, 64, 5),
        # a ragged cell: no side a multiple of a tile or a warp
        _case("fp32_ragged_150x93x77", "steps", "f32", "boiling", 150, 93, 77, 20),
        # a comparison run of a scheme variant (Guo forcing, van der Waals psi)
        _case("fp32_variant_128", "steps", "f32", "boiling", 128, 128, 128, 20, forcing="guo", psi="vdw"),
        # single-phase convection with the time-averaged Nusselt number sampled every 5 steps
        _case("fp32_single_phase_nu_128", "monitor", "f32", "single", 128, 128, 128, 20, nu_every=5),
        # the same cell in FP64: the reference run that the other forms are compared with
        _case("fp64_single_phase_128", "steps", "f64", "single", 128, 128, 128, 10),
        # statistics of a run: profiles, T-rho histogram, heat-flux pdf, structure functions
        _case("fp64_statistics_96", "statistics", "f64", "single", 96, 96, 96, 2),
        # gradient of the time-averaged Nusselt number, checkpoints every 50 steps, forward and backward
        _case("adjoint_fp64_64", "adjoint", "f64", "boiling", 64, 64, 64, 100),
        # 16-bit storage on the boiling cell: deviations, and local references
        _case("fp16dev_boiling_256", "steps", "fp16dev", "boiling", 256, 256, 256, 10),
        _case("fp16loc_boiling_256", "steps", "fp16loc", "boiling", 256, 256, 256, 10),
        # production runs: FP32 at 256^3 and at the paper's 512^3
        _case("fp32_boiling_256", "steps", "f32", "boiling", 256, 256, 256, 20),
        _case("fp32_boiling_512", "steps", "f32", "boiling", 512, 512, 512, 10),
    ]


def _side(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["steps", "steps", "steps", "monitor", "restart", "statistics", "adjoint"])
    if kind == "adjoint":
        n = [_side(rng, 16, 80) for _ in range(3)]
        return _case(None, kind, "f64", "boiling", *n, rng.randint(20, 100))
    if kind == "statistics":
        n = [_side(rng, 24, 128) for _ in range(3)]
        return _case(None, kind, "f64", rng.choice(["boiling", "single"]), *n, rng.randint(1, 4))
    prec = rng.choice(["f32", "f32", "f64", "fp16loc", "fp16dev", "bf16dev"])
    top = {"f64": 160, "f32": 400}.get(prec, 320)
    if kind == "restart":
        prec, top = rng.choice(["f64", "f32"]), 128
    # a multiple of 32 at times, any size at others
    n = [max(16, s // 32 * 32) if rng.random() < 0.4 else s for s in (_side(rng, 16, top) for _ in range(3))]
    scheme = {}
    if kind == "steps" and prec != "bf16dev" and rng.random() < 0.2:
        scheme = {"forcing": rng.choice(["shift", "guo"]), "psi": "vdw"}
    cell = rng.choice(["boiling", "boiling", "single"]) if not scheme else "boiling"
    steps = rng.randint(2, 5) if prec == "bf16dev" else rng.randint(2, 20)
    return _case(None, kind, prec, cell, *n, steps,
                 nu_every=rng.choice([0, 1, 5, 10]) if kind == "monitor" else 0, **scheme)


# the van der Waals psi's liquid-gas mixture of the tests (a = 5/42, b = 2/21: rho_c = 3.5)
VDW_RHO = 3.5


def _params(case):
    cell = config.paper_scale_cell if case["cell"] == "boiling" else config.single_phase_cell
    w = cell(case["nz"], precision=lb.PRECISIONS[case["prec"]])
    p = w.params
    p.nx, p.ny, p.nz, p.nu_every = case["nx"], case["ny"], case["nz"], case["nu_every"]
    p.forcing = lb.LB_FORCE_GUO if case["forcing"] == "guo" else lb.LB_FORCE_SHIFT
    rho_mean = w.rho_mean
    if case["psi"] == "vdw":
        p.psi_kind, rho_mean = lb.LB_PSI_VDW, VDW_RHO
        # conductivity at that density: kappa/(tau_kappa - 1/2) inside the g equilibrium's window
        p.kappa *= VDW_RHO / w.rho_mean
    return p, rho_mean


def _waves(p, gen, device):
    """Sum of six plane waves of random direction and phase, about 40 nodes long (periodic in x
    and y), scaled to a largest magnitude of about 1: the blobs of a separating mixture, or the
    sound and plumes of a single phase."""
    pick = torch.rand((6, 4), generator=gen, device=device, dtype=torch.float64).cpu().tolist()
    axes = [torch.arange(n, device=device, dtype=torch.float64) / n for n in (p.nx, p.ny, p.nz)]
    s = torch.zeros((p.nz, p.ny, p.nx), device=device, dtype=torch.float64)
    for a, b, c, phase in pick:
        kx, ky, kz = (round((2 * r - 1) * max(1.0, n / 40.0)) for r, n in ((a, p.nx), (b, p.ny), (c, p.nz)))
        arg = (kx * axes[0])[None, None, :] + (ky * axes[1])[None, :, None] + ((kz or 1) * axes[2] + phase)[:, None, None]
        s += torch.cos(2.0 * math.pi * arg) / 3.0
    return s


def _fields(case, seed, device="cuda"):
    """Initial rho and T of a cell with motion in it: density waves of 20 % about the mean
    (boiling: liquid and vapour blobs) or of 2 % (single-phase), 1 % noise on the density
    (boiling) or the temperature (single-phase), T linear between the walls."""
    p, rho_mean = _params(case)
    gen = torch.Generator(device=device).manual_seed(seed)
    xi = torch.rand((p.nz, p.ny, p.nx), generator=gen, device=device, dtype=torch.float64) * 2.0 - 1.0
    waves = _waves(p, gen, device)
    z = (torch.arange(p.nz, device=device, dtype=torch.float64) + 0.5) / p.nz
    T = (p.T_d + (p.T_u - p.T_d) * z)[:, None, None]
    if case["cell"] == "boiling":
        return rho_mean * (1.0 + 0.2 * waves + 0.01 * xi), T.expand(p.nz, p.ny, p.nx).contiguous()
    return rho_mean * (1.0 + 0.02 * waves), T * (1.0 + 0.01 * xi)


def prepare(case, seed):
    p, _ = _params(case)
    rho, T = _fields(case, seed)
    state = {"case": case, "params": p}
    if case["kind"] == "adjoint":
        state["rho"] = rho
        state["leaves"] = [torch.tensor(v, dtype=torch.float64, requires_grad=True) for v in (p.T_d, p.T_u, p.G)]
        state["T0"] = T.requires_grad_(True)
        return state
    state["lattice"] = lb.Lattice(p, rho, T)
    return state


def _snapshot(lat, prec):
    rho, u, T = lat.moments(device=True)
    t = SNAPSHOT[prec]
    return {"rho": rho.to(t), "ux": u[0].to(t), "uy": u[1].to(t), "uz": u[2].to(t), "T": T.to(t)}


# ranges of the statistics: bins over the cells' temperatures, densities and heat fluxes
T_RANGE, RHO_RANGE, Q_RANGE, BINS = (0.30, 0.37), (1.0, 3.0), (-0.02, 0.02), 64


def _statistics_planes(case):
    nz = case["nz"]
    return nz // 8, nz - nz // 8, min(32, case["nx"] - 1, case["ny"] - 1)


def run(state):
    case = state["case"]
    if case["kind"] == "adjoint":
        leaves = [*state["leaves"], state["T0"]]
        for x in leaves:
            x.grad = None
        J = nusselt_objective(*leaves, state["rho"], state["params"], case["steps"])
        J.backward()
        return {"J": J.detach(), **{k: x.grad for k, x in zip(("T_d", "T_u", "G", "T0"), leaves)}}
    lat = state["lattice"]
    lat.step(case["steps"])
    if case["kind"] == "restart":
        f, g = lat.populations(device=True)
        return {"f": f.to(SNAPSHOT[case["prec"]]), "g": g.to(SNAPSHOT[case["prec"]])}
    if case["kind"] == "monitor":
        nu, nu_z, avg = lat.nusselt()
        out = _snapshot(lat, case["prec"])
        out["nu"] = nu
        out["nu_z"] = nu_z if case["prec"] == "f64" else nu_z.astype(np.float32 if case["prec"] == "f32" else np.float16)
        if case["nu_every"] and case["steps"] >= case["nu_every"]:
            out["nu_avg"] = avg
        return out
    if case["kind"] == "statistics":
        lo, hi, rmax = _statistics_planes(case)
        rho_z, T_z, pdivu_z = lat.profiles()
        hist = lat.histogram_T_rho(lo, hi, BINS, T_RANGE, BINS, RHO_RANGE)
        counts, moments = lat.heat_flux_pdf(lo, hi, BINS, Q_RANGE)
        return {"rho_z": rho_z, "T_z": T_z, "pdivu_z": pdivu_z, "hist": hist.astype(np.int64),
                "q_counts": counts.astype(np.int64), "q_moments": np.array(moments),
                **lat.structure_functions(rmax, lo, hi)}
    return _snapshot(lat, case["prec"])


STORED = {"f64": (8, 19), "f32": (4, 19), "fp16loc": (2, 21), "fp16dev": (2, 19), "bf16dev": (2, 19)}
OUT_BYTES = {"f64": 8, "f32": 4, "fp16loc": 2, "fp16dev": 2, "bf16dev": 2}
STEP_FLOPS = 400      # per node and step: moments, force, velocities, divergence, two collisions


def work(case):
    """A step reads and writes both distributions once; a snapshot reads them once and writes its
    fields; the adjoint steps forward and sweeps back over as many values; statistics read the state once."""
    n = case["nx"] * case["ny"] * case["nz"]
    size, slots = STORED[case["prec"]]
    lattices = 2 * slots * size * n            # f and g, once
    steps = case["steps"]
    out = OUT_BYTES[case["prec"]] * n
    kind = case["kind"]
    if kind == "adjoint":
        return {"bytes": 4 * lattices * steps + 3 * out, "flops": 3 * STEP_FLOPS * n * steps}
    if kind == "restart":
        end = lattices + 2 * Q * out
    elif kind == "statistics":
        end = lattices
    else:
        end = lattices + 5 * out
    return {"bytes": 2 * lattices * steps + end, "flops": STEP_FLOPS * n * steps + 100 * n}


# ---- the same passes in plain torch, float64 -------------------------------------------------
C = ((0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
     (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
     (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1))
C2 = [a * a + b * b + c * c for a, b, c in C]
W = [1 / 3 if k == 0 else 1 / 18 if k == 1 else 1 / 36 for k in C2]
OPP = [C.index((-a, -b, -c)) for a, b, c in C]


def _along(c, v):
    s = None
    for k, x in zip(c, v):
        if k:
            s = (k * x) if s is None else s + k * x
    return s


def _shift(q, dx, dy, dz, sign=1.0):
    """q(x + d): periodic in x and y, the value of the mirrored plane times sign beyond a z wall."""
    q = torch.roll(q, (-dy, -dx), (1, 2)) if dx or dy else q
    if dz == 1:
        return torch.cat([q[1:], sign * q[-1:]])
    if dz == -1:
        return torch.cat([sign * q[:1], q[:-1]])
    return q


class _Exact:
    def __init__(self, p, rho, T):
        self.p = p
        self.lam = p.kappa / (p.c_v * (p.tau_kappa - 0.5))
        zero = [torch.zeros_like(rho)] * 3
        self.f = [self.feq(l, rho, zero, T) for l in range(Q)]
        self.g = [self.geq(l, rho, zero, T) for l in range(Q)]

    def feq(self, l, rho, v, T):
        vv = v[0] * v[0] + v[1] * v[1] + v[2] * v[2]
        e = 1.0 - 1.5 * vv + 4.5 * (C2[l] - 1) * (T - 1 / 3)
        if l:
            cv = _along(C[l], v)
            e = e + 3.0 * cv + 4.5 * cv * cv
        return W[l] * rho * e

    def geq(self, l, rho, u, T):
        uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2]
        e = 1.0 - 1.5 * uu
        if l:
            cu = _along(C[l], u)
            e = e + 3.0 * cu + 4.5 * cu * cu
        return W[l] * (rho * T * e + 4.5 * (C2[l] - 1) * (self.lam * T - rho * T / 3))

    def macros(self):
        p = self.p
        rho = sum(self.f[1:], self.f[0])
        T = sum(self.g[1:], self.g[0]) / rho
        j = [sum(C[l][a] * self.f[l] for l in range(Q) if C[l][a]) for a in range(3)]
        if p.psi_kind == lb.LB_PSI_VDW:
            psi = rho * torch.sqrt(2.0 / -p.G * (p.vdw_a - p.vdw_b * p.vdw_T / (1.0 - p.vdw_b * rho)))
        else:
            psi = torch.exp(-1.0 / rho)
        F = [torch.zeros_like(rho) for _ in range(3)]
        for l in range(1, Q):
            nb = _shift(psi, *C[l]) * (1 / 6 if C2[l] == 1 else 1 / 12)
            for a in range(3):
                if C[l][a]:
                    F[a] = F[a] + C[l][a] * nb
        F = [-p.G * psi * x for x in F]
        F[2] = F[2] + rho * p.g_z
        u = [(j[a] + 0.5 * F[a]) / rho for a in range(3)]
        v = u if p.forcing == lb.LB_FORCE_GUO else [(j[a] + p.tau_nu * F[a]) / rho for a in range(3)]
        return rho, T, F, u, v

    def divergence(self, u):
        e = ((1, 0, 0), (0, 1, 0), (0, 0, 1))
        return sum(0.5 * (_shift(u[a], *e[a], sign=-1.0) - _shift(u[a], *[-k for k in e[a]], sign=-1.0)) for a in range(3))

    def step(self):
        p, lam = self.p, self.lam
        rho, T, F, u, v = self.macros()
        S = -rho * T * self.divergence(u) / p.c_v
        uF = sum(u[a] * F[a] for a in range(3))
        fs, gs = [], []
        for l in range(Q):
            x = self.f[l] - (self.f[l] - self.feq(l, rho, v, T)) / p.tau_nu
            if p.forcing == lb.LB_FORCE_GUO:
                s = -3.0 * uF
                if l:
                    cF = _along(C[l], F)
                    s = s + 3.0 * cF + 9.0 * _along(C[l], u) * cF
                x = x + (1.0 - 0.5 / p.tau_nu) * W[l] * s
            fs.append(x)
            gs.append(self.g[l] - (self.g[l] - self.geq(l, rho, u, T)) / p.tau_kappa + W[l] * S)
            self.f[l] = self.g[l] = None
        for l in range(Q):
            cx, cy, cz = C[l]
            sf, sg = (torch.roll(x[l], (cy, cx), (1, 2)) for x in (fs, gs))
            if cz:
                w, Tw = (0, p.T_d) if cz > 0 else (-1, p.T_u)
                even = W[l] * (rho[w] * Tw + 4.5 * (lam * Tw - rho[w] * Tw / 3) * (C2[l] - 1))
                bf, bg = fs[OPP[l]][w][None], (2.0 * even - gs[OPP[l]][w])[None]
                sf = torch.cat([bf, sf[:-1]]) if cz > 0 else torch.cat([sf[1:], bf])
                sg = torch.cat([bg, sg[:-1]]) if cz > 0 else torch.cat([sg[1:], bg])
            self.f[l], self.g[l] = sf, sg

    def energy(self, rho, T):
        p = self.p
        if p.psi_kind == lb.LB_PSI_VDW:
            return p.c_v * T - p.vdw_T * torch.log(1.0 - p.vdw_b * rho) - p.vdw_a * rho
        return p.c_v * T + 0.25 * p.G * torch.exp(-2.0 / rho)

    def nusselt(self):
        p = self.p
        rho, T, _, u, _ = self.macros()
        Tz = T.mean((1, 2))
        up = torch.cat([Tz[1:], 2 * p.T_u - Tz[-1:]])
        down = torch.cat([2 * p.T_d - Tz[:1], Tz[:-1]])
        flux = (rho * self.energy(rho, T) * u[2]).mean((1, 2)) - p.kappa * 0.5 * (up - down)
        nu_z = flux / (p.kappa * (p.T_d - p.T_u) / p.nz)
        return float(nu_z.mean()), nu_z.cpu().numpy()


def exact(case, seed):
    nodes = case["nx"] * case["ny"] * case["nz"]
    # about 0.3 s a step at 256^3; the adjoint has no such value (its gradient is pinned by its type)
    if case["kind"] == "adjoint" or nodes * case["steps"] > 20 * 257 ** 3:
        return None
    p, _ = _params(case)
    x = _Exact(p, *_fields(case, seed))
    samples = []
    for n in range(1, case["steps"] + 1):
        x.step()
        if case["nu_every"] and n % case["nu_every"] == 0:
            samples.append(x.nusselt()[0])
    if case["kind"] == "restart":
        return {"f": torch.stack(x.f), "g": torch.stack(x.g)}
    rho, T, _, u, _ = x.macros()
    if case["kind"] == "statistics":
        lo, hi, rmax = _statistics_planes(case)
        P = rho * T + 0.5 * p.G * torch.exp(-2.0 / rho)
        q = (rho * x.energy(rho, T) * u[2])[lo:hi]
        out = {"rho_z": rho.mean((1, 2)).cpu().numpy(), "T_z": T.mean((1, 2)).cpu().numpy(),
               "pdivu_z": (P * x.divergence(u)).mean((1, 2)).cpu().numpy(), "hist": None, "q_counts": None,
               "q_moments": np.array([q.numel(), float(q.mean()), float(((q - q.mean()) ** 2).mean())])}
        for name, v in (("uz", u[2][lo:hi]), ("T", T[lo:hi])):
            d = [[torch.roll(v, -r, a) - v for a in (2, 1)] for r in range(1, rmax + 1)]
            for k in (2, 4):
                out[f"S{k}_{name}"] = np.array([float(sum((e ** k).mean() for e in pair) / 2) for pair in d])
        return out
    out = {"rho": rho, "ux": u[0], "uy": u[1], "uz": u[2], "T": T}
    if case["kind"] == "monitor":
        out["nu"], out["nu_z"] = x.nusselt()
        if samples:
            out["nu_avg"] = sum(samples) / len(samples)
    return out
