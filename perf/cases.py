"""What the speed of this library is measured on: calls that a user's program
makes again and again, through ``paper_1806_06943_gb300.lb`` and
``paper_1806_06943_gb300.autograd``, over the range of lattices, number
formats and options that they are made with.

A pass of a time-stepping case advances a lattice (or a batch, or a 3-D
lattice) by the number of steps between two snapshots and reads the snapshot
(densities, velocities, observables) back, as the sweeps and the parity runs
of this repository do; the next pass goes on from there.  A pass of a gradient
case is one whole ``lb_grad``.  Snapshots of single-precision populations are
kept in single precision.

``exact`` restates the method (arXiv:1806.06943, Sec. II; its 3-D extension
with D3Q19 and the 5^3 mid-range stencil) in plain double-precision torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1806_06943_gb300 import autograd, lb

COUPLINGS = dict(G_AB=3.0, G1=-7.4, G2=6.4)
HI, LO, NOISE = 1.0, 0.03, 1e-3

# ---- the cases ----------------------------------------------------------------

def tau_d(ratio: float) -> float:
    """Relaxation time of the drops at viscosity ratio mu_d / mu_c, tau_c = 1."""
    return 0.5 + 0.5 * ratio


def listed() -> list[dict]:
    return [
        # The plain method's first run: one drop, 64 x 64, FP64, the
        # configuration a new handle has.  Few nodes: latency and launches.
        dict(name="droplet_64_fp64", kind="lattice", nx=64, ny=64, fields="drop", R=12.0, ratio=1.0, fp32=False,
             mode=-1, walls=0, wall_mode=0, g=0.0, shift=False, steps=500),
        # Films of the disjoining-pressure scan: a batch of 128 x 5 strips in
        # FP64 with the pressure tensor read at the end; the smallest lattices.
        dict(name="films_128x5_fp64", kind="films", nx=128, ny=5, n=9, steps=400),
        # A wall-bounded channel of odd size in FP64 with neutral walls and a
        # body force, default configuration (the layered Poiseuille runs).
        dict(name="channel_333x97_fp64", kind="lattice", nx=333, ny=97, fields="emulsion", R=9.0, ratio=3.0,
             fp32=False, mode=-1, walls=1, wall_mode=0, g=1e-6, shift=False, steps=200),
        # The plain FP64 path on a large emulsion, one-pass steps, the FP64 leg
        # beside every FP32 figure.
        dict(name="emulsion_1024_fp64", kind="lattice", nx=1024, ny=1024, fields="emulsion", R=14.0, ratio=5.0,
             fp32=False, mode=2, walls=0, wall_mode=0, g=0.0, shift=False, steps=100),
        # Pressure-driven channel emulsion, non-wetting walls, FP32 in the
        # configuration a new handle has.
        dict(name="channel_1024x256_fp32", kind="lattice", nx=1024, ny=256, fields="emulsion", R=12.0, ratio=3.0,
             fp32=True, mode=-1, walls=1, wall_mode=1, g=1e-6, shift=False, steps=500),
        # The Laplace sweep: 24 periodic lattices of 128^2 to 384^2 in one
        # batch, FP32, TMA steps (the benchmark's own workload).
        dict(name="laplace_sweep_24_fp32", kind="batch", n=24, lo=128, hi=384, multiple=32, walls=0, g=0.0, mode=3,
             steps=400),
        # Emulsion rheology: 28 wall-bounded 220 x 220 channels in one batch,
        # FP32, TMA steps; sides that are no multiple of a tile.
        dict(name="rheology_28x220_fp32", kind="batch", n=28, lo=220, hi=220, multiple=1, walls=1, g=1e-5, mode=3,
             steps=400),
        # The large dense emulsion, 4096 x 4096, FP32, TMA steps: the largest.
        dict(name="emulsion_4096_fp32", kind="lattice", nx=4096, ny=4096, fields="emulsion", R=14.0, ratio=5.0,
             fp32=True, mode=3, walls=0, wall_mode=0, g=0.0, shift=False, steps=500),
        # Calibration gradient: relative viscosity of the 512 x 128 channel
        # emulsion with respect to the couplings and relaxation times, FP64.
        dict(name="grad_mu_r_512x128_fp64", kind="grad", nx=512, ny=128, R=12.0, ratio=1.0, fp32=False, walls=1,
             steps=200, every=50),
        # The same machinery with the FP32 forward sweep, for the Laplace
        # pressure jump of a drop, through torch.autograd.
        dict(name="grad_dp_144_fp32", kind="grad", nx=144, ny=144, R=24.0, ratio=3.0, fp32=True, walls=0, steps=300,
             every=60),
        # 3-D emulsion, 160^3, FP32.
        dict(name="emulsion3d_160_fp32", kind="lattice3", nx=160, ny=160, nz=160, R=8.0, ratio=5.0, fp32=True, g=0.0,
             steps=100),
        # 3-D drop in FP64 on a lattice that no tile divides.
        dict(name="droplet3d_61x66x70_fp64", kind="lattice3", nx=61, ny=66, nz=70, R=15.0, ratio=1.0, fp32=False,
             g=1e-6, steps=60),
    ]


def _logint(rng, lo, hi) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    kind = rng.choice(["lattice", "lattice", "lattice", "batch", "lattice3", "grad", "films"])
    ratio = rng.choice([1.0 / 3.0, 1.0, 3.0, 5.0, 10.0])
    if kind == "lattice":
        fp32 = rng.random() < 0.5
        nodes = _logint(rng, 64 * 64, 2048 * 2048 if fp32 else 1024 * 1024)
        aspect = math.exp(rng.uniform(-math.log(4.0), math.log(4.0)))
        nx = max(24, int(math.sqrt(nodes * aspect)))
        ny = max(24, nodes // nx)
        walls = int(rng.random() < 0.5)
        shift = not fp32 and rng.random() < 0.15
        budget = 2.0e8 if fp32 else 4.0e7          # node updates of a pass
        return dict(kind=kind, nx=nx, ny=ny, fields="emulsion", R=rng.uniform(8.0, 18.0), ratio=1.0 if shift else ratio,
                    fp32=fp32, mode=rng.choice([-1, 3, 3, 2] if fp32 else [-1, -1, 2]), walls=walls,
                    wall_mode=rng.choice([0, 1]), g=rng.choice([0.0, 1e-6]) if walls else 0.0, shift=shift,
                    steps=int(min(500, max(40, budget / (nx * ny)))))
    if kind == "batch":
        lo = rng.randint(96, 200)
        return dict(kind=kind, n=rng.randint(2, 28), lo=lo, hi=rng.randint(lo, 384), multiple=rng.choice([1, 1, 32]),
                    walls=int(rng.random() < 0.4), g=rng.choice([0.0, 1e-6]), mode=rng.choice([-1, 3, 3, 2]),
                    steps=rng.randint(60, 200))
    if kind == "lattice3":
        fp32 = rng.random() < 0.6
        hi = 128 if fp32 else 72
        nx, ny, nz = (_logint(rng, 32, hi) for _ in range(3))
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, R=rng.uniform(6.0, 9.0), ratio=ratio, fp32=fp32,
                    g=rng.choice([0.0, 1e-6]), steps=rng.randint(20, 60))
    if kind == "grad":
        nx, ny = _logint(rng, 48, 400), _logint(rng, 48, 160)
        return dict(kind=kind, nx=nx, ny=ny, R=rng.uniform(8.0, 14.0), ratio=rng.choice([1.0, 3.0]),
                    fp32=rng.random() < 0.5, walls=int(rng.random() < 0.5), steps=rng.randint(60, 160),
                    every=rng.randint(20, 60))
    return dict(kind=kind, nx=rng.randint(96, 200), ny=rng.randint(5, 12), n=rng.randint(2, 12),
                steps=rng.randint(100, 400))


# ---- inputs -------------------------------------------------------------------

def _noisy(mask: torch.Tensor, gen: torch.Generator) -> torch.Tensor:
    """Densities [2][...] of a mask of species A: majority 1, minority 0.03,
    uniform noise of 1e-3."""
    a = torch.where(mask, HI, LO).to(torch.float64)
    rho = torch.stack([a, HI + LO - a])
    return rho + NOISE * (2.0 * torch.rand(rho.shape, generator=gen, dtype=torch.float64, device=mask.device) - 1.0)


def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(seed)


def _drops(shape, R, gen, margin=0.0) -> torch.Tensor:
    """A drop (disk, sphere) in each cell of a regular grid, its radius and
    its centre drawn inside the cell: a dense polydisperse emulsion.  shape
    slowest axis first; `margin` nodes stay free of drops at both ends of the
    slowest axis (walls)."""
    d = torch.zeros(shape, dtype=torch.float64, device="cuda")
    cells, idx, size = [], [], []
    for a, n in enumerate(shape):
        m = margin if a == 0 else 0.0
        k = max(1, int((n - 2 * m) / (2.0 * R + 5.0)))
        h = (n - 2 * m) / k
        x = torch.arange(n, dtype=torch.float64, device="cuda") - m
        i = torch.clamp((x / h).long(), 0, k - 1)
        cells.append(k)
        idx.append(i)
        size.append((x, h))
    r = R * (0.75 + 0.25 * torch.rand(cells, generator=gen, dtype=torch.float64, device="cuda"))
    grid = torch.meshgrid(*idx, indexing="ij")
    rr = r[grid]
    for a, (x, h) in enumerate(size):
        slack = torch.clamp(0.5 * h - 1.5 - r, min=0.0)
        c = 0.5 * h + slack * (2.0 * torch.rand(cells, generator=gen, dtype=torch.float64, device="cuda") - 1.0)
        pos = [1] * len(shape)
        pos[a] = -1
        d += (x.reshape(pos) - (grid[a] * h + c[grid])) ** 2
    return d < rr * rr


def _disk(shape, R, gen) -> torch.Tensor:
    """One drop near the middle (its centre drawn within a node)."""
    off = torch.rand(len(shape), generator=gen, dtype=torch.float64, device="cuda").tolist()
    d = torch.zeros(shape, dtype=torch.float64, device="cuda")
    for a, n in enumerate(shape):
        pos = [1] * len(shape)
        pos[a] = -1
        d += (torch.arange(n, dtype=torch.float64, device="cuda").reshape(pos) - (n / 2 + off[a] - 0.5)) ** 2
    return d < R * R


def _fields(case, seed) -> torch.Tensor:
    gen = _gen(seed)
    k = case["kind"]
    if k == "lattice":
        shape = (case["ny"], case["nx"])
        m = _disk(shape, case["R"], gen) if case["fields"] == "drop" else _drops(shape, case["R"], gen,
                                                                                 3.0 if case["walls"] else 0.0)
    elif k == "lattice3":
        shape = (case["nz"], case["ny"], case["nx"])
        m = _drops(shape, case["R"], gen) if case["R"] < 10.0 else _disk(shape, case["R"], gen)
    else:
        shape = (case["ny"], case["nx"])
        m = _drops(shape, case["R"], gen, 3.0) if case["walls"] else _disk(shape, min(case["R"], min(shape) / 5), gen)
    return _noisy(m, gen)


def _batch_specs(case, seed) -> list[dict]:
    """Sides spread evenly over [lo, hi] (rounded to `multiple`), drop radius
    an eighth of the side (at most 45), viscosity ratios 1, 3, 10 in turn;
    with walls square channels full of drops."""
    specs = []
    for i in range(case["n"]):
        t = i / max(1, case["n"] - 1)
        s = int(round(case["lo"] + t * (case["hi"] - case["lo"])))
        s = max(96, s // case["multiple"] * case["multiple"])
        s2 = dict(nx=s, ny=s, tau=(tau_d((1.0, 3.0, 10.0)[i % 3]), 1.0), R=min(45.0, s / 8.0))
        if case["walls"]:
            s2.update(walls=1, wall_mode=1, wall_rho=(LO, HI), g=(case["g"], 0.0))
        specs.append(s2)
    return specs


def _batch_field(case, spec, gen) -> torch.Tensor:
    shape = (spec["ny"], spec["nx"])
    return _noisy(_drops(shape, 15.0, gen, 3.0) if case["walls"] else _disk(shape, spec["R"], gen), gen)


def _film_field(case, i, gen) -> torch.Tensor:
    """A film of B of width h between regions of A, flat interfaces normal to x."""
    h = 4 + 6 * i
    x = torch.arange(case["nx"], device="cuda").expand(case["ny"], case["nx"])
    return _noisy((x + 0.5 - case["nx"] / 2).abs() >= h / 2, gen)


def _lattice_args(case) -> dict:
    kw = dict(COUPLINGS, tau=(tau_d(case["ratio"]), 1.0), walls=case["walls"], wall_mode=case["wall_mode"],
              g=(case["g"], 0.0), precision=lb.LB_FP32 if case["fp32"] else lb.LB_FP64)
    if case["walls"] and case["wall_mode"] == lb.LB_WALL_FIXED:
        kw["wall_rho"] = (LO, HI)
    if case["shift"]:
        kw["forcing"] = lb.LB_FORCING_SHIFT
    return kw


def prepare(case, seed):
    k = case["kind"]
    s = dict(case=case)
    if k == "lattice":
        L = lb.Lattice(case["nx"], case["ny"], **_lattice_args(case))
        if case["mode"] >= 0:
            L.set_config(case["mode"], 8)
        rho = _fields(case, seed)
        torch.cuda.synchronize()
        L.set_fields_device(rho)
        L.set_probe(case["nx"] / 2, case["ny"] / 2, case["R"])
        L.synchronize()
        s["L"] = L
    elif k in ("batch", "films"):
        gen = _gen(seed)
        if k == "batch":
            specs = _batch_specs(case, seed)
            prec = lb.LB_FP32
        else:
            specs = [dict(nx=case["nx"], ny=case["ny"]) for _ in range(case["n"])]
            prec = lb.LB_FP64
        B = lb.Batch(specs, precision=prec, **COUPLINGS)
        if case.get("mode", 2) >= 0:
            B.set_config(case.get("mode", 2), 8)
        for i, sp in enumerate(specs):
            rho = _batch_field(case, sp, gen) if k == "batch" else _film_field(case, i, gen)
            B.set_fields(i, rho.cpu().numpy())
            if k == "batch":
                B.set_probe(i, sp["nx"] / 2, sp["ny"] / 2, sp["R"])
        B.synchronize()
        s["B"] = B
    elif k == "lattice3":
        L = lb.Lattice3(case["nx"], case["ny"], case["nz"], tau=(tau_d(case["ratio"]), 1.0),
                        g=(case["g"], 0.0, 0.0), precision=lb.LB_FP32 if case["fp32"] else lb.LB_FP64, **COUPLINGS)
        L.set_fields(_fields(case, seed).cpu().numpy())
        L.set_probe(case["nx"] / 2, case["ny"] / 2, case["nz"] / 2, case["R"])
        s["L"] = L
    else:
        s["rho"] = _fields(case, seed).cpu().numpy()
        s["theta"] = torch.tensor([COUPLINGS["G_AB"], COUPLINGS["G1"], COUPLINGS["G2"], tau_d(case["ratio"]), 1.0],
                                  dtype=torch.float64)
        s["spec"] = _grad_spec(case, s["rho"])
    return s


def _grad_spec(case, rho) -> dict:
    spec = dict(nx=case["nx"], ny=case["ny"], rho=rho, nsteps=case["steps"], ckpt_every=case["every"],
                precision=lb.LB_FP32 if case["fp32"] else lb.LB_FP64)
    if case["walls"]:
        spec.update(walls=1, wall_mode=lb.LB_WALL_FIXED, wall_rho=(LO, HI), g=(1e-6, 0.0), objective=lb.LB_OBJ_MU_R)
    else:
        spec.update(objective=lb.LB_OBJ_DP, probe=(case["nx"] / 2, case["ny"] / 2, _probe_R(case)))
    return spec


def _probe_R(case) -> float:
    return min(case["R"], min(case["nx"], case["ny"]) / 5)


# ---- the calls ----------------------------------------------------------------

def _snapshot(fields: dict, fp32: bool) -> dict:
    out = {k: fields[k] for k in ("rho", "ubar")}
    return {k: torch.from_numpy(v).float() for k, v in out.items()} if fp32 else out


def _values(obs: dict, fp32: bool) -> np.ndarray:
    return np.array([float(v) for v in obs.values()], dtype=np.float32 if fp32 else np.float64)


def run(state):
    case = state["case"]
    k = case["kind"]
    if k in ("lattice", "lattice3"):
        L = state["L"]
        L.step(case["steps"])
        return dict(_snapshot(L.fields(), case["fp32"]), obs=_values(L.observables(), case["fp32"]))
    if k == "batch":
        B = state["B"]
        B.step(case["steps"])
        got = [_snapshot(B.fields(i), True) for i in range(B.n)]
        return dict(rho=[g["rho"] for g in got], ubar=[g["ubar"] for g in got],
                    obs=np.stack([_values(o, True) for o in B.observables()]))
    if k == "films":
        B = state["B"]
        B.step(case["steps"])
        got = [_snapshot(B.fields(i), False) for i in range(B.n)]
        P = [B.pressure_tensor(i, field=True) for i in range(B.n)]
        return dict(rho=[g["rho"] for g in got], ubar=[g["ubar"] for g in got], sums=[p[0] for p in P],
                    P=[p[1] for p in P])
    theta = state["theta"].clone().requires_grad_(True)
    J = autograd.observable(theta, state["spec"])
    J.backward()
    return dict(J=J.detach(), dJ=theta.grad)


def work(case) -> dict:
    """Bytes: every step reads and writes each population once (a gradient
    step: the forward sweep twice, the adjoint populations once more), the
    snapshot is written once.  Flops: the sums of the equations as written,
    about 700 a node and step in 2-D, 2000 in 3-D, three times that for a
    gradient step."""
    k = case["kind"]
    if k == "batch":
        nodes = sum(s["nx"] * s["ny"] for s in _batch_specs(case, 0))
    elif k == "films":
        nodes = case["n"] * case["nx"] * case["ny"]
    else:
        nodes = case["nx"] * case["ny"] * case.get("nz", 1)
    size = 4 if case.get("fp32", k == "batch") else 8
    q, fl = (38, 2000) if k == "lattice3" else (18, 700)
    per = 2 * q * size
    if k == "grad":
        return {"bytes": float(nodes * case["steps"] * (2 * per + 2 * 18 * 8)), "flops": float(3 * fl * nodes * case["steps"])}
    return {"bytes": float(nodes * (case["steps"] * per + 5 * size)), "flops": float(fl * nodes * case["steps"])}


# ---- the method in plain torch, 64 bits ---------------------------------------

E9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
W9 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
OPP9 = [0, 3, 4, 1, 2, 7, 8, 5, 6]
P25 = {1: 4 / 63, 2: 4 / 135, 4: 1 / 180, 5: 2 / 945, 8: 1 / 15120}
E19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
       (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
W19 = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
Q125 = {1: 4 / 135, 2: 1 / 63, 3: 2 / 315, 4: 5 / 1512, 5: 1 / 945, 6: 1 / 1890, 8: 1 / 15120}


class Plain:
    """The time step on f [..., 2, Q, (nz,) ny, nx]; tau [..., 2, 1, ...] and
    the couplings may be tensors that need gradients."""

    def __init__(self, dim, tau, G_AB, G1, G2, g, walls=0, wall_mode=0, shift=False):
        self.dim, self.tau, self.G, self.g = dim, tau, (G_AB, G1, G2), g
        self.walls, self.wall_mode, self.shift = walls, wall_mode, shift
        self.E, self.w = (E9, W9) if dim == 2 else (E19, W19)
        self.short = [(e, w) for e, w in zip(self.E, self.w) if any(e)]
        P = P25 if dim == 2 else Q125
        r = range(-2, 3)
        pts = [(x, y) for x in r for y in r] if dim == 2 else [(x, y, z) for x in r for y in r for z in r]
        self.mid = [(e, P[sum(c * c for c in e)]) for e in pts if sum(c * c for c in e) in P]

    def pad(self, a):
        """Two ghost layers on each side of every axis."""
        for ax in range(self.dim):
            d = a.dim() - 1 - ax       # ax 0: x
            n = a.shape[d]
            lo, hi = a.narrow(d, 0, 2), a.narrow(d, n - 2, 2)
            if ax == 1 and self.walls:
                if self.wall_mode == 1:
                    fixed = torch.tensor([LO, HI], dtype=a.dtype, device=a.device).reshape(2, 1, 1)
                    below = above = fixed.expand(a.shape[:-3] + (2, 2, a.shape[-1]))
                else:
                    below, above = lo.flip(d), hi.flip(d)
                a = torch.cat([below, a, above], d)
            else:
                a = torch.cat([hi, a, lo], d)
        return a

    def at(self, padded, e):
        for ax, c in enumerate(e):
            d = padded.dim() - 1 - ax
            padded = padded.narrow(d, 2 + c, padded.shape[d] - 4)
        return padded

    def sums(self, padded, stencil):
        """sum_j w_j s(x + e_j) e_j, opposite vectors taken together."""
        out = [None] * self.dim
        for e, w in stencil:
            if e < tuple(-c for c in e):
                continue
            d = self.at(padded, e) - self.at(padded, tuple(-c for c in e))
            for a, c in enumerate(e):
                if c:
                    out[a] = (w * c) * d if out[a] is None else out[a].add(d, alpha=w * c)
        return out

    def state(self, f):
        """Densities, forces and half-force momenta."""
        ax = -(self.dim + 1)
        rho = f.sum(ax)
        padded = self.pad(rho)
        psi = 1.0 - torch.exp(-padded)
        gab, g1, g2 = self.G
        s1, s2 = self.sums(psi, self.short), self.sums(psi, self.mid)
        s3 = self.sums(padded.flip(-(self.dim + 1)), self.short)
        p0 = self.at(psi, (0,) * self.dim)
        F = [-p0 * (g1 * s1[a] + g2 * s2[a]) - gab * rho * s3[a] + rho * self.g[a] for a in range(self.dim)]
        j = []
        for a in range(self.dim):
            parts = [f.select(ax, i) * float(e[a]) for i, e in enumerate(self.E) if e[a]]
            j.append(sum(parts[1:], parts[0]))
        return rho, F, j

    def step(self, f):
        ax, dim = -(self.dim + 1), self.dim
        rho, F, j = self.state(f)
        m = [j[a] if self.shift else j[a] + 0.5 * F[a] for a in range(dim)]
        om = 1.0 / self.tau
        den = (om * rho).sum(ax, keepdim=True)
        u = [(om * m[a]).sum(ax, keepdim=True) / den for a in range(dim)]
        uu = sum(u[a] * u[a] for a in range(dim))
        new = []
        for i, (e, w) in enumerate(zip(self.E, self.w)):
            eu = sum(u[a] * float(e[a]) for a in range(dim))
            fi = f.select(ax, i)
            feq = (w * rho) * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * uu)
            if self.shift:
                v = [u[a] + self.tau * F[a] / rho for a in range(dim)]
                ev = sum(v[a] * float(e[a]) for a in range(dim))
                C = om * ((w * rho) * (1.0 + 3.0 * ev + 4.5 * ev * ev - 1.5 * sum(c * c for c in v)) - feq)
            else:
                C = sum((3.0 * (float(e[a]) - u[a]) + 9.0 * eu * float(e[a])) * F[a] for a in range(dim))
                C = (1.0 - 0.5 * om) * w * C
            new.append(fi - om * (fi - feq) + C)
        out = []
        for i, e in enumerate(self.E):     # pull: the value that arrives from x - e
            v = torch.roll(new[i], e, tuple(range(-1, -1 - dim, -1)))
            if self.walls and e[1]:
                row = 0 if e[1] > 0 else f.shape[-2] - 1
                back = new[OPP9[i]].narrow(-2, row, 1)
                n = f.shape[-2]
                v = torch.cat([back, v.narrow(-2, 1, n - 1)], -2) if e[1] > 0 else torch.cat([v.narrow(-2, 0, n - 1), back], -2)
            out.append(v)
        return torch.stack(out, ax)

    def start(self, rho):
        w = torch.tensor(self.w, dtype=torch.float64, device=rho.device).reshape((-1,) + (1,) * self.dim)
        return rho.unsqueeze(-(self.dim + 1)) * w

    def fields(self, f):
        rho, F, j = self.state(f)
        ax = -(self.dim + 1)
        rt = rho.sum(ax)
        ubar = torch.stack([(j[a] + 0.5 * F[a]).sum(ax) / rt for a in range(self.dim)], ax)
        return rho, ubar

    def pressure(self, f):
        """[kinetic, interaction][xx, yy, xy] (2-D)."""
        rho = f.sum(-3)
        padded = self.pad(rho)
        psi = 1.0 - torch.exp(-padded)
        gab, g1, g2 = self.G
        p0 = self.at(psi, (0, 0))
        out = []
        for a, b in ((0, 0), (1, 1), (0, 1)):
            out.append(sum(f.select(-3, i).sum(-3) * float(e[a] * e[b]) for i, e in enumerate(self.E)))
        for a, b in ((0, 0), (1, 1), (0, 1)):
            def second(p, st):
                return sum((w * e[a] * e[b]) * self.at(p, e) for e, w in st if e[a] * e[b])
            t = p0 * (g1 * second(psi, self.short) + g2 * second(psi, self.mid))
            t = t + gab * rho * second(padded.flip(-3), self.short)
            out.append(0.5 * t.sum(-3))
        return torch.stack(out, -3).unflatten(-3, (2, 3))


def _tau(values, dim) -> torch.Tensor:
    return torch.tensor(values, dtype=torch.float64, device="cuda").reshape((-1, 2) + (1,) * dim)


def _numpy(x) -> np.ndarray:
    return x.cpu().numpy()


def _exact_grad(case, seed):
    if case["nx"] * case["ny"] * case["steps"] > 2.0e7:
        return None
    rho = _fields(case, seed)
    theta = torch.tensor([COUPLINGS["G_AB"], COUPLINGS["G1"], COUPLINGS["G2"], tau_d(case["ratio"]), 1.0],
                         dtype=torch.float64, device="cuda", requires_grad=True)
    walls = case["walls"]
    g = (1e-6, 0.0) if walls else (0.0, 0.0)

    def method(th):
        return Plain(2, th[3:5].reshape(2, 1, 1), th[0], th[1], th[2], g, walls, 1)

    def some(f, th, n):
        M = method(th)
        for _ in range(n):
            f = M.step(f)
        return f

    f = method(theta).start(rho)
    left = case["steps"]
    while left > 0:
        n = min(left, 10)
        f = torch.utils.checkpoint.checkpoint(some, f, theta, n, use_reentrant=False)
        left -= n
    M = method(theta)
    r, ubar = M.fields(f)
    ny, nx = case["ny"], case["nx"]
    if walls:
        q0 = g[0] * (ny ** 3 + 0.5 * ny) / (12.0 * (theta[4] - 0.5) / 3.0)
        J = q0 / (ubar[0].sum() / nx)
    else:
        R = _probe_R(case)
        d = [torch.arange(n, dtype=torch.float64, device="cuda") - n / 2 for n in (nx, ny)]
        d = [torch.minimum(c.abs(), n - c.abs()) for c, n in zip(d, (nx, ny))]
        rr = (d[0].reshape(1, -1) ** 2 + d[1].reshape(-1, 1) ** 2).sqrt()
        psi = 1.0 - torch.exp(-r)
        p = ((r + 0.5 * (theta[1] + theta[2]) * psi * psi).sum(0) + theta[0] * r[0] * r[1]) / 3.0
        J = p[rr < 0.5 * R].mean() - p[rr > R + 6.0].mean()
    J.backward()
    return dict(J=J.detach().cpu(), dJ=theta.grad.cpu())


def exact(case, seed):
    k = case["kind"]
    if k == "grad":
        return _exact_grad(case, seed)
    c = COUPLINGS
    with torch.no_grad():
        if k in ("lattice", "lattice3"):
            dim = 2 if k == "lattice" else 3
            nodes = case["nx"] * case["ny"] * case.get("nz", 1)
            if nodes * case["steps"] * (1 if dim == 2 else 6) > 9.0e9:
                return None
            M = Plain(dim, _tau([tau_d(case["ratio"]), 1.0], dim)[0], c["G_AB"], c["G1"], c["G2"],
                      (case["g"],) + (0.0,) * (dim - 1), case.get("walls", 0), case.get("wall_mode", 0),
                      case.get("shift", False))
            f = M.start(_fields(case, seed))
            for _ in range(case["steps"]):
                f = M.step(f)
            rho, ubar = M.fields(f)
            return dict(rho=_numpy(rho), ubar=_numpy(ubar), obs=None)
        gen = _gen(seed)
        if k == "batch":
            specs = _batch_specs(case, seed)
            rhos = [_batch_field(case, s, gen) for s in specs]
        else:
            specs = [dict(nx=case["nx"], ny=case["ny"], tau=(1.0, 1.0)) for _ in range(case["n"])]
            rhos = [_film_field(case, i, gen) for i in range(case["n"])]
        sizes = sorted({s["nx"] for s in specs})
        if len(sizes) * case["steps"] > 5000:
            return None
        rho, ubar, P = [None] * len(specs), [None] * len(specs), [None] * len(specs)
        for n in sizes:                 # lattices of one size together
            ids = [i for i, s in enumerate(specs) if s["nx"] == n]
            M = Plain(2, _tau([specs[i]["tau"] for i in ids], 2), c["G_AB"], c["G1"], c["G2"],
                      (case.get("g", 0.0) if case.get("walls") else 0.0, 0.0), case.get("walls", 0), 1)
            f = M.start(torch.stack([rhos[i] for i in ids]))
            for _ in range(case["steps"]):
                f = M.step(f)
            r, u = M.fields(f)
            p = M.pressure(f) if k == "films" else None
            for q, i in enumerate(ids):
                rho[i], ubar[i] = _numpy(r[q]), _numpy(u[q])
                P[i] = _numpy(p[q]) if k == "films" else None
        if k == "films":
            return dict(rho=rho, ubar=ubar, sums=None, P=P)
        return dict(rho=rho, ubar=ubar, obs=None)
