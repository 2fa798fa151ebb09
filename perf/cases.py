"""Timed cases of the cRKFR step: the work that a program has this library do.

A program holds a solver (or a batch of them) for its mesh, puts a state in,
advances it to its next snapshot and takes the snapshot out; that is one pass.
The flows are the library's synthetic workloads (1D density wave, 2D shear
layer, GLM-MHD vortex, 3D Taylor-Green vortex, uneven batch of 2D waves) with
their degrees, fluxes, schemes and CFL numbers, phases and noise drawn from the
seed.  A snapshot has the precision of its form: the FP64 form's is the FP64
state itself; the FP32 pair-flux form's, whose increments are single precision,
is handed on in single precision, as a program writes it to disk.

`exact` advances the same state in FP64 with plain torch operations written
from the scheme's equations, without this library.
"""
import math

import numpy as np
import torch

from paper_2604_02125_gb300 import crkfr, work as counted

DEV = "cuda"
CFL = {1: 0.1, 2: 0.1, 3: 0.1, 4: 0.07, 5: 0.05}


def _case(name, flow, N, cells, prec, steps, vol="ec", scheme="crkfr", limiter=False, entry="solver"):
    nx, ny, nz = (list(cells) + [1, 1])[:3]
    c = {"name": name, "flow": flow, "N": N, "nx": nx, "ny": ny, "nz": nz, "prec": prec, "steps": steps,
         "vol": vol, "scheme": scheme, "limiter": limiter, "entry": entry}
    if name is None:
        del c["name"]
    return c


def listed():
    return [
        # the convergence study's mesh: a few hundred nodes, all latency
        _case("wave_64_N3_fp64", "wave", 3, [64], "fp64", 50),
        # one step without allocation inside another program's loop
        _case("noalloc_shear_64x64_N3_fp32", "shear", 3, [64, 64], "fp32", 1, entry="noalloc"),
        # the paper's Kelvin-Helmholtz run: KEP flux, subcell limiter with alpha_max = 0.008
        _case("kh_limited_64x64_N3_fp32", "shear", 3, [64, 64], "fp32", 32, vol="kep", limiter=True),
        # the headline workload in its fast and its plain form
        _case("shear_256x256_N3_fp32", "shear", 3, [256, 256], "fp32", 16),
        _case("shear_256x256_N3_fp64", "shear", 3, [256, 256], "fp64", 4),
        # high degree on a ragged mesh (partly filled last tile)
        _case("shear_97x61_N5_fp32", "shear", 5, [97, 61], "fp32", 16),
        # the multi-stage scheme that the single-stage one is compared with
        _case("rkfr_shear_256x256_N3_fp32", "shear", 3, [256, 256], "fp32", 8, scheme="rkfr"),
        # GLM-MHD with its non-conservative terms, both forms
        _case("vortex_128x128_N4_fp32", "vortex", 4, [128, 128], "fp32", 8),
        _case("vortex_61x45_N3_fp64", "vortex", 3, [61, 45], "fp64", 4),
        # 3D, the largest state, and the plain form on an odd box
        _case("tgv_64x64x64_N3_fp32", "tgv", 3, [64, 64, 64], "fp32", 4),
        _case("tgv_22x20x19_N3_fp64", "tgv", 3, [22, 20, 19], "fp64", 4),
        # many independent solves of uneven size and degree advanced together
        _case("batch_64_fp32", "batch", 0, [64], "fp32", 8, entry="batch"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    # counted FP32 / FP64 operations of a pass, at most those of the largest listed cases
    room = {"fp32": 1.0e11, "fp64": 4.5e9}
    while True:
        prec = rng.choice(["fp32", "fp32", "fp64"])
        kind = rng.choice(["wave", "shear", "shear", "limited", "rkfr", "vortex", "vortex", "tgv", "noalloc", "batch"])
        N = rng.randint(1, 5)
        vol = rng.choice(["ec", "ec", "kep", "central"])
        steps = _log_int(rng, 1, 32)
        if kind == "wave":
            c = _case(None, "wave", N, [_log_int(rng, 16, 65536)], prec, steps, vol)
        elif kind == "shear":
            c = _case(None, "shear", N, [_log_int(rng, 16, 256), _log_int(rng, 16, 256)], prec, steps, vol)
        elif kind == "limited":
            c = _case(None, "shear", N, [_log_int(rng, 32, 256), _log_int(rng, 32, 256)], prec, steps,
                      rng.choice(["ec", "kep"]), limiter=True)
        elif kind == "rkfr":
            c = _case(None, "shear", N, [_log_int(rng, 32, 256), _log_int(rng, 32, 256)], prec, min(steps, 8), vol,
                      scheme="rkfr")
        elif kind == "vortex":
            c = _case(None, "vortex", N, [_log_int(rng, 16, 128), _log_int(rng, 16, 128)], prec, steps,
                      rng.choice(["ec", "ec", "central"]))
        elif kind == "tgv":
            c = _case(None, "tgv", N, [_log_int(rng, 8, 64) for _ in range(3)], prec, min(steps, 8), vol)
        elif kind == "noalloc":
            c = _case(None, "shear", min(N, 4), [rng.randint(12, 64), rng.randint(12, 40)], prec, 1, vol,
                      entry="noalloc")
        else:
            c = _case(None, "batch", 0, [rng.randint(2, 64)], "fp32", min(steps, 8), vol, entry="batch")
        if work(c)["flops"] <= room[c["prec"]]:
            return c


# ---------------------------------------------------------------------------
# meshes and initial states, on the GPU
# ---------------------------------------------------------------------------
def _gll(N):
    """GLL nodes and weights on [0,1] and the differentiation matrix D_pq = l_q'(xi_p)."""
    P = np.polynomial.legendre.Legendre.basis(N)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    for _ in range(3):   # polish the inner roots of P_N'
        x[1:-1] -= P.deriv()(x[1:-1]) / P.deriv(2)(x[1:-1])
    w = 1.0 / (N * (N + 1) * P(x) ** 2)
    xi = 0.5 * (x + 1.0)
    lam = np.array([1.0 / np.prod([xi[j] - xi[k] for k in range(N + 1) if k != j]) for j in range(N + 1)])
    D = np.zeros((N + 1, N + 1))
    for i in range(N + 1):
        for j in range(N + 1):
            if i != j:
                D[i, j] = lam[j] / lam[i] / (xi[i] - xi[j])
        D[i, i] = -D[i].sum()
    return xi, w, D


def _mesh(eq, dim, N, cells, lo, hi, gamma, vol):
    pad = [1] * (3 - dim)
    return {"eq": eq, "dim": dim, "N": N, "cells": list(cells) + pad, "lo": [lo] * dim + [0.0] * (3 - dim),
            "hi": [hi] * dim + [1.0] * (3 - dim), "gamma": gamma, "cfl": CFL[N], "c_h": 0.0, "vol": vol,
            "surf": "rusanov"}


def _coords(mesh):
    """Node coordinates, shaped like one variable: [elements, last direction first][nodes, likewise]."""
    dim, N = mesh["dim"], mesh["N"]
    xi = torch.tensor(_gll(N)[0], dtype=torch.float64, device=DEV)
    out = []
    for d in range(dim):
        n = mesh["cells"][d]
        dx = (mesh["hi"][d] - mesh["lo"][d]) / n
        x = mesh["lo"][d] + (torch.arange(n, dtype=torch.float64, device=DEV)[:, None] + xi[None, :]) * dx
        shape = [1] * (2 * dim)
        shape[dim - 1 - d], shape[2 * dim - 1 - d] = n, N + 1
        out.append(x.reshape(shape))
    return torch.broadcast_tensors(*out)


def _euler(gamma, rho, vel, p):
    E = p / (gamma - 1.0) + 0.5 * rho * sum(v * v for v in vel)
    return torch.stack([rho] + [rho * v for v in vel] + [E])


def _noise(g, like):
    return 1e-3 * torch.randn(like.shape, generator=g, dtype=torch.float64, device=DEV)


def _initial(case, seed):
    """[(mesh, state)] of a case, one entry per solve; state [var][elements][nodes]."""
    g = torch.Generator(device=DEV)
    g.manual_seed(1 + seed)
    r = np.random.default_rng(seed)
    N, vol, pi = case["N"], case["vol"], math.pi
    cells = [case["nx"], case["ny"], case["nz"]]
    if case["flow"] == "batch":
        out = []
        sizes = np.random.default_rng(case["nx"])   # the sizes belong to the case, the states to the seed
        for _ in range(case["nx"]):
            side, deg = int(sizes.integers(16, 129)), int(sizes.integers(2, 6))
            mesh = _mesh("euler", 2, deg, [side, side], -1.0, 1.0, 1.4, vol)
            x, y = _coords(mesh)
            a, b = r.uniform(0.1, 0.5), r.uniform(0.01, 0.1)
            kx, ky = r.integers(1, 3, size=2)
            rho = 1.0 + a * torch.sin(pi * (int(kx) * x + int(ky) * y))
            out.append((mesh, _euler(1.4, rho, [0.5 + b * torch.sin(pi * y), b * torch.sin(pi * x)],
                                     torch.ones_like(rho))))
        return out
    if case["flow"] == "wave":
        mesh = _mesh("euler", 1, N, cells[:1], 0.0, 2.0, 1.4, vol)
        (x,) = _coords(mesh)
        rho = 1.0 + r.uniform(0.4, 0.5) * torch.sin(pi * x + r.uniform(0, 2 * pi))
        return [(mesh, _euler(1.4, rho, [torch.ones_like(rho)], torch.ones_like(rho)))]
    if case["flow"] == "shear":
        mesh = _mesh("euler", 2, N, cells[:2], -1.0, 1.0, 1.4, vol)
        x, y = _coords(mesh)
        B = torch.tanh(15.0 * y + 7.5) - torch.tanh(15.0 * y - 7.5)
        vy = 0.1 * torch.sin(pi * x + r.uniform(0, 2 * pi)) + _noise(g, x)
        u = _euler(1.4, 0.5 + 0.75 * B, [0.5 * (B - 1.0), vy], torch.ones_like(B))
        if case["limiter"]:
            mesh = dict(mesh, limiter=True, alpha_max=0.008)
        return [(mesh, u)]
    if case["flow"] == "vortex":
        gam = 5.0 / 3.0
        mesh = _mesh("glm_mhd", 2, N, cells[:2], 0.0, 1.0, gam, vol)
        x, y = _coords(mesh)
        x, y = 2 * pi * (x + r.uniform()), 2 * pi * (y + r.uniform())
        rho = torch.full_like(x, 25.0 / (36.0 * pi))
        p = torch.full_like(x, 5.0 / (12.0 * pi))
        v = [-torch.sin(y) + _noise(g, x), torch.sin(x) + _noise(g, x), torch.zeros_like(x)]
        s = 1.0 / math.sqrt(4.0 * pi)
        Bf = [-s * torch.sin(y), s * torch.sin(2 * x), torch.zeros_like(x)]
        B2 = Bf[0] ** 2 + Bf[1] ** 2
        mesh["c_h"] = float(torch.maximum(v[0].abs().max(), v[1].abs().max()) + ((gam * p + B2) / rho).max().sqrt())
        E = p / (gam - 1.0) + 0.5 * rho * (v[0] ** 2 + v[1] ** 2) + 0.5 * B2
        return [(mesh, torch.stack([rho, rho * v[0], rho * v[1], rho * v[2], E] + Bf + [torch.zeros_like(x)]))]
    mesh = _mesh("euler", 3, N, cells, 0.0, 2.0 * pi, 1.4, vol)
    x, y, z = _coords(mesh)
    x, y, z = (q + r.uniform(0, 2 * pi) for q in (x, y, z))
    vel = [torch.sin(x) * torch.cos(y) * torch.cos(z), -torch.cos(x) * torch.sin(y) * torch.cos(z),
           torch.zeros_like(x)]
    p = 1.0 / (1.4 * 0.01) + (torch.cos(2 * x) + torch.cos(2 * y)) * (torch.cos(2 * z) + 2.0) / 16.0
    return [(mesh, _euler(1.4, torch.ones_like(x), vel, p))]


# ---------------------------------------------------------------------------
# the pass through the library
# ---------------------------------------------------------------------------
def prepare(case, seed):
    solves = _initial(case, seed)
    meshes = [dict(m, scheme=case["scheme"]) for m, _ in solves]
    u0 = [u.reshape(u.shape[0], -1).contiguous() for _, u in solves]
    state = {"case": case, "meshes": meshes, "u0": u0, "out": [torch.empty_like(u) for u in u0]}
    if case["prec"] == "fp32":
        state["snapshot"] = [torch.empty(u.shape, dtype=torch.float32, device=DEV) for u in u0]
    if case["entry"] == "noalloc":
        state["dt"] = torch.zeros(1, dtype=torch.float64, device=DEV)
    else:
        state["solver"] = crkfr.Solver(meshes if case["entry"] == "batch" else meshes[0], prec=case["prec"])
    return state


def run(state):
    case = state["case"]
    if case["entry"] == "noalloc":
        crkfr.step_noalloc(state["meshes"][0], state["u0"][0], state["out"][0], state["dt"], prec=case["prec"])
    else:
        s = state["solver"]
        for k, u in enumerate(state["u0"]):
            s.set_state(u, solve=k, sync=False)
        s.step(case["steps"])
        for k, u in enumerate(state["out"]):
            s.get_state(u, solve=k, sync=False)
    if case["prec"] == "fp64":
        return {"state": state["out"]}
    for snap, u in zip(state["snapshot"], state["out"]):
        snap.copy_(u)
    return {"state": state["snapshot"]}


def work(case):
    """The state read and the snapshot written once; the counted operations of every step."""
    if case["flow"] == "batch":
        sizes = np.random.default_rng(case["nx"])
        meshes = []
        for _ in range(case["nx"]):
            side, deg = int(sizes.integers(16, 129)), int(sizes.integers(2, 6))
            meshes.append(_mesh("euler", 2, deg, [side, side], -1.0, 1.0, 1.4, case["vol"]))
    else:
        dim = {"wave": 1, "shear": 2, "vortex": 2, "tgv": 3}[case["flow"]]
        eq = "glm_mhd" if case["flow"] == "vortex" else "euler"
        meshes = [_mesh(eq, dim, case["N"], [case["nx"], case["ny"], case["nz"]][:dim], 0.0, 1.0, 1.4, case["vol"])]
    size = 8 if case["prec"] == "fp64" else 4
    nbytes = flops = 0.0
    for m in meshes:
        values = counted.nvars(m) * float(np.prod(m["cells"][:m["dim"]])) * (m["N"] + 1) ** m["dim"]
        nbytes += values * (8 + size)
        flops += case["steps"] * counted.volume_flops(m)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------------------
# the scheme in plain FP64 torch operations
# ---------------------------------------------------------------------------
def _tableau(N):
    rows = {1: [[1.0]],
            2: [[1 / 3], [0, 2 / 3]],
            3: [[0.5], [0, 0.5], [0, 0, 1.0]],
            4: [[1 / 4], [1 / 8, 1 / 8], [0, -1 / 2, 1.0], [3 / 16, 0, 0, 9 / 16],
                [-3 / 7, 2 / 7, 12 / 7, -12 / 7, 8 / 7]],
            5: [[1 / 3], [0, 2 / 3], [1 / 12, 1 / 3, -1 / 12], [-1 / 16, 9 / 8, -3 / 16, -3 / 8],
                [0, 9 / 8, -3 / 8, -3 / 4, 1 / 2], [9 / 44, -9 / 11, 63 / 44, 18 / 11, 0, -16 / 11]]}[N]
    b = {1: [0.5, 0.5], 2: [0.25, 0, 0.75], 3: [1 / 6, 1 / 3, 1 / 3, 1 / 6],
         4: [7 / 90, 0, 32 / 90, 12 / 90, 32 / 90, 7 / 90],
         5: [11 / 120, 0, 27 / 40, 27 / 40, -4 / 15, -4 / 15, 11 / 120]}[N]
    return [[]] + rows, b


class _Plain:
    """One solve: the cRKFR step (with or without the limiter) and the multi-stage RKFR step.
    Arrays are [var][elements, last direction first][nodes, likewise]: direction d has node axis -(1+d) and
    element axis -(1+dim+d)."""

    def __init__(self, mesh):
        self.m, self.dim, self.N, self.g = mesh, mesh["dim"], mesh["N"], mesh["gamma"]
        self.mhd = mesh["eq"] == "glm_mhd"
        self.xi, self.w, self.D = _gll(self.N)
        self.a, self.b = _tableau(self.N)
        self.idx = [mesh["cells"][d] / (mesh["hi"][d] - mesh["lo"][d]) for d in range(self.dim)]
        self.nv = 3 if self.mhd else self.dim   # velocity components

    # ---- point-wise physics on q = (rho, v.., p, [B1, B2, B3, psi])
    def prim(self, u):
        v = [u[1 + k] / u[0] for k in range(self.nv)]
        e = u[1 + self.nv] - 0.5 * u[0] * sum(x * x for x in v)
        if self.mhd:
            e = e - 0.5 * (u[5] ** 2 + u[6] ** 2 + u[7] ** 2 + u[8] ** 2)
        q = [u[0]] + v + [(self.g - 1.0) * e]
        return torch.stack(q + ([u[5], u[6], u[7], u[8]] if self.mhd else []))

    def energy(self, q):
        nv = self.nv
        E = q[1 + nv] / (self.g - 1.0) + 0.5 * q[0] * sum(q[1 + k] ** 2 for k in range(nv))
        return E + 0.5 * (q[5] ** 2 + q[6] ** 2 + q[7] ** 2 + q[8] ** 2) if self.mhd else E

    def flux(self, d, q):
        nv, vd, p = self.nv, q[1 + d], q[1 + self.nv]
        if not self.mhd:
            f = [q[0] * vd] + [q[0] * vd * q[1 + k] + (p if k == d else 0.0) for k in range(nv)]
            return torch.stack(f + [vd * (self.energy(q) + p)])
        ch, Bd, psi = self.m["c_h"], q[5 + d], q[8]
        B2, vB = sum(q[5 + k] ** 2 for k in range(3)), sum(q[1 + k] * q[5 + k] for k in range(3))
        v2 = sum(q[1 + k] ** 2 for k in range(3))
        f = [q[0] * vd]
        f += [q[0] * vd * q[1 + k] - Bd * q[5 + k] + (p + 0.5 * B2 if k == d else 0.0) for k in range(3)]
        f += [vd * (0.5 * q[0] * v2 + self.g / (self.g - 1.0) * p + B2) - Bd * vB + ch * psi * Bd]
        f += [ch * psi if k == d else vd * q[5 + k] - q[1 + k] * Bd for k in range(3)]
        return torch.stack(f + [ch * Bd])

    @staticmethod
    def logmean(a, b):
        f = (a - b) / (a + b)
        x = f * f
        small = x < 1e-3
        series = 1 + x * (1 / 3 + x * (1 / 5 + x * (1 / 7 + x * (1 / 9 + x * (1 / 11 + x * (1 / 13))))))
        big = torch.where(small, torch.full_like(f, 0.5), f)
        return 0.5 * (a + b) / torch.where(small, series, torch.atanh(big) / big)

    def two_point(self, d, a, b):
        if self.m["vol"] == "central":
            return 0.5 * (self.flux(d, a) + self.flux(d, b))
        nv = self.nv
        v = [0.5 * (a[1 + k] + b[1 + k]) for k in range(nv)]
        pa, pb = a[1 + nv], b[1 + nv]
        if self.m["vol"] == "kep":
            ravg, pavg = 0.5 * (a[0] + b[0]), 0.5 * (pa + pb)
            eavg = 0.5 * (self.energy(a) / a[0] + self.energy(b) / b[0])
            f = [ravg * v[d]] + [ravg * v[d] * v[k] + (pavg if k == d else 0.0) for k in range(nv)]
            return torch.stack(f + [(ravg * eavg + pavg) * v[d]])
        if not self.mhd:
            f0 = self.logmean(a[0], b[0]) * v[d]
            vv = sum(a[1 + k] * b[1 + k] for k in range(nv))
            f = [f0] + [f0 * v[k] + (0.5 * (pa + pb) if k == d else 0.0) for k in range(nv)]
            e = f0 * (0.5 * vv + 1.0 / ((self.g - 1.0) * self.logmean(a[0] / pa, b[0] / pb)))
            return torch.stack(f + [e + 0.5 * (pa * b[1 + d] + pb * a[1 + d])])
        ch = self.m["c_h"]
        B = [0.5 * (a[5 + k] + b[5 + k]) for k in range(3)]
        psi, Bd = 0.5 * (a[8] + b[8]), B[d]
        ba, bb = a[0] / (2.0 * pa), b[0] / (2.0 * pb)
        sq = lambda q, i: q[i] ** 2 + q[i + 1] ** 2 + q[i + 2] ** 2  # noqa: E731
        vB = lambda q: q[1] * q[5] + q[2] * q[6] + q[3] * q[7]       # noqa: E731
        f0 = self.logmean(a[0], b[0]) * v[d]
        pt = (a[0] + b[0]) / (2.0 * (ba + bb)) + 0.25 * (sq(a, 5) + sq(b, 5))
        fm = [f0 * v[k] - Bd * B[k] + (pt if k == d else 0.0) for k in range(3)]
        fB = [ch * psi if k == d else v[d] * B[k] - v[k] * Bd for k in range(3)]
        e = 0.5 * f0 * (1.0 / ((self.g - 1.0) * self.logmean(ba, bb)) - 0.5 * (sq(a, 1) + sq(b, 1)))
        e = e + sum(fm[k] * v[k] + fB[k] * B[k] for k in range(3)) + ch * Bd * psi
        e = e - 0.25 * (a[1 + d] * sq(a, 5) + b[1 + d] * sq(b, 5))
        e = e - 0.5 * ch * (a[8] * a[5 + d] + b[8] * b[5 + d]) + 0.5 * Bd * (vB(a) + vB(b))
        return torch.stack([f0] + fm + [e] + fB + [ch * Bd])

    def speed(self, d, q):
        a2 = self.g * q[1 + self.nv] / q[0]
        if not self.mhd:
            return q[1 + d].abs() + a2.sqrt()
        s = a2 + (q[5] ** 2 + q[6] ** 2 + q[7] ** 2) / q[0]
        c = (0.5 * (s + (s * s - 4.0 * a2 * q[5 + d] ** 2 / q[0]).clamp(min=0.0).sqrt())).sqrt()
        return q[1 + d].abs() + c.clamp(min=self.m["c_h"])

    def nonconservative(self, d, q, g0, g1):
        z, vB = torch.zeros_like(g0), q[1] * q[5] + q[2] * q[6] + q[3] * q[7]
        return torch.stack([z, q[5] * g0, q[6] * g0, q[7] * g0, vB * g0 + q[1 + d] * q[8] * g1,
                            q[1] * g0, q[2] * g0, q[3] * g0, q[1 + d] * g1])

    # ---- element-local residual by flux differencing
    def residual(self, q):
        R = torch.zeros((q.shape[0],) + q.shape[1:], dtype=q.dtype, device=q.device)
        for d in range(self.dim):
            ax, Dx = -(1 + d), self.D * self.idx[d]
            line = [q.select(ax, k) for k in range(self.N + 1)]
            for k in (0, self.N):
                R.select(ax, k).add_(2.0 * Dx[k, k] * self.flux(d, line[k]))
            for i in range(self.N + 1):
                for j in range(i + 1, self.N + 1):
                    f = self.two_point(d, line[i], line[j])
                    R.select(ax, i).add_(2.0 * Dx[i, j] * f)
                    R.select(ax, j).add_(2.0 * Dx[j, i] * f)
            if self.mhd:
                for i in range(self.N + 1):
                    g0 = sum(Dx[i, j] * line[j][5 + d] for j in range(self.N + 1))
                    g1 = sum(Dx[i, j] * line[j][8] for j in range(self.N + 1))
                    R.select(ax, i).add_(self.nonconservative(d, line[i], g0, g1))
        return R

    def at_ends(self, fn):
        """fn(d, node index) at both ends of every direction: {(d, side)}."""
        return {(d, s): fn(d, s * self.N) for d in range(self.dim) for s in (0, 1)}

    def end(self, t, d, k):
        return t.select(-(1 + d), k)

    def shift(self, t, d, by):   # a face array (node axis d already gone) from the neighbour
        return torch.roll(t, by, -(self.dim + d))

    def increment(self, dt, Rbar, U, F, G, qn, fnum=None):
        """-dt times the time-averaged residual with the face jumps; U, F, G: time averages at the ends, qn: u^n."""
        du = -dt * Rbar
        for d in range(self.dim):
            c = dt * self.idx[d]
            Fn = self.rusanov(d, U, F, qn) if fnum is None else fnum[d]
            jN, j0 = Fn - F[d, 1], self.shift(Fn, d, 1) - F[d, 0]
            if self.mhd:
                for i, g in ((0, 5 + d), (1, 8)):
                    m = 0.5 * (U[d, 1][g] + self.shift(U[d, 0], d, -1)[g])
                    z = torch.zeros_like(m)
                    jN = jN + self.nonconservative(d, self.end(qn, d, self.N), *((m, z) if i == 0 else (z, m)))
                    m = self.shift(m, d, 1)
                    j0 = j0 + self.nonconservative(d, self.end(qn, d, 0), *((m, z) if i == 0 else (z, m)))
                jN, j0 = jN - G[d, 1], j0 - G[d, 0]
            self.end(du, d, self.N).sub_(c / self.w[-1] * jN)
            self.end(du, d, 0).add_(c / self.w[0] * j0)
        return du

    def rusanov(self, d, U, F, qn):
        lam = torch.maximum(self.speed(d, self.end(qn, d, self.N)),
                            self.shift(self.speed(d, self.end(qn, d, 0)), d, -1))
        return 0.5 * (F[d, 1] + self.shift(F[d, 0], d, -1)) - 0.5 * lam * (self.shift(U[d, 0], d, -1) - U[d, 1])

    def records(self, u, q):
        U = self.at_ends(lambda d, k: self.end(u, d, k).clone())
        F = self.at_ends(lambda d, k: self.flux(d, self.end(q, d, k)))
        if not self.mhd:
            return U, F, None
        e = lambda d, k: self.end(q, d, k)  # noqa: E731
        return U, F, self.at_ends(lambda d, k: self.nonconservative(d, e(d, k), e(d, k)[5 + d], e(d, k)[8]))

    def step(self, u):
        q0 = self.prim(u)
        dt = self.m["cfl"] / sum(self.speed(d, q0) * self.idx[d] for d in range(self.dim)).max()
        if self.m.get("scheme") == "rkfr":
            K = []
            for j in range(len(self.b)):
                uj = u + sum(c * k for c, k in zip(self.a[j], K) if c) if j else u
                qj = self.prim(uj)
                K.append(self.increment(dt, self.residual(qj), *self.records(uj, qj), qj))
            return u + sum(c * k for c, k in zip(self.b, K) if c)
        Rs, Rbar, avg = [], 0.0, None
        for i, bi in enumerate(self.b):
            ui = u - dt * sum(c * r for c, r in zip(self.a[i], Rs) if c) if i else u
            qi = self.prim(ui)
            Rs.append(self.residual(qi))
            if bi:
                Rbar = Rbar + bi * Rs[-1]
                rec = self.records(ui, qi)
                scaled = [None if r is None else {k: bi * v for k, v in r.items()} for r in rec]
                avg = scaled if avg is None else [None if r is None else {k: a[k] + r[k] for k in r}
                                                  for a, r in zip(avg, scaled)]
        U, F, G = avg
        if not self.m.get("limiter"):
            return u + self.increment(dt, Rbar, U, F, G, q0)
        alpha = self.blending(q0)
        fnum = {d: self.limited_flux(d, u, q0, alpha, dt, self.rusanov(d, U, F, q0)) for d in range(self.dim)}
        high = u + self.increment(dt, Rbar, U, F, G, q0, fnum)
        low = u.clone()
        for d in range(self.dim):
            ax = -(1 + d)
            f = [self.shift(fnum[d], d, 1)]
            for k in range(self.N):
                f.append(self.two_state(d, u.select(ax, k), u.select(ax, k + 1)))
            f.append(fnum[d])
            for k in range(self.N + 1):
                low.select(ax, k).sub_(dt * self.idx[d] / self.w[k] * (f[k + 1] - f[k]))
        a = alpha.reshape(alpha.shape + (1,) * self.dim)
        return torch.where(a >= 1.0, low, (1.0 - a) * high + a * low)

    # ---- subcell blending limiter
    def two_state(self, d, ul, ur):
        ql, qr = self.prim(ul), self.prim(ur)
        lam = torch.maximum(self.speed(d, ql), self.speed(d, qr))
        return 0.5 * (self.flux(d, ql) + self.flux(d, qr)) - 0.5 * lam * (ur - ul)

    def blending(self, q):
        n, N, dim = self.N + 1, self.N, self.dim
        V = np.stack([math.sqrt((2 * j + 1) / 2.0) * np.polynomial.legendre.Legendre.basis(j)(2 * self.xi - 1)
                      for j in range(n)], axis=1)
        Vi = torch.tensor(np.linalg.inv(V), dtype=torch.float64, device=q.device)
        m = q[0] * q[1 + self.nv]
        for d in range(dim):
            m = torch.movedim(torch.movedim(m, -(1 + d), -1) @ Vi.T, -1, -(1 + d))
        top = torch.zeros((n,) * dim, device=q.device)
        for d in range(dim):
            top = torch.maximum(top, torch.arange(n, device=q.device).reshape((n,) + (1,) * d))
        e2, axes = m * m, tuple(range(-dim, 0))
        T, T1, T2 = (torch.where(top <= k, e2, torch.zeros_like(e2)).sum(axes) for k in (N, N - 1, N - 2))
        E = torch.maximum((T - T1) / T, (T1 - T2) / T1) if N >= 2 else (T - T1) / T
        tau = 0.5 * 10.0 ** (-1.8 * n ** 0.25)
        a = 1.0 / (1.0 + torch.exp(-(math.log(9999.0) / tau) * (E - tau)))
        a = torch.where(a < 0.001, torch.zeros_like(a), torch.where(a > 0.999, torch.ones_like(a), a))
        a = a.clamp(max=self.m["alpha_max"])
        out = a
        for d in range(dim):
            for by in (1, -1):
                out = torch.maximum(out, 0.5 * torch.roll(a, by, -(1 + d)))
        return out

    def limited_flux(self, d, u, q, alpha, dt, Fho):
        """The blended and admissibility-corrected flux at every '-' element's end face."""
        N, ax, g1 = self.N, -(1 + d), self.g - 1.0
        um, umi = u.select(ax, N), u.select(ax, N - 1)
        up, upi = self.shift(u.select(ax, 0), d, -1), self.shift(u.select(ax, 1), d, -1)
        af = 0.5 * (alpha + torch.roll(alpha, -1, -(1 + d)))
        af = af.reshape(af.shape + (1,) * (self.dim - 1))
        flo = self.two_state(d, um, up)
        Fb = torch.where(af >= 1.0, flo, (1.0 - af) * Fho + af * flo)
        c = self.dim * dt * self.idx[d]
        lm, dm = um - c / self.w[-1] * (flo - self.two_state(d, umi, um)), -c / self.w[-1] * (Fb - flo)
        lp, dp = up - c / self.w[0] * (self.two_state(d, up, upi) - flo), c / self.w[0] * (Fb - flo)

        def pressure(s):
            return g1 * (s[-1] - 0.5 * sum(s[1 + k] ** 2 for k in range(self.dim)) / s[0])

        def theta(s, ds):
            r0, r1, p0 = s[0], s[0] + ds[0], pressure(s)
            t = torch.where(r1 < 0.1 * r0, 0.9 * r0 / torch.where(r1 < r0, r0 - r1, torch.ones_like(r0)),
                            torch.ones_like(r0))
            pt = pressure(s + t * ds)
            t = torch.where(pt < 0.1 * p0, t * 0.9 * p0 / torch.where(pt < p0, p0 - pt, torch.ones_like(p0)), t)
            return torch.where((r0 > 0) & (p0 > 0), t, torch.zeros_like(t))

        F = flo + torch.minimum(theta(lm, dm), theta(lp, dp)) * (Fb - flo)
        return torch.where(af > 0.0, F, Fb)


def exact(case, seed):
    out = []
    for mesh, u in _initial(case, seed):
        s = _Plain(dict(mesh, scheme=case["scheme"]))
        for _ in range(case["steps"]):
            u = s.step(u)
        out.append(u.reshape(u.shape[0], -1))
    return {"state": out}
