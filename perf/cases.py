"""What is measured: time steps of the library's cases through its public entry points.

A pass of a case is what a time-marching program does between two looks at its solution: it advances the
case (or the batch of cases) by the case's number of steps and packs the whole new state into a device
buffer (``Case.halo_pack``, the call that moves cells between subdomains), which is the pass's output: the
distribution f, the conserved variables W and the heat flux q.  Passes of one state continue the march.

The states are far from equilibrium (two streams of different velocity and temperature, as inside a shock,
on a seeded smooth field around the workload's own start), so every term of the step is at work.  W and q of
an FP32-storage case are handed over in single precision, the precision of its distribution.
"""
import functools
import math

import numpy as np
import torch

from paper_2412_06546_gb300 import _lib, cases, serving

# cell-velocity updates of the largest listed case's pass; a drawn case stays below them
_MOST = 1.0e9


def listed():
    return [
        # the lid-driven cavity of the tests and the smoke run: the smallest case, launch latency counts
        {"name": "cavity20_v24_fp32", "kind": "cavity", "n": 20, "nvx": 24, "nvy": 24, "precision": "fp32", "steps": 10},
        # the same in the plain FP64 form
        {"name": "cavity20_v24_fp64", "kind": "cavity", "n": 20, "nvx": 24, "nvy": 24, "precision": "fp64", "steps": 10},
        # Mach-5 cylinder on the tests' 2,000-cell triangulation, odd velocity grid
        {"name": "cylinder2k_v30x25_fp32", "kind": "cylinder", "cells": 2000, "nvx": 30, "nvy": 25, "precision": "fp32",
         "steps": 10},
        # the benchmark's cylinder: 30k triangles, 60 x 50 velocities
        {"name": "cylinder30k_v60x50_fp32", "kind": "cylinder", "cells": 30000, "nvx": 60, "nvy": 50,
         "precision": "fp32", "steps": 4},
        # the same mesh on the unstructured velocity mesh of 2,060 triangles (no factored face sums)
        {"name": "cylinder30k_dvs2060_fp32", "kind": "cylinder_dvs", "cells": 30000, "nv": 2060, "precision": "fp32",
         "steps": 4},
        # plain FP64 form of the cylinder, the accuracy reference runs
        {"name": "cylinder8k_v60x50_fp64", "kind": "cylinder", "cells": 8000, "nvx": 60, "nvy": 50, "precision": "fp64",
         "steps": 1},
        # 3D cavity of hexahedra, odd extents: six faces per cell
        {"name": "hex15x13x11_v17x16x15_fp32", "kind": "hex", "nx": 15, "ny": 13, "nz": 11, "nvx": 17, "nvy": 16,
         "nvz": 15, "precision": "fp32", "steps": 4},
        # tetrahedra around a body, FP64
        {"name": "body11k_v14_fp64", "kind": "body", "h0": 0.8, "surface": 6000, "nvx": 14, "nvy": 14, "nvz": 14,
         "precision": "fp64", "steps": 1},
        # tetrahedra around a body on a 28^3 tensor grid
        {"name": "body24k_v28_fp32", "kind": "body", "h0": 0.5, "surface": 10000, "nvx": 28, "nvy": 28, "nvz": 28,
         "precision": "fp32", "steps": 2},
        # the benchmark's lifting body (its 100k-cell instance) on the unstructured 3D velocity mesh
        {"name": "body107k_v4548_fp32", "kind": "body_dvs", "h0": 0.2, "surface": 100000, "nv": 4548,
         "precision": "fp32", "steps": 2},
        # a serving tick: eight mixed requests of the stream stepped together
        {"name": "serving8_fp32", "kind": "batch", "requests": 8, "stream": 4, "precision": "fp32", "steps": 25},
    ]


def draw(rng):
    """A case of the ranges above: sizes spread over their logarithm, odd ones among them."""
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["cavity", "cylinder", "cylinder", "cylinder_dvs", "hex", "body", "body_dvs", "batch"])
    c = {"kind": kind, "precision": "fp64" if rng.random() < 0.2 else "fp32", "steps": rng.choice([1, 2, 3, 5])}
    if kind == "cavity":
        c.update(n=log(16, 100), nvx=rng.randint(16, 48), nvy=rng.randint(16, 48))
        cvu = c["n"] ** 2 * c["nvx"] * c["nvy"]
    elif kind == "cylinder":
        c.update(cells=log(1000, 30000), nvx=rng.randint(20, 64), nvy=rng.randint(20, 64))
        cvu = c["cells"] * c["nvx"] * c["nvy"]
    elif kind == "cylinder_dvs":
        c.update(cells=log(2000, 30000), nv=rng.randint(1200, 3420))
        cvu = c["cells"] * c["nv"]
    elif kind == "hex":
        c.update(nx=rng.randint(5, 24), ny=rng.randint(5, 24), nz=rng.randint(5, 24), nvx=rng.randint(12, 24),
                 nvy=rng.randint(12, 24), nvz=rng.randint(12, 24))
        cvu = c["nx"] * c["ny"] * c["nz"] * c["nvx"] * c["nvy"] * c["nvz"]
    elif kind == "body":
        c.update(h0=round(math.exp(rng.uniform(math.log(0.4), math.log(1.0))), 3), surface=10000)
        c.update({a: rng.randint(13, 26) for a in ("nvx", "nvy", "nvz")})
        cvu = 36000 * (0.4 / c["h0"]) ** 2 * c["nvx"] * c["nvy"] * c["nvz"]
    elif kind == "body_dvs":
        c.update(h0=round(math.exp(rng.uniform(math.log(0.25), math.log(0.8))), 3), surface=40000,
                 nv=rng.randint(1500, 4548))
        cvu = 80000 * (0.25 / c["h0"]) ** 2 * c["nv"]
    else:
        c.update(requests=rng.randint(3, 10), stream=rng.randint(10, 40), steps=rng.choice([10, 25]))
        cvu = c["requests"] * 2500 * 600
    if c["precision"] == "fp64":            # the plain form: smaller runs, one step
        c["steps"] = 1
        if kind == "batch" or cvu > 4e7:
            c["precision"] = "fp32"
    while c["steps"] > 1 and cvu * c["steps"] > 0.6 * _MOST:
        c["steps"] -= 1
    return c


# ---------------------------------------------------------------- the set-ups: meshes, velocities, parameters
@functools.lru_cache(maxsize=8)
def _cylinder_mesh(cells):
    return cases.cylinder_mesh(cells, seed=2)


@functools.lru_cache(maxsize=8)
def _body_mesh(h0, surface):
    m = cases.x38_mesh(h0, seed=5, n_surface=surface)
    m.pop("_surface")
    return m


@functools.lru_cache(maxsize=8)
def _disk(nv):
    return cases.cylinder_dvs_vgrid(5.0, "E1", n_target=nv)


@functools.lru_cache(maxsize=8)
def _ball(nv, U):
    R = 4.0 * math.sqrt(1.0 + 64.0 / 3.0)
    return cases.tet_ball_vgrid(nv, R=R, centres=((0.0, 0.0, 0.0), U), seed=5)


@functools.lru_cache(maxsize=4)
def _stream(requests, seed):
    return serving.request_stream(requests, seed=seed)


def _body_start(mesh, U):
    """rho = T = 1 and a velocity that rises from rest at the body to the free stream."""
    s = 1.0 - np.exp(-2.0 * (np.maximum(cases.x38_body_F(mesh["cell_xc"]), 1.0) ** 0.25 - 1.0))
    init = cases.uniform_state(len(s), 3)
    init[:, 1:4] = s[:, None] * np.asarray(U)[None]
    return init


def _setups(case):
    """The case dicts (mesh, vgrid, params, init) of a pass: one, or a batch's several."""
    k = case["kind"]
    if k == "cavity":
        c = cases.cavity_case(n=case["n"], nv=24)
        c["vgrid"] = cases.cartesian_vgrid((case["nvx"], case["nvy"]), (-5.0, -5.0), (5.0, 5.0))
        return [c]
    if k in ("cylinder", "cylinder_dvs"):
        mesh = _cylinder_mesh(case["cells"])
        U = cases.freestream_speed(5.0)
        pr = cases.params(0.1, L_ref=2.0, walls=[{"T": 1.0, "U": [0.0, 0.0, 0.0]}],
                          inf={"rho": 1.0, "U": [U, 0.0, 0.0], "T": 1.0})
        vg = (cases.cartesian_vgrid((case["nvx"], case["nvy"]), (-12.0, -10.0), (12.0, 10.0)) if k == "cylinder"
              else _disk(case["nv"]))
        return [{"mesh": mesh, "vgrid": vg, "params": pr, "init": cases.blended_start(mesh, [U, 0.0])}]
    if k == "hex":
        n = (case["nx"], case["ny"], case["nz"])
        mesh = cases.hex_mesh(*n, sides={"z+": ("wall", 1)})
        vg = cases.cartesian_vgrid((case["nvx"], case["nvy"], case["nvz"]), (-5.0,) * 3, (5.0,) * 3)
        pr = cases.params(0.075, walls=[{"T": 1.0, "U": [0.0] * 3}, {"T": 1.0, "U": [0.16, 0.0, 0.0]}])
        return [{"mesh": mesh, "vgrid": vg, "params": pr, "init": cases.uniform_state(len(mesh["cell_vol"]), 3)}]
    if k in ("body", "body_dvs"):
        mesh = _body_mesh(case["h0"], case["surface"])
        mach, Kn, Tw = (4.0, 0.1, 1.0) if k == "body" else (8.0, 0.005, 302.0 / 56.0)
        a = math.radians(20.0)
        Uinf = cases.freestream_speed(mach)
        U = (Uinf * math.cos(a), 0.0, Uinf * math.sin(a))
        vg = (cases.cartesian_vgrid((case["nvx"], case["nvy"], case["nvz"]), (-10.0,) * 3, (10.0,) * 3)
              if k == "body" else _ball(case["nv"], U))
        pr = cases.params(Kn, L_ref=8.0, walls=[{"T": Tw, "U": [0.0] * 3}], inf={"rho": 1.0, "U": list(U), "T": 1.0})
        return [{"mesh": mesh, "vgrid": vg, "params": pr, "init": _body_start(mesh, U)}]
    return _stream(case["requests"], case["stream"])


def _gpu(a):
    return torch.as_tensor(np.asarray(a), device="cuda")


def _moments(f, u, w, D):
    """W of a distribution f[C][NC][Nv] (FP64 sums)."""
    h = f[:, 0].double() * w
    E = 0.5 * (h @ (u * u).sum(1))
    if D == 2:
        E = E + 0.5 * (f[:, 1].double() @ w)
    return torch.cat([h.sum(1, keepdim=True), h @ u, E[:, None]], 1)


def _state(setup, dtype, seed):
    """A seeded non-equilibrium state (f, W): in every cell two Maxwellian streams, the second faster and
    hotter, around a smooth perturbation of the workload's start."""
    mesh, vg = setup["mesh"], setup["vgrid"]
    D, C, Nv = mesh["dim"], len(mesh["cell_vol"]), len(vg["w"])
    rng = np.random.default_rng(seed)
    x = mesh["cell_xc"]
    size = x.max(0) - x.min(0)
    k = rng.uniform(1.0, 3.0, size=(2 * D + 2, D)) * 2.0 * np.pi / size
    wave = _gpu(np.sin(x @ k.T + rng.uniform(0.0, 2.0 * np.pi, 2 * D + 2)))
    p = _gpu(setup["init"])
    rho, T = p[:, 0] * (1.0 + 0.1 * wave[:, 0]), p[:, D + 1] * (1.0 + 0.1 * wave[:, 1])
    U, dU = p[:, 1:1 + D] + 0.1 * wave[:, 2:2 + D], 0.5 + 0.3 * wave[:, 2 + D:]
    u, w = _gpu(vg["u"]), _gpu(vg["w"])
    f = torch.empty((C, 4 - D, Nv), dtype=dtype, device="cuda")
    W = torch.empty((C, D + 2), dtype=torch.float64, device="cuda")
    n = max(1, 20_000_000 // Nv)
    for c in range(0, C, n):
        s = slice(c, c + n)
        g = 0
        for part, Us, Ts in ((0.75, U[s], T[s]), (0.25, U[s] + dU[s], 1.4 * T[s])):
            c2 = sum((u[None, :, d] - Us[:, d, None]) ** 2 for d in range(D))
            h = part * rho[s, None] * (2.0 * np.pi * Ts[:, None]) ** (-0.5 * D) * torch.exp(-0.5 * c2 / Ts[:, None])
            g = g + torch.stack([h, Ts[:, None] * h][:4 - D], 1)
        f[s] = g.to(dtype)
        W[s] = _moments(f[s], u, w, D)
    return f, W


def _seeds(case, seed):
    return [1000 * seed + i for i in range(len(_setups(case)))]


# ---------------------------------------------------------------- a pass
def prepare(case, seed):
    prec, dtype = (_lib.FP64, torch.float64) if case["precision"] == "fp64" else (_lib.FP32, torch.float32)
    batch = case["kind"] == "batch"
    tiling = {"vtile": 64, "threads": 256} if batch else {}        # the serving loop's
    members = []
    for setup, s in zip(_setups(case), _seeds(case, seed)):
        g = _lib.Case(setup["mesh"], setup["vgrid"], setup["params"], setup["init"], precision=prec, **tiling)
        f, W = _state(setup, dtype, s)
        g.set_state(f.cpu().numpy(), W.cpu().numpy())
        g.halo_set(0, np.arange(g.C))
        row = g.halo_row_bytes()
        buf = torch.empty((g.C, row), dtype=torch.uint8, device="cuda")
        nf = g.nc * g.Nv
        tail = buf[:, row - 8 * (2 * g.D + 2):].view(torch.float64)
        members.append({"case": g, "buf": buf, "f": buf[:, :nf * dtype.itemsize].view(dtype),
                        "W": tail[:, :g.D + 2], "q": tail[:, g.D + 2:]})
    torch.cuda.synchronize()
    mover = _lib.Batch([m["case"] for m in members]) if batch else members[0]["case"]
    return {"members": members, "mover": mover, "steps": case["steps"], "macro": dtype}


def run(state):
    state["mover"].step(state["steps"])
    out = []
    for m in state["members"]:
        m["case"].halo_pack(0, m["buf"].data_ptr())
        out.append({"f": m["f"], "W": m["W"].to(state["macro"]), "q": m["q"].to(state["macro"])})
    return out


def work(case):
    """Per step: f read and written once; the limited slopes, one flux per face, both stages and the moments,
    and the face sums (over the axes' nodes on a tensor grid, over every velocity otherwise)."""
    size = 8 if case["precision"] == "fp64" else 4
    nbytes = flops = 0.0
    for s in _setups(case):
        D, C, F, Nv = s["mesh"]["dim"], len(s["mesh"]["cell_vol"]), len(s["mesh"]["face_S"]), len(s["vgrid"]["w"])
        NC = 4 - D
        nf = 2.0 * F / C
        slope = NC * (nf * (4 * D + 1) + 20 + 3 * D + 3)
        face = (2 * D - 1) + NC * (4 * D - 1) + 3 * D + 2 + NC * (D * D + 6 * D + 10)
        stages = 2 * (5 * D + 7 + 9 * NC) + 4 * D + 7
        sums = 0.0 if s["vgrid"]["cart_n"][0] else F / C * (14 * D + 12 + 6 * D * D + 15 * D)
        flops += case["steps"] * float(C) * Nv * (slope + 0.5 * nf * face + stages + sums)
        nbytes += (case["steps"] * 2 + 1) * float(C) * NC * Nv * size
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- the same step in plain 64-bit torch
class _Plain:
    """One explicit step of the scheme on whole arrays in FP64; velocities are taken in slices."""

    def __init__(self, setup):
        m, v, p = setup["mesh"], setup["vgrid"], setup["params"]
        self.D = D = m["dim"]
        self.M, self.NC = D + 2, 4 - D
        self.C, self.F, self.Nv = len(m["cell_vol"]), len(m["face_S"]), len(v["w"])
        self.nxi, self.p = 3.0 - D, p
        self.u, self.w = _gpu(v["u"]), _gpu(v["w"])
        own, nei, t = m["face_cells"][:, 0], m["face_cells"][:, 1], m["face_type"]
        xc, n = m["cell_xc"], m["face_n"]
        inner = (t == cases.INTERIOR) | (t == cases.PERIODIC)
        far, wall = np.nonzero(t == cases.FARFIELD)[0], np.nonzero(t == cases.WALL)[0]
        shift = np.where((t == cases.PERIODIC)[:, None], m["face_shift"], 0.0)
        rL, rR = m["face_xc"] - xc[own], m["face_xc"] - shift - xc[np.maximum(nei, 0)]
        ghost = np.full(self.F, -1)
        ghost[far] = self.C + np.arange(len(far))
        other = np.where(inner, nei, np.where(ghost >= 0, ghost, own))
        dL = np.where(inner[:, None], rL - rR, 2.0 * (rL * n).sum(1, keepdims=True) * n)
        dL[wall] = 0.0
        # one row per (cell, face), then padded to the same number of faces in every cell
        cell = np.concatenate([own, nei[inner]])
        face = np.concatenate([np.arange(self.F), np.nonzero(inner)[0]])
        nb, r = np.concatenate([other, own[inner]]), np.concatenate([rL, rR[inner]])
        d, sign = np.concatenate([dL, -dL[inner]]), np.concatenate([np.ones(self.F), -np.ones(inner.sum())])
        order = np.lexsort((face, cell))
        cell, face, nb, r, d, sign = (a[order] for a in (cell, face, nb, r, d, sign))
        pos = np.arange(len(cell)) - np.searchsorted(cell, cell)
        NF = int(pos.max()) + 1

        def pad(a, fill):
            out = np.broadcast_to(fill, (self.C, NF) + a.shape[1:]).copy()
            out[cell, pos] = a
            return out

        S = m["face_S"][face]
        dd = (d * d).sum(1)
        wt = np.where(dd > 0, 1.0 / np.where(dd > 0, dd, 1.0), 0.0)
        A = np.zeros((self.C, D, D))
        np.add.at(A, cell, wt[:, None, None] * d[:, :, None] * d[:, None, :])
        ok = np.abs(np.linalg.det(A)) > 1e-12 * (np.trace(A, axis1=1, axis2=2) / D) ** D
        inv = np.where(ok[:, None, None], np.linalg.inv(np.where(ok[:, None, None], A, np.eye(D))), 0.0)
        a = np.einsum("eij,ej->ei", inv[cell], d) * wt[:, None]
        sumS = np.bincount(cell, S, self.C)
        self.nb = _gpu(pad(nb, np.arange(self.C)[:, None]))
        self.a, self.r = _gpu(pad(a, 0.0)), _gpu(pad(r, 0.0))
        self.face, self.cs = _gpu(pad(face, 0)), _gpu(pad(-sign * S / m["cell_vol"][cell], 0.0))
        self.eps2 = _gpu((p["venkat_K"] * 2.0 * D * m["cell_vol"] / sumS) ** 3)[:, None]
        umax = np.sqrt((v["u"] ** 2).sum(1)).max()
        self.dt = p["dt"] if p["dt"] > 0 else p["cfl"] * (2.0 * m["cell_vol"] / sumS).min() / umax
        self.L, self.R, self.n = _gpu(own), _gpu(other), _gpu(n)
        self.rL, self.rR = _gpu(rL), _gpu(np.where(inner[:, None], rR, 0.0))
        self.far, self.wall, self.two = _gpu(far), _gpu(wall), _gpu(inner)[:, None]
        om = p["omega"]
        self.mu = 15.0 * math.sqrt(2.0 * math.pi) * p["Kn"] * p["L_ref"] / (2.0 * (5.0 - 2.0 * om) * (7.0 - 2.0 * om))
        if len(wall):
            tag = m["face_tag"][wall]
            self.Tw = _gpu(np.array([q["T"] for q in p["walls"]])[tag])
            self.Uw = _gpu(np.array([(list(q["U"]) + [0.0] * 3)[:D] for q in p["walls"]])[tag])
        if len(far):
            inf = p["inf"]
            Ui = np.asarray(inf["U"][:D], float)
            self.Winf = _gpu(np.concatenate([[inf["rho"]], inf["rho"] * Ui,
                                             [inf["rho"] * (0.5 * (Ui * Ui).sum() + 1.5 * inf["T"])]]))
            self.inflow = _gpu(n[far] @ Ui < 0.0)[:, None]

    def prim(self, W):
        U = W[:, 1:-1] / W[:, :1]
        T = (2.0 / 3.0) * (W[:, -1] / W[:, 0] - 0.5 * (U * U).sum(1))
        return W[:, 0], U, T

    def maxwell(self, rho, U, T, ks):
        """H of every row's Maxwellian at the velocities ks, and c = u - U, |c|^2."""
        c = [self.u[ks, d] - U[:, d, None] for d in range(self.D)]
        c2 = sum(x * x for x in c)
        lam = 0.5 / T[:, None]
        return rho[:, None] * (lam / math.pi) ** (0.5 * self.D) * torch.exp(-lam * c2), c, c2

    def comps(self, H, T):
        return [H, T[:, None] * H][:self.NC]          # b of a Maxwellian: T h (N = 1 internal dof in 2D)

    def fplus(self, rho, U, T, q, ks):
        H, c, c2 = self.maxwell(rho, U, T, ks)
        lam = 0.5 / T
        k = (4.0 * (1.0 - self.p["Pr"]) * lam * lam / (5.0 * rho))[:, None]
        kqc = k * sum(q[:, d, None] * c[d] for d in range(self.D))
        l2 = 2.0 * lam[:, None] * c2
        out = [H * (1.0 + kqc * (l2 - self.D - 2)), T[:, None] * H * (1.0 + kqc * (l2 - self.D))][:self.NC]
        return out, H, c, c2

    def lsq(self, V, cells):
        """Limited least-squares gradients of the columns of V (cells, then ghosts) at `cells`."""
        vi, nb, a, r = V[:self.C][cells], self.nb[cells], self.a[cells], self.r[cells]
        g, hi, lo = [torch.zeros_like(vi) for _ in range(self.D)], vi.clone(), vi.clone()
        for e in range(nb.shape[1]):
            vj = V[nb[:, e]]
            df = vj - vi
            for d in range(self.D):
                g[d].addcmul_(a[:, e, d, None], df)
            hi, lo = torch.maximum(hi, vj), torch.minimum(lo, vj)
        if self.p["limiter"]:
            phi, e2 = torch.ones_like(vi), self.eps2[cells]
            for e in range(nb.shape[1]):
                d2 = sum(g[d] * r[:, e, d, None] for d in range(self.D))
                d1 = torch.where(d2 > 0, hi, lo) - vi
                s = d1 * d1 + e2
                phi = torch.minimum(phi, torch.where(d2 == 0, 1.0, (s + 2.0 * d1 * d2) / (s + d2 * (2.0 * d2 + d1))))
            g = [x * phi for x in g]
        return g

    def micro(self, V, cells, ks):
        """The same with the positivity scaling at the face centres and the foot of the characteristic."""
        g, vi, r = self.lsq(V, cells), V[:self.C][cells], self.r[cells]
        ug = sum(self.u[ks, d] * g[d] for d in range(self.D))
        low = torch.zeros_like(vi)
        for e in range(r.shape[1]):
            low = torch.minimum(low, sum(g[d] * r[:, e, d, None] for d in range(self.D)))
        low = vi + low + torch.clamp(-self.dt * ug, max=0.0)
        th = torch.where(low < 0, torch.where(vi > 0, vi / (vi - low), 0.0), 1.0)
        return [x * th for x in g]

    def tau(self, rho, T):
        return self.mu * T ** self.p["omega"] / (rho * T)

    def integrals(self, tau):
        dt, x = self.dt, self.dt / tau
        y = torch.clamp(x, max=0.5)
        s, fact, pw = [torch.zeros_like(x) for _ in range(5)], 1.0, torch.ones_like(x)
        for j in range(26):                            # sums over x^j / (j + 1)!, / (j + 2)!
            fact *= j + 1
            sg, f2 = (-1.0) ** j, fact * (j + 2)
            s[0] += sg * pw / fact
            s[1] -= sg * (j + 1) * pw / f2
            if j:
                s[2] -= sg * pw / fact
                s[3] += sg * j * pw / f2
                s[4] -= sg * pw / f2
            pw = pw * y
        e, E = torch.exp(-x), -torch.expm1(-x)
        big = [E / x, (x * e - E) / x ** 2, (x - E) / x, (2.0 * E - x * (1.0 + e)) / x ** 2, (0.5 * x * x - x + E) / x ** 2]
        return [torch.where(x < 0.5, a, b) * (dt if i in (0, 2) else dt * dt) for i, (a, b) in enumerate(zip(s, big))]

    def heat(self, f, W):
        _, U, _ = self.prim(W)
        q = torch.zeros((self.C, self.D), dtype=torch.float64, device="cuda")
        for ks in self.slices(self.C):
            c = [self.u[ks, d] - U[:, d, None] for d in range(self.D)]
            e = sum(x * x for x in c) * f[:, 0, ks] + (f[:, 1, ks] if self.NC == 2 else 0.0)
            for d in range(self.D):
                q[:, d] += 0.5 * (c[d] * e) @ self.w[ks]
        return q

    def slices(self, rows):
        n = max(1, 24_000_000 // max(rows, 1))
        return [slice(k, min(self.Nv, k + n)) for k in range(0, self.Nv, n)]

    def equilibrium(self, W, Wg, q):
        """Per face: g0 (rho, U, T), its heat flux, its slopes in the basis centred at U0, q1..q5."""
        D, M = self.D, self.M
        rho, U, T = self.prim(torch.cat([W, Wg]))
        P = torch.cat([rho[:, None], U, T[:, None]], 1)
        g = self.lsq(P, slice(None))                   # columns: rho, U, T
        gW = []
        for d in range(D):
            dr, dU, dT = g[d][:, :1], g[d][:, 1:-1], g[d][:, -1:]
            Pc, Uc = P[:self.C], P[:self.C, 1:-1]
            gW.append(torch.cat([dr, Uc * dr + Pc[:, :1] * dU,
                                 dr * (0.5 * (Uc * Uc).sum(1, keepdim=True) + 1.5 * Pc[:, -1:])
                                 + Pc[:, :1] * ((Uc * dU).sum(1, keepdim=True) + 1.5 * dT)], 1))

        def side(c, r):
            s = P[c] + sum(g[d][c] * r[:, d, None] for d in range(D))
            return torch.where((s[:, :1] > 0) & (s[:, -1:] > 0), s, P[c])

        L, R, two = self.L, torch.where(self.two[:, 0], self.R, 0), self.two
        sL, sR = side(L, self.rL), torch.where(two, side(R, self.rR), P[self.R])
        dW = [0.5 * (gW[d][L] + torch.where(two, gW[d][R], 0.0)) for d in range(D)]
        q0 = 0.5 * (q[L] + torch.where(two, q[R], 0.0))
        W0 = torch.zeros((self.F, M), dtype=torch.float64, device="cuda")
        for ks in self.slices(self.F):
            un = self.n @ self.u[ks].T
            h = b = 0.0
            for s, on in ((sL, (un > 0) + 0.5 * (un == 0)), (sR, (un < 0) + 0.5 * (un == 0))):
                H = on * self.maxwell(s[:, 0], s[:, 1:-1], s[:, -1], ks)[0]
                h, b = h + H, b + s[:, -1:] * H
            uw = torch.cat([self.w[ks, None], self.w[ks, None] * self.u[ks],
                            0.5 * self.w[ks, None] * (self.u[ks] ** 2).sum(1, keepdim=True)], 1)
            W0 += h @ uw
            if self.NC == 2:
                W0[:, -1] += 0.5 * b @ self.w[ks]
        # walls carry no equilibrium: any positive state keeps their rows finite
        W0 = torch.where((self.R == self.L)[:, None], W[self.L], W0)
        rho0, U0, T0 = self.prim(W0)
        nb, xb = self.nxi * T0, self.nxi * (self.nxi + 2.0) * T0 * T0
        A = torch.zeros((self.F, M, M), dtype=torch.float64, device="cuda")
        B = torch.zeros((D, self.F, M, M), dtype=torch.float64, device="cuda")
        for ks in self.slices(4 * self.F):
            H, c, c2 = self.maxwell(rho0, U0, T0, ks)
            H = H * self.w[ks]
            v = torch.stack([torch.ones_like(c2)] + c + [0.5 * (c2 + nb[:, None])], 1)
            A += (v * H[:, None]) @ v.transpose(1, 2)
            ex = 0.25 * (xb - nb * nb)
            A[:, -1, -1] += ex * H.sum(1)
            for d in range(D):
                Hu = H * self.u[ks, d]
                B[d] += (v * Hu[:, None]) @ v.transpose(1, 2)
                B[d][:, -1, -1] += ex * Hu.sum(1)
        rhs = []
        for g0 in dW:
            rhs.append(torch.cat([g0[:, :1], g0[:, 1:-1] - U0 * g0[:, :1],
                                  g0[:, -1:] - (U0 * g0[:, 1:-1]).sum(1, keepdim=True)
                                  + 0.5 * (U0 * U0).sum(1, keepdim=True) * g0[:, :1]], 1))
        beta = torch.linalg.solve(A, torch.stack(rhs, 2))               # [F][M][D]
        bA = torch.linalg.solve(A, -sum((B[d] @ beta[:, :, d, None]) for d in range(D)))[:, :, 0]
        return rho0, U0, T0, q0, beta, bA, self.integrals(self.tau(rho0, T0))

    def step(self, f, W, q):
        D, C, NC, dt = self.D, self.C, self.NC, self.dt
        Wg = W[self.L[self.far]]
        if len(self.far):
            Wg = torch.where(self.inflow, self.Winf, Wg)
        rho0, U0, T0, q0, beta, bA, qs = self.equilibrium(W, Wg, q)
        nb, xb = self.nxi * T0, self.nxi * (self.nxi + 2.0) * T0 * T0
        rg, Ug, Tg = self.prim(Wg)

        def extended(ks):
            G = self.comps(self.maxwell(rg, Ug, Tg, ks)[0], Tg)
            return [torch.cat([f[:, m, ks], G[m]]) for m in range(NC)]

        wc = self.L[self.wall]                          # wall density: zero net mass flux
        num, den = 0.0, 0.0
        for ks in self.slices(max(len(wc), C // 8)) if len(wc) else []:
            V = extended(ks)
            g = self.micro(V[0], wc, ks)
            un = self.n[self.wall] @ self.u[ks].T
            hin = V[0][wc] + sum(g[d] * self.rL[self.wall][:, d, None] for d in range(D))
            ug = sum(self.u[ks, d] * g[d] for d in range(D))
            num = num + (torch.clamp(un, min=0.0) * (hin - 0.5 * dt * ug)) @ self.w[ks]
            Hw = self.maxwell(torch.ones_like(self.Tw), self.Uw, self.Tw, ks)[0]
            den = den + (torch.clamp(un, max=0.0) * Hw) @ self.w[ks]
        rho, U, T = self.prim(W)
        cc = (0.5 * dt / self.tau(rho, T))[:, None]
        fn, dWc = torch.empty_like(f), torch.zeros_like(W)
        for ks in self.slices(self.F):
            V = extended(ks)
            un = self.n @ self.u[ks].T
            up, F = un > 0, []
            H, c, c2 = self.maxwell(rho0, U0, T0, ks)
            lam0 = 0.5 / T0
            kap = (4.0 * (1.0 - self.p["Pr"]) * lam0 * lam0 / (5.0 * rho0))[:, None]
            kqc, l2 = kap * sum(q0[:, d, None] * c[d] for d in range(D)), 2.0 * lam0[:, None] * c2
            R = torch.where(self.two[:, 0], self.R, 0)
            for m in range(NC):
                g = self.micro(V[m], slice(None), ks)
                vL = V[m][self.L] + sum(g[d][self.L] * self.rL[:, d, None] for d in range(D))
                vR = V[m][self.R] + sum(torch.where(self.two, g[d][R], 0.0) * self.rR[:, d, None] for d in range(D))
                ugL = sum(self.u[ks, d] * g[d][self.L] for d in range(D))
                ugR = sum(self.u[ks, d] * torch.where(self.two, g[d][R], 0.0) for d in range(D))
                Hm, ex = (H, nb) if m == 0 else (nb[:, None] * H, xb)

                def slope(b):                           # int (xi^2) (b.psi_c) g0 over the internal dof
                    poly = b[:, :1] + sum(b[:, 1 + d, None] * c[d] for d in range(D)) + 0.5 * b[:, -1:] * c2
                    return poly * Hm + 0.5 * b[:, -1:] * ex[:, None] * H

                eq = qs[2][:, None] * Hm * (1.0 + kqc * (l2 - D - (2 if m == 0 else 0)))
                for d in range(D):
                    eq = eq + qs[3][:, None] * self.u[ks, d] * slope(beta[:, :, d])
                eq = eq + qs[4][:, None] * slope(bA)
                Fm = un * (qs[0][:, None] * torch.where(up, vL, vR) + qs[1][:, None] * torch.where(up, ugL, ugR) + eq)
                if len(wc):
                    Hw = self.comps(self.maxwell(-num / den, self.Uw, self.Tw, ks)[0], self.Tw)[m]
                    out = dt * vL[self.wall] - 0.5 * dt * dt * ugL[self.wall]
                    Fm[self.wall] = un[self.wall] * torch.where(up[self.wall], out, dt * Hw)
                F.append(Fm)
            plus = self.fplus(rho, U, T, q, ks)[0]
            res = []
            for m in range(NC):
                r = sum(self.cs[:, e, None] * F[m][self.face[:, e]] for e in range(self.face.shape[1]))
                fn[:, m, ks] = f[:, m, ks] + r + cc * (plus[m] - f[:, m, ks])
                res.append(r)
            hw = res[0] * self.w[ks]
            dWc[:, 0] += hw.sum(1)
            dWc[:, 1:-1] += hw @ self.u[ks]
            dWc[:, -1] += 0.5 * hw @ (self.u[ks] ** 2).sum(1)
            if NC == 2:
                dWc[:, -1] += 0.5 * res[1] @ self.w[ks]
        W = W + dWc
        rho, U, T = self.prim(W)
        cc = (0.5 * dt / self.tau(rho, T))[:, None]
        for ks in self.slices(C):
            plus = self.fplus(rho, U, T, q, ks)[0]
            for m in range(NC):
                fn[:, m, ks] = (fn[:, m, ks] + cc * plus[m]) / (1.0 + cc)
        return fn, W, self.heat(fn, W)


def exact(case, seed):
    """The pass in 64 bits from the same (stored) state."""
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    out = []
    for setup, s in zip(_setups(case), _seeds(case, seed)):
        f, W = _state(setup, dtype, s)
        p = _Plain(setup)
        f = f.double()
        q = p.heat(f, W)
        for _ in range(case["steps"]):
            f, W, q = p.step(f, W, q)
        out.append({"f": f.reshape(p.C, -1), "W": W, "q": q})
        del p
    return out
