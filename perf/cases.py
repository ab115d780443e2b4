"""Performance cases of the FVLBM time step: what a program that uses this package has it do.

Each case is one pass of such a program over state that it already holds (a solver on a mesh,
a batch of solvers, host buffers): a run of time steps and the state after it, a state that is
sent up, stepped and read back, a gradient of the wall forces, or their tangent.  The sizes are
those of the meshes that ``meshgen`` stands for: 64 x 64 and 10k-40k-triangle cavities, the
80k-cell backward-facing step, the 50k-200k-cell airfoil, the 48-instance sweep.

``exact`` restates the same equations in 64-bit torch operations (cell-wise gathers, automatic
differentiation for the gradients) and shares no code with the library.
"""
from __future__ import annotations

import ctypes
import dataclasses
import functools
import math

import numpy as np
import torch

from paper_1812_00394_gb300 import fvlbm, meshgen as mg

PREC = {"fp32": fvlbm.FVLBM_FP32_DEV, "fp64": fvlbm.FVLBM_FP64, "tangent": fvlbm.FVLBM_FP64_TANGENT}


# ------------------------------------------------------------------------------- the cases
def _step(mesh, cells, precision, steps, **more):
    return {"kind": "step", "mesh": mesh, "cells": cells, "precision": precision, "steps": steps,
            "scheme": 0, "local_dt": False, "tune": False, "re": 1000.0, "alpha": 4.0} | more


def listed():
    return [
        # the smallest run in use: the plain 64 x 64 cavity in 64 bits, between two looks at it
        _step("quad", 4096, "fp64", 20, re=400.0) | {"name": "cavity64_fp64"},
        # one small instance of the sweep alone, in the fast precision: launches count
        _step("delaunay", 10000, "fp32", 40, re=400.0) | {"name": "cavity10k_fp32"},
        # the 40k-triangle cavity run to a steady state
        _step("delaunay", 40000, "fp32", 40) | {"name": "cavity40k_fp32"},
        # the comparison scheme on the same mesh
        _step("delaunay", 40000, "fp32", 40, scheme=1, cfl=0.2, re=400.0) | {"name": "cavity40k_euler_fp32"},
        # the turbulent backward-facing step
        _step("bfs", 80000, "fp32", 20) | {"name": "step80k_sst_fp32"},
        # the airfoil at its full size, steady state with local steps
        _step("naca", 200000, "fp32", 20, local_dt=True) | {"name": "airfoil200k_sst_local_fp32"},
        # the airfoil in 64 bits, as the gradients and the accuracy checks run it
        _step("naca", 50000, "fp64", 5) | {"name": "airfoil50k_sst_fp64"},
        # the uneven sweep in one batch: the headline workload
        _step("sweep", 2571456, "fp32", 10, n_cavity=32, n_bfs=4, n_naca=12) | {"name": "sweep48_fp32"},
        # a part of the sweep in 64 bits on the kernels that the tuner picks
        _step("sweep", 640000, "fp64", 3, n_cavity=8, n_bfs=1, n_naca=3, tune=True) | {"name": "sweep12_fp64"},
        # a coupled program: the batch's state goes up, takes a step and comes back
        {"kind": "roundtrip", "mesh": "sweep", "cells": 640000, "precision": "fp32", "n_cavity": 8, "n_bfs": 1,
         "n_naca": 3, "steps": 1, "scheme": 0, "name": "roundtrip12_fp32"},
        # shape and inflow gradients of drag and lift, reverse mode
        {"kind": "adjoint", "mesh": "naca", "cells": 50000, "steps": 10, "sst": True, "re": 6e6, "alpha": 4.0,
         "shape": True, "name": "airfoil50k_adjoint"},
        # two parameter directions in forward mode
        {"kind": "tangent", "mesh": "naca", "cells": 20000, "steps": 3, "sst": True, "re": 6e6, "alpha": 2.0,
         "directions": 2, "name": "airfoil20k_tangent"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step"] * 7 + ["roundtrip", "adjoint", "tangent"])
    if kind == "step":
        mesh = rng.choice(["quad", "delaunay", "delaunay", "bfs", "naca", "naca", "sweep"])
        prec = rng.choice(["fp32", "fp32", "fp64"])
        if mesh == "sweep":
            n = rng.randint(2, 12)
            parts = {"n_cavity": n, "n_bfs": rng.randint(0, 2), "n_naca": rng.randint(0, 3)}
            return _step("sweep", 0, prec, rng.randint(2, 5), tune=prec == "fp64", **parts)
        scheme = rng.choice([0, 0, 0, 1]) if mesh in ("quad", "delaunay") else 0
        cells = _log(rng, 1000, 200000 if prec == "fp32" else 60000)
        more = {"scheme": 1, "cfl": 0.1} if scheme else {"local_dt": rng.random() < 0.25, "cfl": 0.5}
        re = float(_log(rng, 100, 400 if scheme else 3200))   # the explicit scheme needs dt < 2 tau
        return _step(mesh, cells, prec, rng.randint(3, 40 if prec == "fp32" else 12), re=re,
                     alpha=round(rng.uniform(0.0, 12.0), 2), tune=prec == "fp64" and rng.random() < 0.5, **more)
    if kind == "roundtrip":
        return {"kind": kind, "mesh": "sweep", "cells": 0, "precision": "fp32", "n_cavity": rng.randint(1, 12),
                "n_bfs": rng.randint(0, 1), "n_naca": rng.randint(0, 3), "steps": rng.randint(1, 4), "scheme": 0}
    sst = rng.random() < 0.7
    more = {"mesh": "naca", "cells": _log(rng, 2000, 50000 if kind == "adjoint" else 20000), "sst": sst,
            "re": 6e6 if sst else 2000.0, "alpha": round(rng.uniform(0.0, 12.0), 2)}
    if kind == "adjoint":
        return {"kind": kind, "steps": rng.randint(2, 10), "shape": rng.random() < 0.5} | more
    return {"kind": kind, "steps": rng.randint(1, 3), "directions": rng.randint(1, 2)} | more


# ------------------------------------------------------------------------------ the inputs
@functools.lru_cache(maxsize=24)
def _meshes(key):
    """The meshes of a case with the parameters that do not depend on the seed."""
    c = dict(key)
    n, cfl = int(c["cells"]), float(c.get("cfl", 0.5))
    if c["mesh"] == "quad":
        out = [mg.cavity_quad(max(8, round(math.sqrt(n))), re=c["re"], cfl=cfl)]
    elif c["mesh"] == "delaunay":
        out = [mg.cavity_delaunay(h_boundary=1.0 / max(8, round(math.sqrt(n))), n_target=n, re=c["re"], cfl=cfl)]
    elif c["mesh"] == "bfs":
        out = [mg.bfs_hybrid(n_target=n, cfl=cfl)]
    elif c["mesh"] == "naca":
        out = [mg.naca0012_cmesh(n_target=n, alpha_deg=c["alpha"], cfl=cfl,
                                 re_c=c["re"] if c["kind"] in ("adjoint", "tangent") else 6e6)]
    else:
        out = mg.batched_sweep(n_cavity=c["n_cavity"], n_bfs=c["n_bfs"], n_naca=c["n_naca"])
    if not c.get("sst", True):
        out = [dataclasses.replace(x, sst=False) for x in out]
    return [dataclasses.replace(x, local_dt=bool(c.get("local_dt", False))) for x in out]


def _modes(rng, x, y, n=6):
    """A smooth random field of about unit size."""
    s = np.zeros_like(x)
    for _ in range(n):
        a, b = rng.integers(1, 5, 2)
        s += rng.normal() * np.sin(2.1 * a * x + 6.28 * rng.random()) * np.sin(2.1 * b * y + 6.28 * rng.random())
    return s / math.sqrt(n / 4.0)


def _flow(case, rng):
    """The case with a flow under way in it: vortices in a cavity; a wall layer, disturbances and a
    turbulence field with its wall behaviour around the step and the airfoil; noise from cell to cell."""
    m = case.mesh
    ptr = m.cell_ptr.astype(np.int64)
    num = np.diff(ptr)
    x, y = (np.add.reduceat(m.xy[m.cell_nodes, c], ptr[:-1]) / num for c in (0, 1))
    n, U = m.n_cells, case.uref
    name = case.name
    if name.startswith("bfs"):
        H = float(m.xy[:, 1].max())
        d = np.minimum(H - y, np.where(x < 0.0, y - 1.0, y))
        d = np.where((x >= 0.0) & (y < 1.0), np.minimum(d, x), d)
        ub, vb, width = U * np.tanh(d / 0.3) * np.where(y > 1.0, 1.0, 0.1), np.zeros(n), 0.3
    elif name.startswith("naca"):
        d = np.hypot(np.maximum(np.maximum(-x, x - 1.0), 0.0), y)
        a = math.radians(case.alpha_deg)
        ub, vb, width = U * math.cos(a) * np.tanh(d / 0.1), U * math.sin(a) * np.tanh(d / 0.1), 0.1
    else:
        d = np.minimum(np.minimum(x, 1.0 - x), np.minimum(y, 1.0 - y))
        ub, vb, width = np.zeros(n), np.zeros(n), 0.1
    near = np.tanh(d / width)
    u = ub + 0.1 * U * near * _modes(rng, x, y) + 1e-4 * U * rng.uniform(-1, 1, n)
    v = vb + 0.1 * U * near * _modes(rng, x, y) + 1e-4 * U * rng.uniform(-1, 1, n)
    rho = 1.0 + 1e-3 * _modes(rng, x, y) + 1e-6 * rng.uniform(-1, 1, n)
    more = {}
    if case.sst:
        k = case.k * np.exp(0.3 * _modes(rng, x, y)) * (0.1 + 0.9 * near ** 2) * (1 + 1e-3 * rng.uniform(-1, 1, n))
        w = case.omega * np.exp(0.2 * _modes(rng, x, y)) + 6.0 * case.nu / (0.075 * (d + 1e-3 * width) ** 2)
        more = {"k": k, "omega": w * (1 + 1e-3 * rng.uniform(-1, 1, n))}
    return dataclasses.replace(case, rho=rho, u=u, v=v, **more)


def _cases(case, seed):
    rng = np.random.default_rng(seed)
    key = tuple(sorted((k, v) for k, v in case.items() if k != "name"))
    return [_flow(c, rng) for c in _meshes(key)]


def _seeds(case, c, seed):
    """The input derivatives of the tangent directions: the angle of attack, then a smooth bump of the mesh."""
    m = c.mesh
    a = math.radians(c.alpha_deg)
    far = (m.bedge_type == mg.BC_FARFIELD).astype(float)
    db = np.zeros((m.n_bedges, 5))
    db[:, 1], db[:, 2] = -c.uref * math.sin(a) * far, c.uref * math.cos(a) * far
    out = [{"dbedge_val": db, "dalpha": 1.0}]
    x0 = np.random.default_rng(seed).uniform(0.2, 0.8)
    bump = np.exp(-((m.xy[:, 0] - x0) ** 2 + m.xy[:, 1] ** 2) / 0.02)
    out.append({"dxy": np.stack([0.0 * bump, bump], 1), "dalpha": 0.0})
    return out[:case["directions"]]


@functools.lru_cache(maxsize=1)
def _stream():
    """The one stream of the program: its solvers take their turns on it."""
    torch.cuda.init()
    return torch.cuda.Stream()


def prepare(case, seed):
    cs = _cases(case, seed)
    st = _stream()
    kind, prec = case["kind"], case.get("precision", "fp64")
    if kind == "tangent":
        s = fvlbm.Solver(cs * case["directions"], precision=PREC["tangent"], stream=st.cuda_stream)
        dirs = _seeds(case, cs[0], seed)
        for i, d in enumerate(dirs):
            if "dxy" in d:
                s.tangent_seed_nodes(d["dxy"], i=i)
            else:
                s.tangent_seed(d["dbedge_val"], i=i)
        return {"case": case, "solver": s, "stream": st, "dirs": dirs}
    s = fvlbm.Solver(cs if len(cs) > 1 else cs[0], precision=PREC[prec], stream=st.cuda_stream,
                     scheme=case.get("scheme", 0))
    out = {"case": case, "solver": s, "stream": st}
    if case.get("tune"):
        s.autotune(3)
    if kind == "step":
        n = sum(s.cells)
        out["lists"] = [s.set_exchange_list(np.arange(s.cells[i]), i) for i in range(s.n)]
        w = [4.0 / 9.0] + [1.0 / 9.0] * 4 + [1.0 / 36.0] * 4
        with torch.cuda.stream(st):
            out["rows"] = torch.empty((n, 12), dtype=torch.float64, device="cuda")
            out["rest"] = torch.tensor(w, dtype=torch.float64, device="cuda") * cs[0].rho0
    elif kind == "roundtrip":
        n = sum(s.cells)
        out["up"] = torch.empty((n, 9), dtype=torch.float32, pin_memory=True)
        out["down"] = torch.empty((n, 9), dtype=torch.float32, pin_memory=True)
        _fdev(s, out["up"])
    torch.cuda.synchronize()
    return out


def _fdev(s, to):
    rc = fvlbm.load().fvlbm_get_fdev_f32(s.h, -1, ctypes.c_void_p(to.data_ptr()))
    if rc:
        raise fvlbm.FvlbmError(rc, "fvlbm_get_fdev_f32")
    return to


# --------------------------------------------------------------------------------- a pass
def run(state):
    case, s = state["case"], state["solver"]
    kind = case["kind"]
    if kind == "step":
        # the steps, then the state in the caller's cell order on the device: f less its rest
        # value, k, omega and nu_t (in the precision that the solver holds)
        s.step(case["steps"])
        at = 0
        for i, lid in enumerate(state["lists"]):
            s.pack_cells_dev(lid, state["rows"][at:].data_ptr())
            at += s.cells[i]
        with torch.cuda.stream(state["stream"]):
            f, turb = state["rows"][:, :9] - state["rest"], state["rows"][:, 9:]
            if case["precision"] == "fp32":
                f, turb = f.float(), turb.float()
            else:
                turb = turb.clone()
        return {"f": f, "k": turb[:, 0], "omega": turb[:, 1], "nut": turb[:, 2]}
    if kind == "roundtrip":
        rc = fvlbm.load().fvlbm_set_fdev_f32_async(s.h, -1, ctypes.c_void_p(state["up"].data_ptr()))
        if rc:
            raise fvlbm.FvlbmError(rc, "fvlbm_set_fdev_f32_async")
        s.step(case["steps"])
        return {"f": _fdev(s, state["down"])}
    if kind == "adjoint":
        J, df, db, dxy = s.adjoint(case["steps"], 1.0, 0.5, shape=case["shape"])
        return {"J": J, "df": df, "db": db} | ({"dxy": dxy} if case["shape"] else {})
    s.step(case["steps"])
    out = {}
    for i, d in enumerate(state["dirs"]):
        val, grad = s.forces_tangent(i, d["dalpha"])
        out["df%d" % i] = s.get_f_tangent(i)
        out["force%d" % i] = np.array([val["fx"], val["fy"], grad["fx"], grad["fy"], grad["cd"], grad["cl"]])
    return out


def work(case):
    """The mesh and the state read once and the state written once per step (a state larger than the
    caches passes through memory at every step), and the operations of the step's formulas: per stage
    and cell the differences to 3.5 neighbours in 8 directions, 4 upwind values a face from them, the
    flux sums and the collision; the SST about half of a stage.  The gradients cost their forward
    steps once more in each of their two sweeps."""
    cs = _meshes(tuple(sorted((k, v) for k, v in case.items() if k != "name")))
    cells = sum(c.mesh.n_cells for c in cs)
    sst = sum(c.mesh.n_cells for c in cs if c.sst)
    word = 4 if case.get("precision") == "fp32" else 8
    stages = 1 if case.get("scheme") == 1 else 3
    flops = (cells * (300.0 * stages + (80 if stages == 3 else 0)) + sst * 250.0) * case["steps"]
    byte = (cells * ((9 + 9 + 1 + 8) * word + 14.0) + sst * 6.0 * word) * case["steps"]
    if case["kind"] == "roundtrip":
        byte += 2 * 9 * 4.0 * cells
    if case["kind"] == "adjoint":
        flops, byte = 3 * flops, 3 * byte
    if case["kind"] == "tangent":
        flops, byte = 3 * flops * case["directions"], 2 * byte * case["directions"]
    return {"bytes": byte, "flops": flops}


# --------------------------------------------------------- the same equations in 64 bits
_EX = [0.0, 1.0, 0.0, -1.0, 0.0, 1.0, -1.0, -1.0, 1.0]
_EY = [0.0, 0.0, 1.0, 0.0, -1.0, 1.0, 1.0, -1.0, -1.0]
_W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


class _Exact:
    """One instance: the discrete equations on [cells, faces, directions] tensors.  ``xy`` and ``bval``
    may carry derivatives."""

    def __init__(self, c, dev, xy=None, bval=None):
        m = c.mesh
        t = lambda a, k=torch.float64: torch.as_tensor(np.ascontiguousarray(a), dtype=k, device=dev)  # noqa: E731
        self.c, self.dev = c, dev
        self.e = t(np.array([_EX, _EY]))
        self.w = t(np.array(_W))
        self.xy = t(m.xy) if xy is None else xy
        self.bval = t(m.bedge_val) if bval is None else bval
        self.bkind = t(m.bedge_type, torch.int64)
        ptr = m.cell_ptr.astype(np.int64)
        num = np.diff(ptr)
        N = self.N = len(num)
        nodes = np.zeros((N, 4), np.int64)
        nodes[:, :3] = m.cell_nodes[ptr[:-1, None] + np.arange(3)]
        nodes[:, 3] = np.where(num == 4, m.cell_nodes[np.minimum(ptr[:-1] + 3, len(m.cell_nodes) - 1)], nodes[:, 0])
        ends = np.roll(nodes, -1, 1)
        ends[num == 3, 2] = nodes[num == 3, 0]
        has = np.ones((N, 4), bool)
        has[:, 3] = num == 4
        # partners by sorted node pairs; what is left over is a boundary edge
        key = (np.minimum(nodes, ends) * (m.n_nodes + 1) + np.maximum(nodes, ends))[has]
        cell, slot = np.nonzero(has)
        bn = m.bedge_nodes.astype(np.int64)
        bkey = bn.min(1) * (m.n_nodes + 1) + bn.max(1)
        order = np.argsort(key, kind="stable")
        ks = key[order]
        pair = np.nonzero(ks[1:] == ks[:-1])[0]
        nbr = np.full((N, 4), -1, np.int64)
        a, b = order[pair], order[pair + 1]
        nbr[cell[a], slot[a]] = cell[b]
        nbr[cell[b], slot[b]] = cell[a]
        single = has & (nbr < 0)
        border = np.argsort(bkey)
        skey = (np.minimum(nodes, ends) * (m.n_nodes + 1) + np.maximum(nodes, ends))[single]
        eid = border[np.searchsorted(bkey[border], skey)]
        sc, ss = np.nonzero(single)
        idx = np.where(has, nbr, np.arange(N)[:, None])
        idx[sc, ss] = N + eid
        owner = np.zeros(m.n_bedges, np.int64)
        owner[eid] = sc
        self.has, self.idx, self.owner = t(has, torch.bool), t(idx, torch.int64), t(owner, torch.int64)
        self.inner = t(nbr >= 0, torch.bool)
        self.nb = torch.where(self.inner, self.idx, torch.zeros_like(self.idx))
        mask = self.has.double()[..., None]
        # geometry, relative to the first node of the cell
        nd, en = t(nodes, torch.int64), t(ends, torch.int64)
        p, q = self.xy[nd] - self.xy[nd[:, :1]], self.xy[en] - self.xy[nd[:, :1]]
        cross = (p[..., 0] * q[..., 1] - q[..., 0] * p[..., 1]) * mask[..., 0]
        area = self.area = 0.5 * cross.sum(1)
        rel = ((p + q) * cross[..., None]).sum(1) / (6.0 * area[:, None])
        mid = 0.5 * (p + q) - rel[:, None]                       # face midpoint from the centroid
        cen = self.xy[nd[:, 0]] + rel
        edge = (q - p) * mask
        self.sn = torch.stack([edge[..., 1], -edge[..., 0]], -1) / area[:, None, None]  # n dl / A
        d = torch.where(self.inner[..., None], cen[self.nb] - cen[:, None], mid) * mask
        M = (d[..., :, None] * d[..., None, :]).sum(1)
        det = M[:, 0, 0] * M[:, 1, 1] - M[:, 0, 1] ** 2
        inv = torch.stack([torch.stack([M[:, 1, 1], -M[:, 0, 1]], -1), torch.stack([-M[:, 0, 1], M[:, 0, 0]], -1)], 1)
        self.lsq = torch.einsum("ncd,nmd->nmc", inv / det[:, None, None], d)
        self.r = mid * mask
        self.rn = (mid - d) * mask                               # from the neighbour's centroid
        self.dist = torch.where(self.has, (d * d).sum(-1), torch.ones_like(d[..., 0])).sqrt()
        self.en = self.sn @ self.e                               # [N, 4, 9]
        rate = torch.clamp(self.en.detach(), min=0.0).sum(1).amax(1)
        if c.local_dt:
            self.dt = (c.cfl / rate)[:, None]
        else:
            self.dt = torch.tensor(c.dt, dtype=torch.float64, device=dev) if c.dt > 0 else c.cfl / rate.max()
        bnd = (bn, self.xy[t(bn, torch.int64)])
        tang = bnd[1][:, 1] - bnd[1][:, 0]
        nrm = torch.stack([tang[:, 1], -tang[:, 0]], -1)
        out = ((0.5 * (bnd[1][:, 1] + bnd[1][:, 0]) - cen[self.owner]) * nrm).sum(-1).detach()
        self.bn = torch.where(out[:, None] < 0, -nrm, nrm)       # n dl, out of the fluid
        if c.sst:
            self.wall_distance(cen, bnd[1][self.bkind == mg.BC_WALL])

    def wall_distance(self, cen, seg):
        a, b = seg[:, 0], seg[:, 1]

        def dist(x, a, b):
            s = (((x - a) * (b - a)).sum(-1) / ((b - a) ** 2).sum(-1)).clamp(0.0, 1.0)
            return ((a + s[..., None] * (b - a) - x) ** 2).sum(-1).sqrt()

        near = [dist(x[:, None], a[None], b[None]).argmin(1) for x in cen.detach().split(4096)]
        near = torch.cat(near)
        self.wd = dist(cen, a[near], b[near])

    # ---- f^eq, moments and boundary values
    def feq(self, rho, u):
        eu = u @ self.e
        return self.w * rho[:, None] * (1.0 + 3.0 * eu + 4.5 * eu * eu - 1.5 * (u * u).sum(1, keepdim=True))

    def macros(self, f):
        rho = f.sum(1)
        return rho, (f @ self.e.T) / rho[:, None]

    def bvalues(self, f):
        fP, v, kind = f[self.owner], self.bval, self.bkind[:, None]
        rho, u = self.macros(fP)
        neq = fP - self.feq(rho, u)
        far = torch.where(self.bn.detach() @ self.e < 0.0, self.feq(v[:, 0], v[:, 1:3]), fP)
        out = torch.where(kind == mg.BC_OUTLET, self.feq(v[:, 0], u) + neq, self.feq(rho, v[:, 1:3]) + neq)
        return torch.where(kind == mg.BC_FARFIELD, far, out)

    def gradient(self, f, fb):
        d = torch.cat([f, fb])[self.idx] - f[:, None]
        return torch.einsum("nmc,nma->nca", self.lsq, d)

    def convection(self, f):
        fb = self.bvalues(f)
        g = self.gradient(f, fb)
        own = f[:, None] + torch.einsum("nmc,nca->nma", self.r, g)
        nbr = f[self.nb] + torch.einsum("nmc,nmca->nma", self.rn, g[self.nb])
        face = torch.where(self.en >= 0.0, own, nbr)
        face = torch.where(self.inner[..., None], face, torch.cat([f, fb])[self.idx])
        return -(self.en * face).sum(1)

    def step(self, f, turb, scheme):
        c, dt = self.c, self.dt
        if c.sst:
            turb = self.sst(f, turb)
            tau = (3.0 * (c.nu + turb[2]))[:, None]
        else:
            tau = torch.tensor(3.0 * c.nu, dtype=torch.float64, device=self.dev)
        if scheme == 1:
            return f + dt * (self.convection(f) + (self.feq(*self.macros(f)) - f) / tau), turb
        z = dt / tau

        def relax(x, rhs, s):
            eq = self.feq(*self.macros(x))
            fj = (rhs + s * z * eq) / (1.0 + s * z)
            return fj, (s * z * eq - s * z * rhs) / (1.0 + s * z) / s      # f^(J), dt Gamma^c(J)

        f1, c1 = relax(f, f, 0.25)
        a1 = dt * self.convection(f1)
        x2 = f + 0.5 * a1
        f2, c2 = relax(x2, x2, 0.25)
        a2 = dt * self.convection(f2)
        x3 = x2 + 0.5 * a2
        f3, c3 = relax(x3, x3 + (c1 + c2) / 3.0, 1.0 / 3.0)
        a3 = dt * self.convection(f3)
        return f + (a1 + a2 + a3 + c1 + c2 + c3) / 3.0, turb

    # ---- the k-omega SST transport step
    def sst(self, f, turb):
        c = self.c
        k, w, nut = turb
        nu, dt, d = c.nu, (self.dt[:, 0] if c.local_dt else self.dt), self.wd
        a1, bs, kap = 0.31, 0.09, 0.41
        sk1, sw1, b1, sk2, sw2, b2 = 0.85, 0.5, 0.075, 1.0, 0.856, 0.0828
        _, u = self.macros(f)
        phi = torch.cat([u, k[:, None], w[:, None]], 1)
        v, kind, o = self.bval, self.bkind[:, None], self.owner
        wall = torch.stack([v[:, 1], v[:, 2], 0.0 * v[:, 1], 60.0 * nu / (b1 * d[o] ** 2)], 1)
        pb = torch.where(kind == mg.BC_WALL, wall, torch.where(kind == mg.BC_OUTLET, phi[o], v[:, 1:5]))
        q = torch.cat([phi, pb])[self.idx]                       # [N, 4, 4]
        g = torch.einsum("nmc,nma->nac", self.lsq, q - phi[:, None])
        kw = phi[:, 2:]
        inc = torch.einsum("nac,nmc->nma", g[:, 2:], self.r)     # increments to the faces
        hi, lo = torch.maximum(q[..., 2:].amax(1), kw), torch.minimum(q[..., 2:].amin(1), kw)
        safe = torch.where(inc == 0.0, torch.ones_like(inc), inc)
        ratio = torch.where(inc > 0, (hi - kw)[:, None] / safe, torch.where(inc < 0, (lo - kw)[:, None] / safe,
                                                                            torch.ones_like(inc)))
        lim = torch.clamp(torch.where(self.has[..., None], ratio, torch.ones_like(ratio)).amin(1), max=1.0)
        gl = g[:, 2:] * lim[..., None]
        s11, s22, s12 = g[:, 0, 0], g[:, 1, 1], 0.5 * (g[:, 0, 1] + g[:, 1, 0])
        SS, div = s11 ** 2 + s22 ** 2 + 2.0 * s12 ** 2, s11 + s22
        gg = (g[:, 2] * g[:, 3]).sum(1)
        cd = torch.clamp(2.0 * sw2 / w * gg, min=1e-20)
        arg1 = torch.minimum(torch.maximum(k.sqrt() / (bs * w * d), 500.0 * nu / (w * d * d)),
                             4.0 * sw2 * k / (cd * d * d))
        f1 = torch.tanh(arg1 ** 4)
        sig = torch.stack([f1 * sk1 + (1 - f1) * sk2, f1 * sw1 + (1 - f1) * sw2], 1)
        own = kw[:, None] + torch.einsum("nac,nmc->nma", gl, self.r)
        nbr = kw[self.nb] + torch.einsum("nmac,nmc->nma", gl[self.nb], self.rn)
        inner = self.inner[..., None]
        uf = torch.where(inner, 0.5 * (u[:, None] + q[..., :2]), q[..., :2])
        un = (uf * self.sn).sum(-1, keepdim=True)
        up = torch.where(un >= 0.0, own, torch.where(inner, nbr, q[..., 2:]))
        gam = nu + sig * nut[:, None]
        gam = torch.where(inner, 0.5 * (gam[:, None] + gam[self.nb]), gam[:, None])
        dl = torch.where(self.has, (self.sn ** 2).sum(-1), torch.ones_like(self.dist)).sqrt() * self.has
        diff = gam * (q[..., 2:] - kw[:, None]) * (dl / self.dist)[..., None]
        R = (diff - un * up).sum(1)
        gamma = f1 * (b1 / bs - sw1 * kap * kap / 0.3) + (1 - f1) * (b2 / bs - sw2 * kap * kap / 0.3)
        shear = 2.0 * SS - 2.0 / 3.0 * div * div
        ok = nut > 0
        pk = nut * shear - 2.0 / 3.0 * k * div
        pw = gamma * shear - torch.where(ok, 2.0 / 3.0 * gamma * k * div / torch.where(ok, nut, torch.ones_like(nut)),
                                         torch.zeros_like(nut))
        cross = 2.0 * (1 - f1) * sw2 / w * gg
        beta = f1 * b1 + (1 - f1) * b2
        k1 = torch.clamp((k + dt * (R[:, 0] + pk)) / (1 + dt * bs * w), min=0.0)
        w1 = torch.clamp((w + dt * (R[:, 1] + pw + cross)) / (1 + dt * beta * w), min=1e-12 * c.uref / c.lref)
        pos = k1 > 0
        root = torch.where(pos, torch.where(pos, k1, torch.ones_like(k1)).sqrt(), torch.zeros_like(k1))
        arg2 = torch.maximum(2.0 * root / (bs * w1 * d), 500.0 * nu / (w1 * d * d))
        nut1 = a1 * k1 / torch.maximum(a1 * w1, (2.0 * SS).sqrt() * torch.tanh(arg2 ** 2))
        return k1, w1, nut1

    def start(self):
        c = self.c
        t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=self.dev)  # noqa: E731
        f = self.feq(t(c.rho), torch.stack([t(c.u), t(c.v)], 1))
        k, w = (t(c.k), t(c.omega)) if c.sst else (torch.zeros_like(f[:, 0]), torch.ones_like(f[:, 0]))
        return f, (k, w, k / w if c.sst else torch.zeros_like(k))

    def force(self, f):
        fb = self.bvalues(f)
        m = ((self.bn @ self.e) * fb) @ self.e.T
        return m[self.bkind == mg.BC_WALL].sum(0)

    def coefficients(self, F, a):
        c = self.c
        s = 0.5 * c.rho0 * c.uref ** 2 * c.lref
        ca, sa = torch.cos(a), torch.sin(a)
        return (F[0] * ca + F[1] * sa) / s, (-F[0] * sa + F[1] * ca) / s


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    cs = _cases(case, seed)
    kind = case["kind"]
    if kind in ("step", "roundtrip"):
        out = {"f": [], "k": [], "omega": [], "nut": []}
        with torch.no_grad():
            for c in cs:
                X = _Exact(c, dev)
                f, turb = X.start()
                for _ in range(case["steps"]):
                    f, turb = X.step(f, turb, case["scheme"])
                for k, v in zip(out, (f - X.w * c.rho0,) + tuple(turb)):
                    out[k].append(v)
        out = {k: torch.cat(v) for k, v in out.items()}
        return {"f": out["f"].cpu()} if kind == "roundtrip" else out
    c = cs[0]
    angle = torch.tensor(math.radians(c.alpha_deg), dtype=torch.float64, device=dev)
    if kind == "adjoint":
        xy = torch.tensor(c.mesh.xy, dtype=torch.float64, device=dev, requires_grad=case["shape"])
        bval = torch.tensor(c.mesh.bedge_val, dtype=torch.float64, device=dev, requires_grad=True)
        X = _Exact(c, dev, xy, bval)
        f0, turb = X.start()
        f0 = f0.detach().requires_grad_(True)
        f = f0
        for _ in range(case["steps"]):
            f, turb = X.step(f, turb, 0)
        cd, cl = X.coefficients(X.force(f), angle)
        J = cd + 0.5 * cl
        g = torch.autograd.grad(J, [f0, bval] + ([xy] if case["shape"] else []))
        out = {"J": float(J.detach()), "df": g[0].cpu().numpy(), "db": g[1].cpu().numpy()}
        return out | ({"dxy": g[2].cpu().numpy()} if case["shape"] else {})
    out = {}
    with torch.no_grad(), torch.autograd.forward_ad.dual_level():
        fwd = torch.autograd.forward_ad
        for i, d in enumerate(_seeds(case, c, seed)):
            pairs = []
            for base, dot in ((c.mesh.xy, d.get("dxy")), (c.mesh.bedge_val, d.get("dbedge_val"))):
                base = torch.tensor(base, dtype=torch.float64, device=dev)
                dot = torch.zeros_like(base) if dot is None else torch.tensor(dot, dtype=torch.float64, device=dev)
                pairs.append(fwd.make_dual(base, dot))
            a = fwd.make_dual(angle, torch.full_like(angle, d["dalpha"]))
            X = _Exact(c, dev, *pairs)
            f, turb = X.start()
            for _ in range(case["steps"]):
                f, turb = X.step(f, turb, 0)
            F = X.force(f)
            tangents = [fwd.unpack_dual(v).tangent for v in (f, F) + X.coefficients(F, a)]
            out["df%d" % i] = tangents[0].cpu().numpy()
            Fp = fwd.unpack_dual(F).primal
            out["force%d" % i] = np.array([float(v) for v in (Fp[0], Fp[1], tangents[1][0], tangents[1][1],
                                                              tangents[2], tangents[3])])
    return out
