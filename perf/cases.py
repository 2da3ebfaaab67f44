"""What users of the HDG shallow-water solver have it do, as timed cases.

A case is one pass through the public calls of ``paper_2004_09389_gb300``:

* ``step``    one implicit step of a time loop on device tensors: ``solve_dev``, then ``recover_dev`` of its solution;
* ``host``    the same step for a program whose fields are NumPy arrays: ``solve_recover``;
* ``retime``  a step after a change of the time step: ``set_tau`` (which rebuilds the operators), solve, recover;
* ``imex``    one ARS2(2,3,2) step of the IMEX time loop: two stage solves, two recoveries, the stage rates;
* ``batch``   many uneven problems in one merged batch: ``MergedBatch.solve_dev``;
* ``local``   what a program with a Krylov method of its own calls: ``condensed_rhs_dev``, ``trace_apply_dev`` and
  ``recover_dev`` with explicit right-hand side and trace.

Meshes, degrees, Courant numbers and depths are those of the benchmark and of the tests: the doubly periodic square
with 20 km cells (256 x 256 x 2 is the benchmark's 5,120 km square) or the unit square of the small configuration, and
the icosahedral sphere of the Earth's radius.  Right-hand sides are random smooth fields with a k^-3 power spectrum.

``exact`` discretises the same equations once more in plain 64-bit torch (cell systems by batched LU, the trace system
by GMRES to round-off), from the mesh arrays alone.
"""
from __future__ import annotations

import functools
import math
from fractions import Fraction

import numpy as np
import torch

import hdg_inputs as I
from paper_2004_09389_gb300 import (HDG_FP64, HDG_MIXED_BF16, HDG_MIXED_FGMRES64, HDG_MIXED_FP32, HDGSolver,
                                    MergedBatch)

PRECISION = {"fp64": HDG_FP64, "mixed": HDG_MIXED_FP32, "bf16": HDG_MIXED_BF16, "fgmres64": HDG_MIXED_FGMRES64}
RADIUS, OMEGA, GRAVITY = 6.371e6, 7.292e-5, 9.81


# ---------------------------------------------------------------------------------------------------------- the cases

def listed():
    # the benchmark solves to 1e-8; loops and ensembles here to 1e-10, as the small configuration and the tests do
    flat = {"mesh": "flat", "depth": 1000.0, "courant": 8.0, "rtol": 1e-10}
    sphere = {"mesh": "sphere", "depth": 8185.0, "courant": 8.0, "rtol": 1e-10}
    bench = {**flat, "rtol": 1e-8}
    return [
        # the smallest call: the 512-cell unit square, plain FP64, to 1e-10 (latency and launches count)
        {"name": "step_unit16_p1_fp64", "kind": "step", "mesh": "unit", "size": 16, "p": 1, "precision": "fp64",
         "depth": 1.0, "courant": 8.0, "rtol": 1e-10},
        # the benchmark's headline step: 131,072 cells, mixed precision
        {"name": "step_flat256_p3_mixed", "kind": "step", **bench, "size": 256, "p": 3, "precision": "mixed"},
        # the same step as a user who wants plain FP64 throughout takes it
        {"name": "step_flat256_p3_fp64", "kind": "step", **bench, "size": 256, "p": 3, "precision": "fp64"},
        # the largest mesh: the r = 7 sphere (327,680 cells), f varying over every cell
        {"name": "step_sphere7_p2_mixed", "kind": "step", **sphere, "size": 7, "p": 2, "precision": "mixed"},
        # the highest degree, on a mesh whose sizes are no powers of two, with the BF16 smoother copy
        {"name": "step_flat100_p4_bf16", "kind": "step", **flat, "size": 100, "p": 4, "precision": "bf16"},
        # FP64 Krylov space with the FP32 V-cycle, the lowest degree, a mid-sized sphere
        {"name": "step_sphere5_p1_fgmres64", "kind": "step", **sphere, "size": 5, "p": 1, "precision": "fgmres64"},
        # a model that keeps its fields in (pageable) host memory
        {"name": "host_flat144_p2_mixed", "kind": "host", **flat, "size": 144, "p": 2, "precision": "mixed"},
        # adaptive time step: the operators are rebuilt before the step, mixed precision on the sphere ...
        {"name": "retime_sphere5_p3_mixed", "kind": "retime", **sphere, "size": 5, "p": 3, "precision": "mixed"},
        # ... and plain FP64 on a flat mesh
        {"name": "retime_flat96_p2_fp64", "kind": "retime", **flat, "size": 96, "p": 2, "precision": "fp64"},
        # the time loop of the benchmark's IMEX workload (r = 6, p = 3)
        {"name": "imex_sphere6_p3_mixed", "kind": "imex", **sphere, "size": 6, "p": 3, "precision": "mixed"},
        # an ensemble of uneven problems solved together (flat 16..128, sphere r = 3..5, p = 1..3, Courant 4..16)
        {"name": "batch16_mixed", "kind": "batch", "count": 16, "largest": 128, "pick": 1, "precision": "mixed",
         "rtol": 1e-10},
        # a program with its own Krylov method: condensed right-hand side, one operator application, recovery
        {"name": "local_sphere6_p3_fp64", "kind": "local", **sphere, "size": 6, "p": 3, "precision": "fp64"},
    ]


_MOST_WORK = 131072 * 30.0 ** 2     # cells x (unknowns per cell)^2 of the largest drawn mesh


def draw(rng):
    kind = rng.choice(["step", "step", "step", "host", "retime", "imex", "batch", "local"])
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(3, 16), "largest": rng.choice([32, 48, 64, 96, 128]),
                "pick": rng.randint(2, 10 ** 6), "precision": rng.choice(["mixed", "mixed", "bf16"]), "rtol": 1e-10}
    while True:
        on_sphere = kind == "imex" or rng.random() < 0.4
        p = rng.randint(1, 3 if on_sphere else 4)
        if on_sphere:
            size = rng.randint(3, 6)
            cells = 20 * 4 ** size
        else:
            # log-uniform 12..256 with nested coarse levels down to a grid of at most 32 x 32
            k = round(2.0 ** rng.uniform(math.log2(3.0), 6.0))
            size = 4 * (k if k <= 32 else 2 * round(k / 2))
            cells = 2 * size * size
        if cells * (1.5 * (p + 1) * (p + 2)) ** 2 <= _MOST_WORK:
            break
    precision = rng.choice(["mixed", "mixed", "fp64", "fp64", "bf16", "fgmres64"])
    if kind == "imex":
        precision = rng.choice(["mixed", "fp64"])
    elif kind == "local":
        precision = rng.choice(["fp64", "fgmres64"])     # a caller's own Krylov method runs in FP64
    return {"kind": kind, "mesh": "sphere" if on_sphere else "flat", "size": size, "p": p, "precision": precision,
            "depth": round(rng.uniform(5e3, 1e4), 1) if on_sphere else 1000.0,
            "courant": round(2.0 ** rng.uniform(2.0, 3.0 if on_sphere else 4.0), 2), "rtol": 1e-10}


def _problems(case):
    """The problems of a batch case, the choice made by its ``pick`` alone."""
    rng = np.random.default_rng(int(case["pick"]))
    flats = [n for n in (16, 24, 32, 48, 64, 96, 128) if n <= case["largest"]]
    spheres = [3, 4, 5] if case["largest"] >= 64 else [3, 4]
    out = []
    for i in range(case["count"]):
        on_sphere = i % 2 == 1
        out.append({"kind": "step", "mesh": "sphere" if on_sphere else "flat",
                    "size": int(rng.choice(spheres if on_sphere else flats)), "p": int(rng.integers(1, 4)),
                    "precision": case["precision"], "depth": float(rng.uniform(5e3, 1e4)) if on_sphere else 1000.0,
                    "courant": float(4.0 * 2.0 ** rng.uniform(0, 2)), "rtol": case["rtol"]})
    return out


# ------------------------------------------------------------------------------------------------- meshes and inputs

@functools.lru_cache(maxsize=None)
def _mesh(kind, size):
    if kind == "sphere":
        return I.sphere_hierarchy(size, RADIUS, r_coarsest=max(1, size - 5))
    return I.periodic_square_hierarchy(size, side=1.0 if kind == "unit" else 2.0e4 * size, n_coarsest=4)


class _Setting:
    """Physical parameters of a case: g, H, tau, the Coriolis values and the smoother that suits them."""

    def __init__(self, case):
        self.mesh = _mesh(case["mesh"], case["size"])
        self.p, self.H = case["p"], case["depth"]
        self.g = 1.0 if case["mesh"] == "unit" else GRAVITY
        self.tau = case["courant"] * self.mesh.h / math.sqrt(self.g * self.H)
        if case["mesh"] == "sphere":
            self.f = I.coriolis_sphere(self.mesh, OMEGA)
        else:
            self.f = I.coriolis_flat(self.mesh, 1.0 if case["mesh"] == "unit" else 1e-4)
        # strong rotation needs the Chebyshev smoother (damped block-Jacobi diverges there)
        self.smoother = 1 if float(np.abs(self.f).max()) * self.tau > 1.5 else 0


def _device(seed):
    gen = torch.Generator().manual_seed(int(seed))
    return torch.device("cuda"), gen


def _waves(mesh, points, gen, fields, count=192):
    """Random smooth fields [fields, ...] at the points [..., dim]: waves whose wave numbers are log-uniform up to 64
    per side (or radius), amplitudes as for a k^-3 power spectrum, unit RMS."""
    dev, dim = points.device, points.shape[-1]
    k = 2.0 ** (torch.rand(fields, count, 1, generator=gen, dtype=torch.float64) * 6.0)
    d = torch.randn(fields, count, dim, generator=gen, dtype=torch.float64)
    d = k * d / d.norm(dim=-1, keepdim=True)
    amp = torch.randn(fields, count, generator=gen, dtype=torch.float64) * k[..., 0] ** -1.0
    phase = torch.rand(fields, count, generator=gen, dtype=torch.float64) * (2.0 * math.pi)
    if mesh.dim == 2:
        d = torch.round(d) * (2.0 * math.pi / mesh.side)     # whole wave numbers: periodic
    else:
        d = d / mesh.radius
    x = points.reshape(-1, dim)
    out = torch.zeros(fields, x.shape[0], dtype=torch.float64, device=dev)
    for f in range(fields):
        df, af, pf = d[f].to(dev), amp[f].to(dev), phase[f].to(dev)
        for a in range(0, x.shape[0], 1 << 18):
            out[f, a:a + (1 << 18)] = torch.cos(x[a:a + (1 << 18)] @ df.T + pf) @ af
    out = out / out.square().mean(dim=1, keepdim=True).sqrt()
    return out.reshape(fields, *points.shape[:-1])


@functools.lru_cache(maxsize=None)
def _geometry(kind, size):
    """From the mesh arrays alone, on the GPU: cell vertices [N,3,dim], the cells' 2-D coordinates [N,3,2], the sphere
    cells' frames, facet ids in order of first appearance, and the edges that run from the higher to the lower id."""
    mesh = _mesh(kind, size)
    x = np.asarray(mesh.vertex_xyz)[mesh.cell_vertices]
    if mesh.cell_shift is not None:
        x = x + mesh.cell_shift
    if mesh.dim == 2:
        flat, frames = x, None
    else:
        d1, d2 = x[:, 1] - x[:, 0], x[:, 2] - x[:, 0]
        e1 = d1 / np.linalg.norm(d1, axis=1, keepdims=True)
        n = np.cross(d1, d2)
        n /= np.linalg.norm(n, axis=1, keepdims=True)
        e2 = np.cross(n, e1)
        frames = np.stack([e1, e2], axis=1)
        flat = np.einsum("kvd,kcd->kvc", x - x[:, :1], frames)
    cv = np.asarray(mesh.cell_vertices, np.int64)
    a, b = cv[:, [1, 2, 0]].ravel(), cv[:, [2, 0, 1]].ravel()
    key = np.minimum(a, b) * mesh.n_vertices + np.maximum(a, b)
    _, first, inverse = np.unique(key, return_index=True, return_inverse=True)
    rank = np.empty(first.size, np.int64)
    order = np.argsort(first)
    rank[order] = np.arange(first.size)
    facet = rank[inverse.ravel()].reshape(-1, 3)
    dev = torch.device("cuda")
    up = lambda v, t=torch.float64: None if v is None else torch.as_tensor(v, dtype=t, device=dev)  # noqa: E731
    return {"x": up(x), "flat": up(flat), "frames": up(frames), "facet": up(facet, torch.int64),
            "flip": up((a > b).reshape(-1, 3), torch.bool), "n_facets": int(first.size),
            "first": up(first[order], torch.int64), "cells": up(cv, torch.int64)}


def _nodes(p):
    return [(a, b) for b in range(p + 1) for a in range(p + 1 - b)]


def _cell_points(geo, p):
    ab = torch.tensor(_nodes(p), dtype=torch.float64, device=geo["x"].device) / p
    x = geo["x"]
    return (x[:, None, 0] + ab[None, :, 0:1] * (x[:, None, 1] - x[:, None, 0])
            + ab[None, :, 1:2] * (x[:, None, 2] - x[:, None, 0]))


def _state_fields(case, gen):
    """Nodal velocity [N,2,n_p] and height [N,n_p] of a random smooth state."""
    geo, mesh = _geometry(case["mesh"], case["size"]), _mesh(case["mesh"], case["size"])
    points = _cell_points(geo, case["p"])
    if mesh.dim == 2:
        w = _waves(mesh, points, gen, 3)
        u, h = w[:2].permute(1, 0, 2), w[2]
    else:
        w = _waves(mesh, points, gen, 4)
        u, h = torch.einsum("dkp,kcd->kcp", w[:3], geo["frames"]), w[3]
    return u.contiguous(), h.contiguous()


def _trace_field(case, gen):
    """A random smooth trace [n_facets, p+1], nodes from the lower to the higher vertex id."""
    geo, mesh, p = _geometry(case["mesh"], case["size"]), _mesh(case["mesh"], case["size"]), case["p"]
    t = torch.linspace(0.0, 1.0, p + 1, dtype=torch.float64, device=geo["x"].device)
    a, b = geo["x"][:, [1, 2, 0]], geo["x"][:, [2, 0, 1]]
    lo = torch.where(geo["flip"][..., None], b, a)
    hi = torch.where(geo["flip"][..., None], a, b)
    pts = (lo[..., None, :] + t[:, None] * (hi - lo)[..., None, :]).reshape(-1, p + 1, mesh.dim)
    return _waves(mesh, pts[geo["first"]], gen, 1)[0].contiguous()


def _solver(case, **more):
    s = _Setting(case)
    more = {"f_vertex": s.f, "smoother": s.smoother, **more}
    return HDGSolver(s.mesh, s.p, more.pop("tau", s.tau), s.g, s.H, precision=PRECISION[case["precision"]],
                     rtol=case["rtol"], **more)


def _gamma():
    return 1.0 - 1.0 / math.sqrt(2.0)


def prepare(case, seed):
    dev, gen = _device(seed)
    kind = case["kind"]
    if kind == "batch":
        solvers, ru, rh, lam = [], [], [], []
        for q in _problems(case):
            s = _solver(q, keep_rhs=0)
            u, h = _state_fields(q, gen)
            solvers.append(s)
            ru.append(u)
            rh.append(h)
            lam.append(torch.empty(s.n_facets, q["p"] + 1, dtype=torch.float64, device=dev))
        return {"kind": kind, "batch": MergedBatch(solvers), "ru": ru, "rh": rh, "lam": lam}
    ru, rh = _state_fields(case, gen)
    if case["mesh"] == "unit":      # noisy data, as the small configuration has
        ru = ru + 1e-3 * torch.randn(ru.shape, generator=gen, dtype=torch.float64).to(dev)
    if kind == "imex":
        st = _Setting(case)
        solver = _solver(case, f_vertex=None, smoother=0, tau=_gamma() * st.tau)
        solver.imex_init(st.f)
        return {"kind": kind, "solver": solver, "dt": st.tau, "u0": ru, "h0": rh, "u": torch.empty_like(ru),
                "h": torch.empty_like(rh)}
    solver = _solver(case)
    if kind == "host":
        return {"kind": kind, "solver": solver, "ru": ru.cpu().numpy(), "rh": rh.cpu().numpy()}
    state = {"kind": kind, "solver": solver, "kept": case["precision"] in ("mixed", "bf16"), "ru": ru, "rh": rh,
             "u": torch.empty_like(ru), "h": torch.empty_like(rh),
             "lam": torch.empty(solver.n_facets, case["p"] + 1, dtype=torch.float64, device=dev)}
    if kind == "retime":
        state["tau"] = _Setting(case).tau
    if kind == "local":
        state["lam"] = _trace_field(case, gen)
        state["g"], state["y"] = torch.empty_like(state["lam"]), torch.empty_like(state["lam"])
    return state


def run(state):
    kind = state["kind"]
    if kind == "batch":
        state["batch"].solve_dev(state["ru"], state["rh"], state["lam"])
        return list(state["lam"])
    s = state["solver"]
    if kind == "host":
        lam, u, h, _ = s.solve_recover(state["ru"], state["rh"])
        return {"lam": lam, "u": u, "h": h}
    if kind == "imex":
        state["u"].copy_(state["u0"])
        state["h"].copy_(state["h0"])
        s.imex_step_dev("ARS2", state["dt"], state["u"], state["h"])
        return {"u": state["u"], "h": state["h"]}
    if kind == "local":
        s.condensed_rhs_dev(state["ru"], state["rh"], state["g"])
        s.trace_apply_dev(state["lam"], state["y"])
        s.recover_dev(state["ru"], state["rh"], state["lam"], state["u"], state["h"])
        return {"g": state["g"], "y": state["y"], "u": state["u"], "h": state["h"]}
    if kind == "retime":
        s.set_tau(state["tau"])
    s.solve_dev(state["ru"], state["rh"], state["lam"])
    # the two-float modes recover from what the solve kept, the FP64 ones take the right-hand side again
    s.recover_dev(*((None, None) if state["kept"] else (state["ru"], state["rh"])), None, state["u"], state["h"])
    return {"lam": state["lam"], "u": state["u"], "h": state["h"]}


# --------------------------------------------------------------------------------------------- the work of one pass

def work(case):
    """Inputs and outputs once, the assembled trace operator once (8 bytes an entry, 4 in the modes whose V-cycle is
    FP32 or below); the flops of eleven V-cycle-preconditioned Krylov iterations of five operator applications each
    (the counts of these problems), and of the cell solves by their n_p x n_p Schur complements."""
    if case["kind"] == "batch":
        each = [work(q) for q in _problems(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    p, mesh = case["p"], case["mesh"]
    n = 20 * 4 ** case["size"] if mesh == "sphere" else 2 * case["size"] ** 2
    npn, pp, facets = (p + 1) * (p + 2) // 2, p + 1, 3 * n // 2
    fields, trace = 8.0 * 3 * npn * n, 8.0 * pp * facets
    operator = (8.0 if case["precision"] == "fp64" else 4.0) * 5 * pp * pp * facets
    apply = 2.0 * 5 * pp * pp * facets
    cell = 2.0 * n * (9 * npn * npn + 3 * pp * 3 * pp)
    kind = case["kind"]
    if kind == "local":
        return {"bytes": 2 * fields + 3 * trace + 2 * operator, "flops": apply + 2 * cell}
    solves = 2 if kind == "imex" else 1
    flops = solves * (11 * 5 * apply + 2 * cell)
    bytes_ = 2 * fields + operator + (0.0 if kind == "imex" else trace)
    if kind == "retime":
        flops += 2.0 * n * (npn ** 3 + 3 * npn * npn * 3 * pp + 9 * pp * pp * 3 * pp)
        bytes_ += operator
    return {"bytes": bytes_, "flops": flops}


# ------------------------------------------------------------------------------------------- the same in plain 64 bits

@functools.lru_cache(maxsize=None)
def _reference(p):
    """Reference matrices of the triangle (0,0),(1,0),(0,1) in exact rational arithmetic, as float64 on the GPU."""
    nodes, exps = _nodes(p), [(a, b) for s in range(p + 1) for a in range(s, -1, -1) for b in [s - a]]
    n = len(nodes)
    V = [[Fraction(x, p) ** a * Fraction(y, p) ** b for a, b in exps] for x, y in nodes]
    A = [row[:] + [Fraction(int(i == j)) for j in range(n)] for i, row in enumerate(V)]
    for k in range(n):
        piv = next(r for r in range(k, n) if A[r][k] != 0)
        A[k], A[piv] = A[piv], A[k]
        inv = 1 / A[k][k]
        A[k] = [v * inv for v in A[k]]
        for r in range(n):
            if r != k and A[r][k] != 0:
                f = A[r][k]
                A[r] = [v - f * w for v, w in zip(A[r], A[k])]
    coef = np.array([[A[j][n + i] for j in range(n)] for i in range(n)], dtype=object)   # node i: sum_j coef[i,j] x^a y^b
    fact = math.factorial

    def tri(a, b):
        return Fraction(fact(a) * fact(b), fact(a + b + 2))

    def over(weight):
        return coef.dot(np.array([[weight(e, f) for f in exps] for e in exps], dtype=object)).dot(coef.T)

    M = over(lambda e, f: tri(e[0] + f[0], e[1] + f[1]))
    L1 = over(lambda e, f: tri(e[0] + f[0] + 1, e[1] + f[1]))
    L2 = over(lambda e, f: tri(e[0] + f[0], e[1] + f[1] + 1))
    Dx = over(lambda e, f: f[0] * tri(e[0] + f[0] - 1, e[1] + f[1]) if f[0] else Fraction(0))
    Dy = over(lambda e, f: f[1] * tri(e[0] + f[0], e[1] + f[1] - 1) if f[1] else Fraction(0))
    # one-dimensional trace basis: equispaced Lagrange polynomials of degree p as coefficient lists
    line = []
    for j in range(p + 1):
        c = [Fraction(1)]
        for k in range(p + 1):
            if k != j:
                d = Fraction(j - k, p)
                c = [(c[i - 1] / d if i else 0) - (c[i] * Fraction(k, p) / d if i < len(c) else 0)
                     for i in range(len(c) + 1)]
        line.append(c)
    M1 = np.array([[sum(a * b / (i + j + 1) for i, a in enumerate(f) for j, b in enumerate(g)) for g in line]
                   for f in line], dtype=object)
    # the cell nodes on each edge i, from vertex i + 1 to vertex i + 2, as a 0/1 map [3][n][p+1]
    at = {ab: i for i, ab in enumerate(nodes)}
    edge = np.zeros((3, n, p + 1))
    for j in range(p + 1):
        edge[0, at[(p - j, j)], j] = 1
        edge[1, at[(0, p - j)], j] = 1
        edge[2, at[(j, 0)], j] = 1
    up = lambda v: torch.as_tensor(np.asarray(v, dtype=np.float64), device="cuda")  # noqa: E731
    return {"M": up(M), "L": torch.stack([up(M - L1 - L2), up(L1), up(L2)]), "Dx": up(Dx), "Dy": up(Dy), "M1": up(M1),
            "N": up(edge) @ up(M1), "edge": up(edge)}


class _Exact:
    """The upwind HDG system of one mesh in 64 bits."""

    def __init__(self, mesh_kind, size, p, tau, g, H, f):
        self.geo, self.ref, self.p = _geometry(mesh_kind, size), _reference(p), p
        self.tau, self.g, self.H, self.ts = tau, g, H, math.sqrt(g * H)
        X, R = self.geo["flat"], self.ref
        J = torch.stack([X[:, 1] - X[:, 0], X[:, 2] - X[:, 0]], dim=2)
        self.det = J[:, 0, 0] * J[:, 1, 1] - J[:, 0, 1] * J[:, 1, 0]
        inv = torch.stack([torch.stack([J[:, 1, 1], -J[:, 0, 1]], 1), torch.stack([-J[:, 1, 0], J[:, 0, 0]], 1)], 1)
        inv = inv / self.det[:, None, None]                                       # [ref, xy]
        t = X[:, [2, 0, 1]] - X[:, [1, 2, 0]]
        self.len = t.norm(dim=2)
        self.nrm = torch.stack([t[..., 1], -t[..., 0]], dim=2)                    # outward, times the edge length
        sc = lambda v, m: v[:, None, None] * m  # noqa: E731
        self.M = sc(self.det, R["M"])
        self.D = [sc(self.det * inv[:, 0, c], R["Dx"]) + sc(self.det * inv[:, 1, c], R["Dy"]) for c in (0, 1)]
        self.F = torch.einsum("ki,iab->kab", self.det[:, None] * f[self.geo["cells"]], R["L"])
        self.N = [torch.einsum("ki,ibj->kbij", self.nrm[..., c], R["N"]).flatten(2) for c in (0, 1)]
        self.N.append(torch.einsum("ki,ibj->kbij", self.len, R["N"]).flatten(2))  # [k][b][(i, j)]
        E = torch.einsum("ibj,iaj->iab", R["edge"], R["N"])
        self.E = torch.einsum("ki,iab->kab", self.len, E)
        i, j = torch.arange(3, device=X.device), torch.arange(p + 1, device=X.device)
        jj = torch.where(self.geo["flip"][..., None], p - j, j)
        self.dof = (self.geo["facet"][..., None] * (p + 1) + jj).flatten(1)       # [k][(i, j)]
        self.nt = self.geo["n_facets"] * (p + 1)
        self.C = torch.cat([H * self.N[0], H * self.N[1], self.ts * self.N[2]], dim=1).mT

    def condense(self):
        tau, g, H, ts = self.tau, self.g, self.H, self.ts
        row = lambda *b: torch.cat(b, dim=2)  # noqa: E731
        A = torch.cat([row(self.M, -tau * self.F, -tau * g * self.D[0].mT), row(tau * self.F, self.M, -tau * g * self.D[1].mT),
                       row(tau * H * self.D[0], tau * H * self.D[1], self.M + tau * ts * self.E)], dim=1)
        B = torch.cat([tau * g * self.N[0], tau * g * self.N[1], -tau * ts * self.N[2]], dim=1)
        self.lu = torch.linalg.lu_factor(A)
        self.X = torch.linalg.lu_solve(*self.lu, B)
        S = self.C @ self.X
        k = self.p + 1
        for i in range(3):
            S[:, i * k:(i + 1) * k, i * k:(i + 1) * k] += ts * self.len[:, i, None, None] * self.ref["M1"]
        self.S = S
        D = torch.zeros(self.geo["n_facets"], k, k, dtype=torch.float64, device=S.device)
        for i in range(3):
            blk = S[:, i * k:(i + 1) * k, i * k:(i + 1) * k]
            blk = torch.where(self.geo["flip"][:, i, None, None], blk.flip(1, 2), blk)
            D.index_add_(0, self.geo["facet"][:, i], blk)
        self.Dinv = torch.linalg.inv(D)
        return self

    def gather(self, y):
        return torch.zeros(self.nt, dtype=torch.float64, device=y.device).index_add_(0, self.dof.flatten(), y.flatten())

    def apply(self, x):
        return self.gather((self.S @ x[self.dof][..., None])[..., 0])

    def jacobi(self, r):
        return (self.Dinv @ r.view(-1, self.p + 1, 1)).flatten()

    def local(self, ru, rh):
        """A^-1 M r per cell, [N][3 n_p]."""
        r = torch.cat([ru, rh[:, None]], dim=1) @ self.M.mT
        return torch.linalg.lu_solve(*self.lu, r.flatten(1)[..., None])[..., 0]

    def rhs(self, z):
        return self.gather((self.C @ z[..., None])[..., 0])

    def recover(self, z, lam):
        q = z - (self.X @ lam[self.dof][..., None])[..., 0]
        n = q.shape[1] // 3
        return q[:, :2 * n].reshape(-1, 2, n), q[:, 2 * n:]

    def solve(self, b, m=400):
        """GMRES (block-Jacobi from the right, Gram-Schmidt twice), restarted until the residual stops falling."""
        x, last = torch.zeros_like(b), math.inf
        for _ in range(8):
            r = b - self.apply(x)
            beta = float(r.norm())
            if beta <= 2e-15 * float(b.norm()) or beta > 0.2 * last:
                break
            last = beta
            V = torch.empty(m + 1, self.nt, dtype=torch.float64, device=b.device)
            V[0] = r / beta
            Hm, cols = np.zeros((m + 1, m)), 0
            R, cs, sn, s = np.zeros((m + 1, m)), [], [], np.zeros(m + 1)
            s[0] = beta
            for j in range(m):
                w = self.apply(self.jacobi(V[j]))
                h = V[:j + 1] @ w
                w = w - V[:j + 1].T @ h
                h2 = V[:j + 1] @ w
                w = w - V[:j + 1].T @ h2
                nw = w.norm()
                col = torch.cat([h + h2, nw[None]]).cpu().numpy()
                Hm[:j + 2, j] = col
                V[j + 1] = w / nw
                for i in range(j):
                    col[i], col[i + 1] = cs[i] * col[i] + sn[i] * col[i + 1], -sn[i] * col[i] + cs[i] * col[i + 1]
                d = math.hypot(col[j], col[j + 1])
                cs.append(col[j] / d)
                sn.append(col[j + 1] / d)
                R[:j + 1, j] = col[:j + 1]
                R[j, j] = d
                s[j], s[j + 1] = cs[j] * s[j], -sn[j] * s[j]
                cols = j + 1
                if abs(s[j + 1]) < 1e-12 * beta or abs(s[j + 1]) < 1e-15 * float(b.norm()):
                    break
            y = np.linalg.solve(np.triu(R[:cols, :cols]), s[:cols])
            x = x + self.jacobi(V[:cols].T @ torch.as_tensor(y, device=b.device))
            del V
        return x

    def step(self, ru, rh):
        z = self.local(ru, rh)
        lam = self.solve(self.rhs(z))
        return (lam, *self.recover(z, lam))

    def rates(self, u, h, f):
        """(M^-1 N(q), M^-1 L(q)): explicit Coriolis and the gravity waves with the upwind trace of the state."""
        n, k = h.shape[1], self.p + 1
        on_edge = torch.einsum("kb,ibj->kij", h, self.ref["edge"])
        un = torch.einsum("kcb,ibj,kic->kij", u, self.ref["edge"], self.nrm / self.len[..., None])
        lam = self.gather(0.5 * on_edge + self.H / (2.0 * self.ts) * un)[self.dof]                   # [k][(i, j)]
        mv = lambda m, v: (m @ v[..., None])[..., 0]  # noqa: E731
        lu = [self.g * (mv(self.D[c].mT, h) - mv(self.N[c], lam)) for c in (0, 1)]
        jump = mv(self.E, h) - mv(self.N[2], lam)
        lh = -self.H * (mv(self.D[0], u[:, 0]) + mv(self.D[1], u[:, 1])) - self.ts * jump
        F = torch.einsum("ki,iab->kab", self.det[:, None] * f[self.geo["cells"]], self.ref["L"])
        minv = torch.linalg.inv(self.ref["M"])
        inv = lambda v: v @ minv.mT / self.det[:, None]  # noqa: E731
        nu = torch.stack([inv(mv(F, u[:, 1])), -inv(mv(F, u[:, 0]))], dim=1)
        return nu, torch.stack([inv(v) for v in lu], dim=1), inv(lh)


def _exact_of(case, f=None, tau=None):
    s = _Setting(case)
    f = torch.as_tensor(s.f if f is None else f, dtype=torch.float64, device="cuda")
    return _Exact(case["mesh"], case["size"], case["p"], s.tau if tau is None else tau, s.g, s.H, f).condense()


def exact(case, seed):
    dev, gen = _device(seed)
    kind = case["kind"]
    if kind == "batch":
        out = []
        for q in _problems(case):
            u, h = _state_fields(q, gen)
            out.append(_exact_of(q).step(u, h)[0].view(-1, q["p"] + 1))
        return out
    ru, rh = _state_fields(case, gen)
    if case["mesh"] == "unit":
        ru = ru + 1e-3 * torch.randn(ru.shape, generator=gen, dtype=torch.float64).to(dev)
    k = case["p"] + 1
    if kind == "imex":
        st = _Setting(case)
        dt, g = st.tau, _gamma()
        d = -2.0 * math.sqrt(2.0) / 3.0
        f = torch.as_tensor(st.f, dtype=torch.float64, device=dev)
        ex = _exact_of(case, f=np.zeros_like(st.f), tau=g * dt)
        n1, _, _ = ex.rates(ru, rh, f)
        _, u, h = ex.step(ru + dt * g * n1, rh)
        n2, lu2, lh2 = ex.rates(u, h, f)
        _, u, h = ex.step(ru + dt * (d * n1 + (1 - d) * n2 + (1 - g) * lu2), rh + dt * (1 - g) * lh2)
        n3, lu3, lh3 = ex.rates(u, h, f)
        return {"u": ru + dt * ((1 - g) * (n2 + lu2) + g * (n3 + lu3)), "h": rh + dt * ((1 - g) * lh2 + g * lh3)}
    ex = _exact_of(case)
    if kind == "local":
        lam = _trace_field(case, gen)
        z = ex.local(ru, rh)
        u, h = ex.recover(z, lam.flatten())
        return {"g": ex.rhs(z).view(-1, k), "y": ex.apply(lam.flatten()).view(-1, k), "u": u, "h": h}
    lam, u, h = ex.step(ru, rh)
    return {"lam": lam.view(-1, k), "u": u, "h": h}
