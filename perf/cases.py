"""The work that users of the multigrid solver have it do, as cases to time and compare.

A case is a mesh or point cloud, a system on it and one call sequence of the public entry points
(`paper_2307_04886_gb300`).  The surface and its prolongation hierarchy are what a program keeps from one call to
the next, so they are fixed by the case's sizes; the right-hand sides, initial values, matrix values and diffusion
times that it passes in come from the seed.
"""
from __future__ import annotations

import functools
import math
import random

import numpy as np
import torch

import gmg_inputs
import paper_2307_04886_gb300 as gmg
from paper_2307_04886_gb300.autograd import smooth
from gmg_inputs import meshes, operators

PRECISION = {"fp64": gmg.GMG_FP64, "fp32_refine": gmg.GMG_FP32_REFINE, "fp32_pcg": gmg.GMG_FP32_PCG,
             "fp64_pcg": gmg.GMG_FP64_PCG}


def listed():
    return [
        # the smallest call: smoothing on a mesh of a few thousand vertices, where launches and latency are all
        {"name": "solve_sphere_2562", "call": "solve", "surface": "sphere", "level": 4, "t": 1e-3,
         "precision": "fp32_pcg", "tol": 1e-10},
        # the paper's own iteration, FP64 V-cycles, on its usual small mesh (10,242 vertices)
        {"name": "solve_sphere_10242_fp64", "call": "solve", "surface": "sphere", "level": 5, "t": 1e-3,
         "precision": "fp64", "tol": 1e-10},
        # a mid-size mesh with the default options (FP32 cycles in FP64 refinement); no size is a multiple of 32
        {"name": "solve_torus_250x122_refine", "call": "solve", "surface": "torus", "a": 250, "b": 122, "t": 1e-4,
         "precision": "fp32_refine", "tol": 1e-10},
        # bi-Laplacian smoothing: 19 entries per row on the finest level
        {"name": "solve_bilaplacian_256x120", "call": "solve", "surface": "bilaplacian", "a": 256, "b": 120,
         "t": 1e-3, "precision": "fp32_pcg", "tol": 1e-10},
        # smoothing on a non-manifold mesh, 149,200 vertices
        {"name": "solve_book_5x150x200", "call": "solve", "surface": "book", "pages": 5, "a": 150, "b": 200,
         "t": 1e-3, "precision": "fp32_pcg", "tol": 1e-10},
        # a point cloud in random order with about 35 entries per row
        {"name": "solve_cloud_262144", "call": "solve", "surface": "cloud", "n": 262144, "t": 1e-3,
         "precision": "fp32_pcg", "tol": 1e-10},
        # a time step with new matrix values on the headline mesh (1,048,576 vertices)
        {"name": "refresh_solve_torus_1m", "call": "refresh_solve", "surface": "torus", "a": 2048, "b": 512,
         "t": 1e-4, "precision": "fp32_pcg", "tol": 1e-10},
        # the same step from and to host arrays: values and right-hand side in, solution out
        {"name": "refresh_solve_host_512x256", "call": "refresh_solve_host", "surface": "torus", "a": 512, "b": 256,
         "t": 1e-4, "precision": "fp32_pcg", "tol": 1e-10},
        # differentiable heat diffusion: a new diffusion time, forward solve, adjoint solve, gradients
        {"name": "heat_gradient_1024x512", "call": "heat_gradient", "surface": "torus", "a": 1024, "b": 512,
         "t": 1e-3, "precision": "fp32_pcg", "tol": 1e-12},
        # several signals on one mesh
        {"name": "batched_512x256_8rhs", "call": "batched", "surface": "torus", "a": 512, "b": 256, "t": 1e-4,
         "nrhs": 8, "precision": "fp32_refine", "tol": 1e-10},
        # many meshes of uneven size in one solve
        {"name": "many_12_spheres_8rhs", "call": "many", "surface": "spheres", "count": 12, "lo": 5000, "hi": 50000,
         "t": 1e-3, "nrhs": 8, "precision": "fp32_refine", "tol": 1e-10},
        # the hierarchy of a mesh that has just been loaded
        {"name": "hierarchy_torus_1024x512", "call": "hierarchy", "surface": "torus", "a": 1024, "b": 512},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _torus_sizes(rng, lo, hi):
    n = _log(rng, lo, hi)
    b = max(24, int(round(math.sqrt(n / rng.uniform(1.8, 4.2)))))
    return {"a": max(24, n // b), "b": b}


def draw(rng: random.Random):
    call = rng.choice(["solve", "solve", "solve", "refresh_solve", "refresh_solve_host", "heat_gradient", "batched",
                       "many", "hierarchy"])
    t = 10.0 ** rng.uniform(-4.0, -3.0)
    case = {"call": call, "surface": "torus", "t": t, "precision": "fp32_pcg", "tol": 1e-10}
    if call == "solve":
        case["precision"] = rng.choice(["fp32_pcg", "fp32_pcg", "fp32_refine", "fp64_pcg", "fp64"])
        surface = rng.choice(["torus", "torus", "book", "bilaplacian", "cloud"])
        case["surface"] = surface
        if surface == "torus":
            case.update(_torus_sizes(rng, 2500, 1000000))
        elif surface == "book":
            case.update({"pages": rng.randint(3, 6), "a": rng.randint(40, 150), "b": rng.randint(60, 200)})
        elif surface == "bilaplacian":
            case.update(_torus_sizes(rng, 5000, 30000))
            case["t"] = 1e-3
        else:
            case.update({"n": _log(rng, 16000, 262144), "t": 1e-3})
    elif call == "refresh_solve":
        case.update(_torus_sizes(rng, 10000, 1000000))
    elif call == "refresh_solve_host":
        case.update(_torus_sizes(rng, 10000, 300000))
    elif call == "heat_gradient":
        case.update(_torus_sizes(rng, 4000, 500000))
        case["tol"] = 1e-12
    elif call == "batched":
        case.update(_torus_sizes(rng, 5000, 130000))
        case.update({"nrhs": rng.randint(1, 16), "precision": "fp32_refine"})
    elif call == "many":
        lo = _log(rng, 800, 5000)
        case.update({"surface": "spheres", "count": rng.randint(3, 12), "lo": lo, "hi": lo * rng.randint(2, 8),
                     "nrhs": rng.randint(1, 8), "t": 1e-3, "precision": "fp32_refine"})
    else:
        case = {"call": call, "surface": "torus"}
        case.update(_torus_sizes(rng, 5000, 500000))
    return case


# ---- surfaces and their hierarchies (host; kept per process, as a program keeps its meshes) ----

@functools.lru_cache(maxsize=None)
def _geometry(surface, *sizes):
    """(mass diagonal, Laplacian, prolongations, points, graph row pointers, graph columns)."""
    if surface == "sphere":
        V, F = meshes.icosphere(sizes[0])
    elif surface in ("torus", "bilaplacian"):
        V, F, _ = meshes.jittered_torus(sizes[0], sizes[1], sizes[0] + 7 * sizes[1])
    elif surface == "book":
        V, F, _ = meshes.book(sizes[0], sizes[1], sizes[2], seed=7)
    else:
        V = meshes.noisy_sphere_cloud(sizes[0], np.random.default_rng(2))
        F = None
    if F is None:
        E, h = operators.knn_graph(V, 30)
        L, Md = operators.knn_laplacian(V, E, h), np.ones(V.shape[0])
        edges = operators.knn_graph(V, 6)[0]
    else:
        L, Md = operators.cotan_laplacian(V, F), operators.lumped_mass(V, F)
        edges = meshes.mesh_edges(F)
    rp, ci = operators.edges_to_adjacency(V.shape[0], edges)
    return Md, L, gmg_inputs.build_hierarchy(V, rp, ci), V, rp, ci


@functools.lru_cache(maxsize=None)
def _spheres(count, lo, hi):
    rng = np.random.default_rng(3)
    sizes = np.round(np.exp(rng.uniform(np.log(lo), np.log(hi), size=count))).astype(np.int64)
    out = []
    for n in sizes:
        V, F = meshes.jittered_sphere(int(n), rng)
        rp, ci = operators.edges_to_adjacency(V.shape[0], meshes.mesh_edges(F))
        out.append((operators.lumped_mass(V, F), operators.cotan_laplacian(V, F),
                    gmg_inputs.build_hierarchy(V, rp, ci)))
    return out


def _sizes(case):
    return tuple(case[k] for k in ("level", "pages", "n", "a", "b") if k in case)


def _matrix(case, Md, L, t):
    if case["surface"] == "bilaplacian":
        return operators.bilaplacian_matrix(Md, L, t, 1e-4 * t)
    return operators.system_matrix(Md, L, t)


def _time(case, rng):
    """The diffusion time of one step: the case's, varied by the seed."""
    return case["t"] * float(rng.uniform(0.8, 1.25))


def _inputs(case, seed):
    """Host arrays of one pass, from the seed alone."""
    rng = np.random.default_rng(seed)
    call = case["call"]
    if call == "many":
        parts, t = _spheres(case["count"], case["lo"], case["hi"]), _time(case, rng)
        return {"systems": [(_matrix(case, Md, L, t), Ps) for Md, L, Ps in parts],
                "B": [Md[:, None] * rng.standard_normal((Md.size, case["nrhs"])) for Md, _, _ in parts]}
    Md, L, Ps, V, rp, ci = _geometry(case["surface"], *_sizes(case))
    n = Md.size
    if call == "hierarchy":
        # the mesh at another scale: other coordinates, levels of the same sizes
        return {"V": V * float(rng.uniform(0.5, 2.0)), "rp": rp, "ci": ci}
    t = _time(case, rng)
    if call == "heat_gradient":
        u0 = np.zeros(n)
        u0[rng.choice(n, size=16, replace=False)] = 1.0
        return {"Md": Md, "L": L, "Ps": Ps, "t": t, "t_first": case["t"], "u0": u0, "g": rng.standard_normal(n)}
    if call == "batched":
        return {"A": _matrix(case, Md, L, t), "Ps": Ps, "b": Md[:, None] * rng.standard_normal((n, case["nrhs"]))}
    return {"A": _matrix(case, Md, L, t), "Ps": Ps, "b": Md * rng.standard_normal(n)}


def _cuda(a):
    return torch.tensor(a, dtype=torch.float64, device="cuda")


def prepare(case, seed):
    d, call = _inputs(case, seed), case["call"]
    s = {"call": call, "tol": case.get("tol")}
    if call == "hierarchy":
        return s | d
    if call == "many":
        return s | {"solver": gmg.SolverMany(d["systems"]), "B": [_cuda(B) for B in d["B"]]}
    precision = PRECISION[case["precision"]]
    if call == "heat_gradient":
        solver = gmg.Solver(None, d["Ps"], precision=precision, ml=(d["Md"], d["L"], d["t_first"]))
        return s | {"solver": solver, "t": torch.tensor(d["t"], dtype=torch.float64, requires_grad=True),
                    "u0": _cuda(d["u0"]).requires_grad_(True), "g": _cuda(d["g"])}
    solver = gmg.Solver(d["A"], d["Ps"], precision=precision)
    if call == "refresh_solve_host":
        return s | {"solver": solver, "values": torch.tensor(d["A"].data).pin_memory().numpy(),
                    "b": torch.tensor(d["b"]).pin_memory().numpy()}
    return s | {"solver": solver, "values": _cuda(d["A"].data) if call == "refresh_solve" else None,
                "b": _cuda(d["b"])}


def run(state):
    call, tol = state["call"], state["tol"]
    if call == "hierarchy":
        levels, _ = gmg.build_hierarchy(state["V"], state["rp"], state["ci"])
        return [{"idx": P.idx, "w": P.w, "samples": P.samples, "cell": P.cell, "points": P.Xc,
                 "graph_rowptr": P.graph_rowptr, "graph_col": P.graph_col} for P in levels]
    solver = state["solver"]
    if call == "many":
        return solver.solve(state["B"], tol=tol)[0]
    if call == "batched":
        return solver.solve_batched(state["b"], tol=tol)[0]
    if call == "heat_gradient":
        solver.set_t(float(state["t"].detach()))
        x = smooth(state["t"], state["u0"], solver, tol)
        return (x, *torch.autograd.grad(x, (state["t"], state["u0"]), state["g"]))
    if call != "solve":
        solver.set_values(state["values"])
    return solver.solve(state["b"], tol=tol)[0]


# ---- what a pass cannot do without ----

def _rows_entries(case):
    """Rows and stored entries of the finest system, to within a few per cent for the book and the cloud."""
    surface = case["surface"]
    if surface == "sphere":
        n = 10 * 4 ** case["level"] + 2
        return n, 7 * n - 12
    if surface == "torus":
        return case["a"] * case["b"], 7 * case["a"] * case["b"]
    if surface == "bilaplacian":
        return case["a"] * case["b"], 19 * case["a"] * case["b"]
    if surface == "book":
        n = case["b"] * (1 + case["pages"] * (case["a"] - 1))
        return n, 7 * n
    if surface == "cloud":
        return case["n"], 34 * case["n"]
    rng = np.random.default_rng(3)
    n = int(np.round(np.exp(rng.uniform(np.log(case["lo"]), np.log(case["hi"]), size=case["count"]))).sum())
    return n, 7 * n


def work(case):
    """The finest system's values and columns once, its vectors once, one multiply-add per entry and right-hand
    side; for a hierarchy its points, graph, prolongations and by-products once."""
    n, nnz = _rows_entries(case)
    if case["call"] == "hierarchy":
        graph = nnz - n
        return {"bytes": 24 * n + 12 * graph + 1.2 * (3 * 12 + 4) * n, "flops": 1.2 * (20 * n + 8 * graph)}
    k = case.get("nrhs", 1)
    solves = 2 if case["call"] == "heat_gradient" else 1
    return {"bytes": 12 * nnz + 8 * n + 16 * n * k * solves + (8 * n if solves == 2 else 0),
            "flops": 2 * nnz * k * solves}


# ---- the same answers in 64 bits, by plain conjugate gradients on the assembled system ----

def _csr(A):
    return torch.sparse_csr_tensor(torch.tensor(A.indptr, dtype=torch.int64), torch.tensor(A.indices, dtype=torch.int64),
                                   torch.tensor(A.data, dtype=torch.float64), size=A.shape).cuda()


def _solve(A, B, tol=1e-15, limit=4000):
    """Diagonally preconditioned conjugate gradients on every column of B, with the residual taken anew and the
    correction solved for again until it no longer falls."""
    At = _csr(A)
    d = torch.tensor(A.diagonal(), device="cuda")[:, None]
    B = _cuda(B).reshape(d.shape[0], -1)
    X, norm = torch.zeros_like(B), B.norm(dim=0).clamp_min(1e-300)
    last = torch.full_like(norm, math.inf)
    for _ in range(4):
        R = B - At @ X
        rel = (R.norm(dim=0) / norm).max()
        if rel <= tol or rel > 0.5 * last.max():
            break
        last = rel.reshape(1)
        E, Z = torch.zeros_like(R), R / d
        P, rz, r0 = Z.clone(), (R * Z).sum(0), R.norm(dim=0).clamp_min(1e-300)
        for it in range(limit):
            Q = At @ P
            pq = (P * Q).sum(0)
            alpha = torch.where(pq > 0, rz / pq.clamp_min(1e-300), torch.zeros_like(pq))
            E += alpha * P
            R -= alpha * Q
            if it % 10 == 9 and bool(((R.norm(dim=0) / r0) < 1e-13).all()):
                break
            Z = R / d
            new = (R * Z).sum(0)
            P = Z + torch.where(rz > 0, new / rz.clamp_min(1e-300), torch.zeros_like(rz)) * P
            rz = new
        X += E
    return X


def exact(case, seed):
    call = case["call"]
    if call == "hierarchy":
        return None  # points swept one after another: far too long in plain torch or numpy
    d = _inputs(case, seed)
    if call == "many":
        return [_solve(A, B) for (A, _), B in zip(d["systems"], d["B"])]
    if call == "batched":
        return _solve(d["A"], d["b"])
    if call == "heat_gradient":
        A = operators.system_matrix(d["Md"], d["L"], d["t"])
        x, lam = (_solve(A, v)[:, 0] for v in (d["Md"] * d["u0"], d["g"]))
        return x, -(lam * (_csr(d["L"]) @ x[:, None])[:, 0]).sum(), _cuda(d["Md"]) * lam
    return _solve(d["A"], d["b"])[:, 0]
