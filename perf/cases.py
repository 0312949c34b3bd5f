"""Performance cases: the calls a user of this library makes, over their real range of sizes.

A program that uses the library builds one handle per mesh (``amg_setup``)
and then solves, applies operators and takes sensitivities on it many times,
with new right-hand sides (and, when it inverts for a coefficient, a new
coefficient field) each time.  So a case's mesh comes from the case alone and
its handle is kept, while every vector and coefficient field comes from the
seed; the handle of the most recent meshes is held in a small cache.
"""
from __future__ import annotations

import functools
import math
import time

import numpy as np
import torch

from paper_1410_2153_gb300 import asmg, autograd, meshgen

RTOL = 1e-8
DEVICE = "cuda:0"


def listed():
    return [
        # the smallest solve: 65^2 Poisson problem, FP64, 3969 unknowns (launch latency)
        dict(name="solve_jitter65_fp64", kind="solve", mesh="jitter", nside=65, precision="fp64"),
        # an ordinary solve in the middle of the batched workload's sizes, at an odd side
        dict(name="solve_jitter331_mixed", kind="solve", mesh="jitter", nside=331, precision="mixed"),
        # a non-box domain (square with a hole): Dirichlet auxiliary grids
        dict(name="solve_hole257_mixed", kind="solve", mesh="hole", nside=257, precision="mixed"),
        # strongly graded mesh, plain FP64 form
        dict(name="solve_graded513_fp64", kind="solve", mesh="graded", nside=513, precision="fp64"),
        # the benchmark's workload: 4.2 M unknowns, mixed form with BF16 level matrices
        dict(name="solve_graded2049_bf16", kind="solve", mesh="graded", nside=2049, precision="bf16"),
        # 3D tetrahedra with a 1 / 1e3 coefficient, mixed form
        dict(name="solve_kuhn129_mixed", kind="solve", mesh="kuhn", nside=129, precision="mixed"),
        # four right-hand sides of one operator in one call
        dict(name="multi_jitter513_mixed", kind="multi", mesh="jitter", nside=513, precision="mixed", nrhs=4),
        # many small independent problems, four right-hand sides each, one graph launch
        dict(name="batch_jitter_mixed", kind="batch", mesh="jitter", nside=150, precision="mixed", nrhs=4, nprob=12),
        # one preconditioner application, for a caller with its own Krylov method
        dict(name="precond_kuhn65_fp64", kind="precond", mesh="kuhn", nside=65, precision="fp64"),
        # operator product and load vector on a large mesh, as a time stepper or a residual check uses them
        dict(name="operators_graded1025", kind="operators", mesh="graded", nside=1025, precision="mixed"),
        # element sensitivities of a solution and its adjoint in 3D
        dict(name="gradient_kuhn65", kind="gradient", mesh="kuhn", nside=65, precision="mixed"),
        # one step of a coefficient inversion: new coefficients, forward solve, adjoint solve, gradient
        dict(name="inversion_jitter129_mixed", kind="inversion", mesh="jitter", nside=129, precision="mixed"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "multi", "batch", "precond", "operators", "gradient", "inversion"])
    mesh = rng.choice(["jitter", "jitter", "graded", "L", "hole", "kuhn", "kuhn"])
    precision = rng.choice(["fp64", "mixed", "bf16"])
    if kind == "batch":
        return dict(kind=kind, mesh="jitter", nside=_log_int(rng, 60, 250), precision=precision,
                    nrhs=rng.randint(2, 6), nprob=rng.randint(2, 10))
    if kind == "inversion":
        return dict(kind=kind, mesh="jitter", nside=_log_int(rng, 33, 180), precision=rng.choice(["fp64", "mixed"]))
    top = {"jitter": 900, "graded": 700, "L": 500, "hole": 500, "kuhn": 65}[mesh]
    if kind == "multi":
        top = {"kuhn": 49}.get(mesh, min(top, 500))
    if kind == "precond":
        precision = "fp64"  # a caller's own Krylov method in FP64; the mixed form runs inside the solves
    case = dict(kind=kind, mesh=mesh, nside=_log_int(rng, 13 if mesh == "kuhn" else 33, top), precision=precision)
    if kind == "multi":
        case["nrhs"] = rng.randint(1, 4)
    return case


# ------------------------------------------------------------------- inputs
@functools.lru_cache(maxsize=16)
def _mesh(mesh, nside, which):
    if mesh == "jitter":
        return meshgen.grid2d(nside, 1 + which)
    if mesh == "graded":
        return meshgen.grid2d(nside, 1 + which, graded=True)
    if mesh in ("L", "hole"):
        return meshgen.grid2d_domain(nside, 1 + which, mesh)
    m = meshgen.grid3d(nside, 1 + which)
    if (nside - 1) % 8 == 0:  # the subcubes of the coefficient hold whole cells
        m.coeff = meshgen.subcube_coefficient(m, 2001 + which)
    return m


def _options(case):
    opts = dict(precision=asmg.ASMG_FP64 if case["precision"] == "fp64" else asmg.ASMG_MIXED)
    if case["precision"] == "bf16":
        opts["level_bf16"] = 1
    if case["mesh"] == "kuhn":
        opts["n_min"] = 6  # one cell of six tetrahedra per leaf
    return opts


class _Batch:
    """The solvers of a batch and the batch over them, which goes first."""

    def __init__(self, solvers, nrhs):
        self.solvers = solvers
        self.batch = asmg.amg_batch_create([s.h for s in solvers], nrhs, RTOL)

    def __del__(self):
        asmg.amg_batch_destroy(self.batch)


@functools.lru_cache(maxsize=1)
def _handle(items):
    """The handle(s) a program keeps for the case's mesh(es)."""
    case = dict(items)
    if case["kind"] == "inversion":
        return autograd.CoefficientSolver(_mesh(case["mesh"], case["nside"], 0), rtol=RTOL, **_options(case))
    if case["kind"] == "batch":
        return _Batch([asmg.Solver(_mesh(case["mesh"], _side(case, i), i), **_options(case))
                       for i in range(case["nprob"])], case["nrhs"])
    return asmg.Solver(_mesh(case["mesh"], case["nside"], 0), **_options(case))


def _side(case, i):
    """Sides of a batch's grids: uneven, 0.7 to 1.4 times the case's side."""
    return max(9, int(round(case["nside"] * (0.7 + 0.7 * ((0.618 * (i + 1)) % 1.0)))))


def _loads(solver, mesh, seed, k):
    """k load vectors b = M f of nodal sources f ~ U[-1, 1]."""
    f = meshgen.nodal_uniform(mesh, seed, k).reshape(k, -1)
    return [solver.mass_apply(torch.from_numpy(f[j]).to(DEVICE)) for j in range(k)]


def _field(mesh, seed):
    """A smooth log-coefficient field (unit variance, correlation length 0.1)."""
    return torch.from_numpy(meshgen.grf_coefficient_field(meshgen.centroids(mesh), seed, nfeat=64)).to(DEVICE)


def _vectors(mesh, seed, k):
    """k nodal vectors U[-1, 1], 0 at Dirichlet vertices, on the device."""
    return torch.from_numpy(meshgen.nodal_uniform(mesh, seed, k).reshape(k, -1)).to(DEVICE)


def prepare(case, seed):
    case = {k: v for k, v in case.items() if k != "name"}
    kind, handle = case["kind"], _handle(tuple(sorted(case.items())))
    mesh = _mesh(case["mesh"], case["nside"], 0) if kind != "batch" else None
    st = dict(kind=kind, handle=handle)
    if kind == "solve":
        st["b"] = _loads(handle, mesh, seed, 1)[0]
    elif kind == "multi":
        st["b"] = torch.cat(_loads(handle, mesh, seed, case["nrhs"]))
        st["k"] = case["nrhs"]
    elif kind == "batch":
        st["bs"] = [b for i, s in enumerate(handle.solvers)
                    for b in _loads(s, _mesh(case["mesh"], _side(case, i), i), seed * 64 + i, case["nrhs"])]
    elif kind == "precond":
        st["r"] = _loads(handle, mesh, seed, 1)[0]
    elif kind == "operators":
        st["x"], st["f"] = _vectors(mesh, seed, 2)
    elif kind == "gradient":
        st["u"], st["lam"] = _vectors(mesh, seed, 2)
    elif kind == "inversion":
        st["g"] = _field(mesh, seed)
        st["b"] = _loads(handle.solver, mesh, seed, 1)[0]
        st["u_obs"] = 1e-3 * _vectors(mesh, seed + 1, 1)[0]
    return st


def run(st):
    kind, h = st["kind"], st["handle"]
    if kind == "solve":
        u, status, iterations, _ = h.solve(st["b"], rtol=RTOL)
        return dict(u=u, status=status, iterations=iterations)
    if kind == "multi":
        u = torch.zeros_like(st["b"])
        status, iterations, _ = asmg.amg_solve_multi(h.h, st["k"], st["b"], u, RTOL)
        return dict(u=u, status=status, iterations=iterations)
    if kind == "batch":
        us = [torch.zeros_like(b) for b in st["bs"]]
        status, iterations, _ = asmg.amg_batch_solve(h.batch, st["bs"], us)
        return dict(u=us, status=status, iterations=iterations)
    if kind == "precond":
        return dict(z=h.precond(st["r"]))
    if kind == "operators":
        return dict(y=h.spmv(st["x"]), b=h.mass_apply(st["f"]))
    if kind == "gradient":
        return dict(g=h.element_grad(st["u"], st["lam"]))
    loss, dg, u = autograd.inversion_loss_and_grad(h, st["g"], st["b"], st["u_obs"])
    return dict(loss=loss, dg=dg, u=u)


# --------------------------------------------------------------------- work
def _sizes(case):
    """(vertices, elements, stored entries of A) of the case's mesh, up to boundary terms."""
    n = case["nside"]
    if case["mesh"] == "kuhn":
        return n ** 3, 6 * (n - 1) ** 3, 15 * n ** 3
    part = 0.75 if case["mesh"] in ("L", "hole") else 1.0
    return part * n * n, part * 2 * (n - 1) ** 2, part * 7 * n * n


def work(case):
    """Compulsory bytes and flops of one pass.

    A solve cannot do without reading, in every step, each of its operators
    once (the FP64 fine matrix; in the preconditioner's precision the fine
    matrix for the two smoothing sweeps, the transfer both ways, and the level
    matrices, 4/3 of the fine rows) and each of its vectors once; the number of
    steps is the usual one of the mesh family."""
    kind, dim = case["kind"], 3 if case["mesh"] == "kuhn" else 2
    nv, ne, nnz = _sizes(case)
    s = 8 if case["precision"] == "fp64" else 4
    sl = 2 if case["precision"] == "bf16" else s
    precond = 2 * nnz * (s + 4) + 2 * 8 * nv * (s + 4) + 4 / 3 * nnz * (sl + 4) + 10 * nv * s
    step = nnz * 12 + 8 * 8 * nv + precond
    flops = 2 * (nnz + 2 * nnz + 16 * nv + 4 * 4 / 3 * nnz + 6 * nv)
    if case["mesh"] == "graded":
        steps = 37 * (case["nside"] / 257) ** 0.61
    else:
        steps = 30 if case["mesh"] == "kuhn" and (case["nside"] - 1) % 8 == 0 else 9
    if kind == "solve":
        return dict(bytes=steps * step + 16 * nv, flops=steps * flops)
    if kind == "inversion":
        return dict(bytes=2 * steps * step + ne * (24 + 8 * 3), flops=2 * steps * flops)
    if kind in ("multi", "batch"):
        k, share = case["nrhs"], case.get("nprob", 1)
        vec = 8 * 8 * nv + 10 * nv * s
        groups = -(-k // 4)
        return dict(bytes=share * steps * (groups * (step - vec) + k * vec), flops=share * k * steps * flops)
    if kind == "precond":
        return dict(bytes=precond + 16 * nv, flops=flops)
    element = ne * (dim + 1) * 4 + nv * dim * 8
    if kind == "operators":
        return dict(bytes=nnz * 12 + 16 * nv + element + 16 * nv, flops=2 * nnz + 12 * ne)
    return dict(bytes=element + 16 * nv + 8 * ne, flops=40 * ne)


# -------------------------------------------------------------------- exact
def _geometry(mesh):
    """Device tensors: elements [ne, d+1], basis gradients [ne, d+1, d], measures [ne], free mask [nv]."""
    x = torch.from_numpy(mesh.verts).to(DEVICE)
    e = torch.from_numpy(mesh.elems.astype(np.int64)).to(DEVICE)
    p = x[e]
    edges = p[:, 1:] - p[:, :1]
    meas = torch.linalg.det(edges) / math.factorial(mesh.dim)
    inv = torch.linalg.inv(edges)  # columns: gradients of the last d basis functions
    grads = torch.cat([-inv.sum(2, keepdim=True), inv], 2).transpose(1, 2)
    return e, grads, meas, torch.from_numpy(mesh.bflag == 0).to(DEVICE)


def _matrix(mesh, coeff, geo):
    """Stiffness matrix in CSR, identity rows at Dirichlet vertices; its diagonal."""
    e, grads, meas, free = geo
    k = torch.bmm(grads, grads.transpose(1, 2)) * (meas if coeff is None else meas * coeff)[:, None, None]
    r, c = e[:, :, None].expand_as(k).reshape(-1), e[:, None, :].expand_as(k).reshape(-1)
    keep = free[r] & free[c]
    fixed = torch.nonzero(~free).reshape(-1)
    r, c, v = torch.cat([r[keep], fixed]), torch.cat([c[keep], fixed]), torch.cat([k.reshape(-1)[keep], torch.ones_like(fixed, dtype=torch.float64)])
    a = torch.sparse_coo_tensor(torch.stack([r, c]), v, (mesh.nv, mesh.nv)).coalesce()
    i, d = a.indices(), torch.zeros(mesh.nv, dtype=torch.float64, device=DEVICE)
    on = i[0] == i[1]
    d[i[0][on]] = a.values()[on]
    return a.to_sparse_csr(), d


def _cg(a, d, b, limit_s):
    """Jacobi-preconditioned CG to the rounding floor; None when it takes too long."""
    x, r = torch.zeros_like(b), b.clone()
    z = r / d
    p, rz, target = z.clone(), torch.dot(r, z), 1e-13 * float(b.norm())
    began = time.perf_counter()
    for it in range(200000):
        q = a @ p
        alpha = rz / torch.dot(p, q)
        x += alpha * p
        r -= alpha * q
        z = r / d
        new = torch.dot(r, z)
        p = z + (new / rz) * p
        rz = new
        if it % 50 == 49:
            if float(r.norm()) <= target:
                return x
            if time.perf_counter() - began > limit_s:
                return None
    return None


def _mass(mesh, geo, f):
    e, _, meas, free = geo
    fe = f[e]
    scale = meas / ((mesh.dim + 1) * (mesh.dim + 2))
    be = (fe + fe.sum(1, keepdim=True)) * scale[:, None]
    out = torch.zeros_like(f).index_add_(0, e.reshape(-1), be.reshape(-1))
    return torch.where(free, out, torch.zeros_like(out))


def exact(case, seed):
    """The same outputs from a plain FP64 assembly and Jacobi-CG in torch.

    Step counts belong to the method and have no exact value, nor does one
    application of the preconditioner."""
    case = {k: v for k, v in case.items() if k != "name"}
    kind = case["kind"]
    if kind == "precond" or (case["mesh"] == "graded" and kind != "operators" and case["nside"] > 1100):
        return None
    if kind == "batch":
        us, began = [], time.perf_counter()
        for i in range(case["nprob"]):
            mesh = _mesh(case["mesh"], _side(case, i), i)
            geo = _geometry(mesh)
            a, d = _matrix(mesh, None, geo)
            f = meshgen.nodal_uniform(mesh, seed * 64 + i, case["nrhs"]).reshape(case["nrhs"], -1)
            us += [_cg(a, d, _mass(mesh, geo, torch.from_numpy(f[j]).to(DEVICE)), 15) for j in range(case["nrhs"])]
            if time.perf_counter() - began > 18:
                return None
        return dict(u=us, status=None, iterations=None)
    mesh = _mesh(case["mesh"], case["nside"], 0)
    geo = _geometry(mesh)
    e, grads, meas, free = geo
    coeff = None if mesh.coeff is None else torch.from_numpy(mesh.coeff).to(DEVICE)
    if kind == "operators":
        x, f = _vectors(mesh, seed, 2)
        a, _ = _matrix(mesh, coeff, geo)
        return dict(y=torch.where(free, a @ torch.where(free, x, torch.zeros_like(x)), torch.zeros_like(x)),
                    b=_mass(mesh, geo, f))
    if kind == "gradient":
        u, lam = _vectors(mesh, seed, 2)
        return dict(g=-((u[e][:, :, None] * grads).sum(1) * (lam[e][:, :, None] * grads).sum(1)).sum(1) * meas)
    if kind == "inversion":
        g = _field(mesh, seed)
        a, d = _matrix(mesh, g.exp(), geo)
        u = _cg(a, d, _mass(mesh, geo, _vectors(mesh, seed, 1)[0]), 8)
        if u is None:
            return None
        misfit = torch.where(free, u - 1e-3 * _vectors(mesh, seed + 1, 1)[0], torch.zeros_like(u))
        lam = _cg(a, d, misfit, 8)
        if lam is None:
            return None
        dg = -((u[e][:, :, None] * grads).sum(1) * (lam[e][:, :, None] * grads).sum(1)).sum(1) * meas * g.exp()
        return dict(loss=0.5 * (misfit ** 2).sum(), dg=dg, u=u)
    a, d = _matrix(mesh, coeff, geo)
    k = case.get("nrhs", 1)
    f = meshgen.nodal_uniform(mesh, seed, k).reshape(k, -1)
    us = [_cg(a, d, _mass(mesh, geo, torch.from_numpy(f[j]).to(DEVICE)), 15 / k) for j in range(k)]
    if any(u is None for u in us):
        return None
    return dict(u=torch.cat(us), status=None, iterations=None)
