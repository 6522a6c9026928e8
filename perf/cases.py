"""Workloads for timing the library through its public entry points.

A case is a mesh family and size, a rank, the number of right-hand sides, a
precision and what is done with them:

  apply     Y = A X of an operator that the program holds (vfd_apply)
  solve     A U = F by CG or preconditioned CG, FP64 (vfd_solve)
  mixed     A U = F for 64 columns on low-precision operators with FP64 true
            residuals, one mesh (vfd_solve) or several (vfd_batch_solve)
  step      new fields on a known mesh: assembly, load, solve, density
  gradient  the misfit of an inverse problem and its gradient with respect to
            nodal s, log kappa and the load (autograd: two solves, vfd_grad)

Meshes, fields, ranks and tolerances are those of the tests and of the
benchmark: disks of rings with an annulus to R = 1.1, squares (-1,1)^2 inside
(-2,2)^2, intervals with an exterior tail, balls of Kuhn tetrahedra; fields
with a few Fourier modes or a sigmoid of them.  Solves run to 1e-11, between
the benchmark's 1e-10 and the 1e-12 of the differentiable solve.
"""
from __future__ import annotations

import functools
import itertools
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2302_02863_gb300 import autograd, vfd

S_BAR = 0.9
RTOL = 1e-11
TAIL_R = 1.1
PRECISION = {"fp64": vfd.VFD_FP64, "fp32": vfd.VFD_FP32, "bf16": vfd.VFD_BF16}
PREC_KIND = {"none": vfd.VFD_PREC_NONE, "two_level": vfd.VFD_PREC_TWO_LEVEL, "jacobi": vfd.VFD_PREC_BLOCK_JACOBI}


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------
def _case(task, mesh, size, p, nrhs=1, **more):
    c = {"task": task, "mesh": mesh, "size": size, "p": p, "nrhs": nrhs, "leaf": 64, "precision": "fp64",
         "precond": "none", "fields": "modes", "count": 1, "ratio": 1.0}
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: one column on the parity-size disk of 397 DoFs, a
        # handful of short launches
        dict(_case("apply", "disk", 12, 4), name="apply_disk_small"),
        # a few columns at once on a mid-size square with short leaves (ragged
        # leaf sizes, odd column count)
        dict(_case("apply", "square", 62, 5, nrhs=5, leaf=40), name="apply_square_5cols"),
        # the matvec of the benchmark disk: 27,361 DoFs, rank 64, one column
        dict(_case("apply", "disk", 96, 8), name="apply_disk"),
        # the same operator on a block of 64 columns (multi-RHS applies, the true
        # residuals of the mixed-precision solves)
        dict(_case("apply", "disk", 96, 8, nrhs=64), name="apply_disk_64cols"),
        # 1D problem with the exterior tail, 512 interior nodes: assembly and
        # solve of a small problem, where launches and host work count
        dict(_case("step", "interval", 512, 4, fields="const"), name="step_interval"),
        # plain CG on the square of the paper's experiments (16,129 DoFs, rank 16)
        dict(_case("solve", "square", 128, 4), name="solve_square"),
        # preconditioned CG, three load cases, on a disk of 10k DoFs
        dict(_case("solve", "disk", 59, 6, nrhs=3, precond="two_level"), name="solve_disk_precond"),
        # the mixed-precision solve: 64 columns, BF16 inner operator,
        # preconditioned, on the benchmark disk
        dict(_case("mixed", "disk", 96, 8, nrhs=64, precision="bf16", precond="two_level"), name="mixed_disk_64rhs"),
        # many meshes of uneven size in one batch, TF32 inner operators, plain
        dict(_case("mixed", "mixed", 1500, 4, nrhs=64, precision="fp32", fields="sigmoid", count=4, ratio=1.7),
             name="mixed_batch_4meshes"),
        # the benchmark's step: assembly of the benchmark disk for new fields,
        # then the solve for f = 1
        dict(_case("step", "disk", 96, 8), name="step_disk"),
        # differentiation: misfit and gradient with P1 fields on a disk of 4k DoFs
        dict(_case("gradient", "disk", 37, 6, fields="nodal"), name="gradient_disk"),
        # 3D: tetrahedra in a ball (K + M), rank 64, assembly and solve
        dict(_case("step", "ball", 14, 4, fields="bump"), name="step_ball"),
    ]


def _logint(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    task = rng.choice(["apply", "apply", "solve", "mixed", "step", "step", "gradient"])
    mesh = rng.choice(["disk", "square"])
    n = {"apply": 27000, "solve": 16000, "mixed": 12000, "step": 27000, "gradient": 6000}[task]
    n = _logint(rng, 300, n)
    size = (max(5, int(round(0.5 + math.sqrt(n / 3.0)))) if mesh == "disk"
            else 2 * max(6, int(round(0.5 * (math.sqrt(n) + 1)))))
    c = _case(task, mesh, size, rng.randint(3, 8), leaf=rng.choice([24, 32, 48, 64, 64]))
    if task == "apply":
        c["nrhs"] = _logint(rng, 1, 96)
    elif task == "solve":
        c["nrhs"] = rng.randint(1, 4)
        c["precond"] = rng.choice(["none", "two_level", "jacobi"])
    elif task == "mixed":
        c["nrhs"] = 64
        c["precision"] = rng.choice(["fp32", "bf16"])
        c["precond"] = rng.choice(["none", "two_level"])
        if rng.random() < 0.4:
            c.update(mesh="mixed", size=_logint(rng, 300, 2500), count=rng.randint(2, 4), ratio=round(rng.uniform(1.1, 1.7), 3))
    elif task == "step":
        other = rng.random()
        if other < 0.15:
            c.update(mesh="interval", size=_logint(rng, 40, 3000), fields="const", p=rng.randint(3, 8))
        elif other < 0.3:
            c.update(mesh="ball", size=rng.randint(8, 13), fields="bump", p=rng.randint(2, 4))
    if task == "gradient":
        c["fields"] = "nodal"
    elif c["fields"] == "modes" and rng.random() < 0.3:
        c["fields"] = "sigmoid"
    return c


# ----------------------------------------------------------------------------
# meshes
# ----------------------------------------------------------------------------
def _positive(X, T):
    e = X[T[:, 1:]] - X[T[:, :1]]
    neg = np.linalg.det(e) < 0
    T[neg, 1], T[neg, 2] = T[neg, 2].copy(), T[neg, 1].copy()
    return T


def _disk(K, seed):
    """Rings k = 1..K at radius k/K with 6k nodes, an annulus of about K/10
    further rings to R = 1.1; every node off the two circles jittered."""
    rng = np.random.default_rng(seed)
    next_ = max(1, int(round((TAIL_R - 1.0) * K)))
    radii = np.concatenate([np.arange(K + 1) / K, 1.0 + np.arange(1, next_ + 1) * (TAIL_R - 1.0) / next_])
    X, ring, first, cells = [np.zeros((1, 2))], [np.zeros(1, dtype=int)], [0], []
    for k in range(1, len(radii)):
        first.append(1 + 3 * k * (k - 1))
        th = 2.0 * math.pi * np.arange(6 * k) / (6 * k)
        X.append(radii[k] * np.stack([np.cos(th), np.sin(th)], axis=1))
        ring.append(np.full(6 * k, k))
    for k in range(len(radii) - 1):
        t, j = np.meshgrid(np.arange(6), np.arange(k + 1), indexing="ij")
        t, j = t.ravel(), j.ravel()
        inner = lambda i: first[k] + (i % (6 * k) if k else 0 * i)  # noqa: E731
        outer = lambda i: first[k + 1] + i % (6 * (k + 1))  # noqa: E731
        o = t * (k + 1) + j
        cells.append(np.stack([inner(t * k + j), outer(o), outer(o + 1)], axis=1))
        m = j < k
        cells.append(np.stack([inner(t * k + j)[m], outer(o + 1)[m], inner(t * k + j + 1)[m]], axis=1))
    X, ring, T = np.concatenate(X), np.concatenate(ring), np.concatenate(cells).astype(np.int32)
    inside = (ring[T].max(axis=1) <= K).astype(np.uint8)
    free = (ring != K) & (ring != len(radii) - 1)
    ang, move = 2.0 * math.pi * rng.random(len(X)), 0.2 / K * np.sqrt(rng.random(len(X))) * free
    X = X + move[:, None] * np.stack([np.cos(ang), np.sin(ang)], axis=1)
    return 2, X, _positive(X, T), inside


def _square(mc, seed):
    """(-2,2)^2 in squares of leg 2/mc cut along their diagonals, (-1,1)^2
    interior, nodes jittered off the lines +-1, +-2."""
    n, h = 2 * mc, 2.0 / mc
    g = -2.0 + h * np.arange(n + 1)
    X = np.stack([a.ravel() for a in np.meshgrid(g, g, indexing="xy")], axis=1)
    i, j = (a.ravel() for a in np.meshgrid(np.arange(n), np.arange(n), indexing="xy"))
    a = j * (n + 1) + i
    b, c, e = a + 1, a + n + 2, a + n + 1
    T = np.concatenate([np.stack([a, b, c], 1), np.stack([a, c, e], 1)]).astype(np.int32)
    inside = ((np.abs(g[i] + 0.5 * h) < 1.0) & (np.abs(g[j] + 0.5 * h) < 1.0)).astype(np.uint8)
    move = 0.2 * h * (2.0 * np.random.default_rng(seed).random(X.shape) - 1.0)
    move[np.isclose(np.abs(X), 1.0) | np.isclose(np.abs(X), 2.0)] = 0.0
    X = X + move
    return 2, X, _positive(X, T), np.concatenate([inside, inside])


def _interval(n):
    h = 2.0 / (n + 1)
    m = max(1, int(math.ceil((TAIL_R - 1.0) / h - 1e-12)))
    right = 1.0 + (TAIL_R - 1.0) * np.arange(1, m + 1) / m
    x = np.concatenate([-right[::-1], np.linspace(-1.0, 1.0, n + 2), right])
    T = np.stack([np.arange(len(x) - 1), np.arange(1, len(x))], axis=1).astype(np.int32)
    return 1, x[:, None].copy(), T, (np.abs(0.5 * (x[1:] + x[:-1])) < 1.0).astype(np.uint8)


def _ball(n):
    """The cubes of [-1.1, 1.1]^3 in 6 Kuhn tetrahedra each, those with
    centroid inside radius 1.1 kept, inside radius 1 interior."""
    g = np.arange(n + 1) * (2.2 / n) - 1.1
    X = np.stack([a.ravel() for a in np.meshgrid(g, g, g, indexing="ij")], axis=1)
    o = np.stack([a.ravel() for a in np.meshgrid(*3 * [np.arange(n)], indexing="ij")], axis=1)
    cells = []
    for perm in itertools.permutations(range(3)):
        at, path = o.copy(), []
        for ax in (None,) + perm:
            if ax is not None:
                at = at.copy()
                at[:, ax] += 1
            path.append((at[:, 0] * (n + 1) + at[:, 1]) * (n + 1) + at[:, 2])
        cells.append(np.stack(path, axis=1))
    T = np.concatenate(cells)
    r = np.linalg.norm(X[T].mean(axis=1), axis=1)
    T, r = T[r < 1.1], r[r < 1.1]
    used, T = np.unique(T, return_inverse=True)
    T = T.reshape(-1, 4).astype(np.int32)
    X = X[used]
    e = X[T[:, 1:]] - X[T[:, :1]]
    neg = np.linalg.det(e) < 0
    T[neg, 2], T[neg, 3] = T[neg, 3].copy(), T[neg, 2].copy()
    return 3, X, T, (r < 1.0).astype(np.uint8)


@functools.lru_cache(maxsize=16)
def _geometry(kind, size):
    if kind == "disk":
        return _disk(size, 2000 + size)
    if kind == "square":
        return _square(size, 3000 + size)
    return _interval(size) if kind == "interval" else _ball(size)


def _geometries(case):
    """(kind, size) of every mesh of the case."""
    if case["mesh"] != "mixed":
        return [(case["mesh"], case["size"])]
    out = []
    for i in range(case["count"]):
        n = case["size"] * case["ratio"] ** i
        out.append(("square", 2 * int(round(0.5 * (math.sqrt(n) + 1)))) if i % 2 == 0 else
                   ("disk", int(round(0.5 + math.sqrt(n / 3.0)))))
    return out


@functools.lru_cache(maxsize=6)
def _mesh(kind, size, p, leaf, inner):
    # a program builds the handle of its mesh once and assembles operators for
    # many fields on it
    d, X, T, inside = _geometry(kind, size)
    opts = dict(leaf_m=leaf, cheb_p=p, lam=0.75, tail_mode=1 if kind == "interval" else 0, tail_R=TAIL_R)
    if inner:
        opts["inner_p"] = min(p, 4)   # the benchmark's inner operator
    return vfd.vfd_mesh(d, X, T, inside, **opts)


def _meshes(case):
    return [_mesh(k, n, case["p"], case["leaf"], case["task"] == "mixed") for k, n in _geometries(case)]


# ----------------------------------------------------------------------------
# fields
# ----------------------------------------------------------------------------
def _modes(rng, d, sigma):
    rows = np.zeros((16, 5))
    while (empty := np.all(rows[:, :3] == 0.0, axis=1)).any():
        rows[empty, :d] = rng.integers(-3, 4, (empty.sum(), d))
    rows[:, 3] = rng.standard_normal(16)
    rows[:, 4] = 2.0 * math.pi * rng.random(16)
    rows[:, 3] *= sigma / math.sqrt(0.5 * np.sum(rows[:, 3] ** 2))
    return rows


def _fields(case, d, X, seed):
    """Descriptors of s and log kappa."""
    rng = np.random.default_rng(seed)
    logk = SimpleNamespace(c0=0.0, fourier=_modes(rng, d, 0.5))
    kind = case["fields"]
    if kind == "const":
        return SimpleNamespace(c0=0.2 + 0.5 * rng.random()), SimpleNamespace(c0=float(rng.uniform(-1.0, 0.0)))
    if kind == "sigmoid":
        return SimpleNamespace(c0=0.0, fourier=_modes(rng, d, 1.0), squash=1, lo=0.1, hi=0.9), logk
    if kind == "bump":
        x0 = rng.uniform(-0.3, 0.3, 3)
        return SimpleNamespace(c0=0.2, gauss=np.array([[*x0, 0.6, 4.0]])), logk
    ph = 2.0 * math.pi * rng.random(2)
    s = SimpleNamespace(c0=0.5, fourier=np.array([[2, 2, 0, 0.125, ph[0]], [2, -2, 0, 0.125, ph[1]]]))
    if kind == "nodal":
        x = torch.tensor(X, device="cuda")
        return (SimpleNamespace(nodal=_evaluate(s, x).contiguous()),
                SimpleNamespace(nodal=_evaluate(logk, x).contiguous()))
    return s, logk


def _evaluate(f, x):
    """A field descriptor at points x (..., d)."""
    v = torch.full(x.shape[:-1], float(f.c0), dtype=torch.float64, device=x.device)
    d = x.shape[-1]
    for r in getattr(f, "fourier", ()):
        v = v + r[3] * torch.cos(math.pi * (x @ torch.tensor(r[:d], device=x.device)) + r[4])
    for r in getattr(f, "gauss", ()):
        v = v + r[3] * torch.exp(-r[4] * ((x - torch.tensor(r[:d], device=x.device)) ** 2).sum(-1))
    if getattr(f, "squash", 0):
        v = f.lo + (f.hi - f.lo) * torch.sigmoid(v)
    return v


# ----------------------------------------------------------------------------
# what a program holds before the call, and the call
# ----------------------------------------------------------------------------
def _normal(shape, seed):
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(seed))


def _rhs(case, m, i, seed):
    return _normal((case["nrhs"], m.n_dof) if case["nrhs"] > 1 or case["task"] == "mixed" else (m.n_dof,),
                   seed + 1 + 7919 * i)


def _smooth(case, seed):
    """A smooth function near 1 at the vertices (loads are f = 1 or smooth)."""
    X = torch.tensor(_geometry(*_geometries(case)[0])[1], device="cuda")
    amp = 0.2 * _normal((2,), seed)
    return 1.0 + amp[0] * torch.sin(2.0 * X[:, 0]) + amp[1] * torch.cos(3.0 * X.sum(-1))


def prepare(case, seed):
    meshes = _meshes(case)
    st = SimpleNamespace(case=case, meshes=meshes)
    st.fields = [_fields(case, m.d, _geometry(*g)[1], seed + 100 * i)
                 for i, (m, g) in enumerate(zip(meshes, _geometries(case)))]
    task = case["task"]
    if task in ("apply", "solve", "mixed"):
        st.ops = [vfd.vfd_assemble(m, s, k, S_BAR, precision=PRECISION[case["precision"]])
                  for m, (s, k) in zip(meshes, st.fields)]
        for op in st.ops:
            if case["precond"] != "none":
                vfd.vfd_precondition(op, PREC_KIND[case["precond"]])
        st.rhs = [_rhs(case, m, i, seed) for i, m in enumerate(meshes)]
        if len(st.ops) > 1:
            st.batch = vfd.vfd_batch_create(st.ops)
    elif task == "step":
        st.f = _smooth(case, seed + 1)   # the load function at the vertices
    else:
        m = meshes[0]
        dof = torch.tensor(vfd.vfd_mesh_dofs(m)[0], device="cuda").long()
        st.s, st.logk = (f.nodal for f in st.fields[0])
        st.F, st.mass = (vfd.vfd_load(m, f, torch.empty(m.n_dof, dtype=torch.float64, device="cuda"))
                         for f in (_smooth(case, seed + 1), torch.ones_like(st.s)))
        st.u_obs = torch.empty_like(st.F)
        st.u_obs[dof[dof >= 0]] = 0.2 * _smooth(case, seed + 2)[dof >= 0]
    return st


def run(st):
    task = st.case["task"]
    if task == "apply":
        Y = torch.empty_like(st.rhs[0])
        return vfd.vfd_apply(st.ops[0], st.rhs[0], Y)
    if task == "solve" or (task == "mixed" and len(st.ops) == 1):
        U = torch.zeros_like(st.rhs[0])
        vfd.vfd_solve(st.ops[0], st.rhs[0], U, rtol=RTOL, max_it=20000, raise_on_noconv=True)
        return U
    if task == "mixed":
        Us = [torch.zeros_like(F) for F in st.rhs]
        vfd.vfd_batch_solve(st.batch, st.rhs, Us, rtol=RTOL, max_it=20000, raise_on_noconv=True)
        return Us
    m = st.meshes[0]
    if task == "step":
        s, k = st.fields[0]
        op = vfd.vfd_assemble(m, s, k, S_BAR)
        F = vfd.vfd_load(m, st.f, torch.empty(m.n_dof, dtype=torch.float64, device="cuda"))
        U = torch.zeros_like(F)
        vfd.vfd_solve(op, F, U, rtol=RTOL, max_it=20000, raise_on_noconv=True)
        rho = vfd.vfd_op_rho(op, torch.empty(m.info["n_qint"], dtype=torch.float64, device="cuda"))
        return {"U": U, "rho": rho}
    s, k, F = (t.clone().requires_grad_(True) for t in (st.s, st.logk, st.F))
    U = autograd.solve(s, k, F, m, S_BAR)
    e = U - st.u_obs
    J = (st.mass * e * e).sum()
    gs, gk, gF = torch.autograd.grad(J, (s, k, F))
    return {"U": U.detach(), "g_s": gs, "g_logkappa": gk, "g_F": gF}


# ----------------------------------------------------------------------------
# work that a pass cannot do without
# ----------------------------------------------------------------------------
@functools.lru_cache(maxsize=64)
def _info(kind, size, p, leaf, inner):
    return dict(_mesh(kind, size, p, leaf, inner).info, d=_geometry(kind, size)[0])


def work(case):
    total = {"bytes": 0.0, "flops": 0.0}
    for kind, size in _geometries(case):
        i = _info(kind, size, case["p"], case["leaf"], case["task"] == "mixed")
        N, k, nrhs = i["n_dof"], i["rank"], case["nrhs"]
        # near entries, B + M, coupling blocks, leaf bases and transfers: each read
        # once (nested bases; one multiply-add per entry and column)
        far = i["far_blocks"] * k * k + (2 * N * k + 2 * i["nodes"] * k * k if i["far_blocks"] else 0)
        entries = i["near_entries"] + i["nnz"] + far
        width = {"fp64": 8, "fp32": 4, "bf16": 2}[case["precision"]]
        op_bytes = width * (i["near_entries"] + far) + 12.0 * i["nnz"]
        # kernel evaluations of an assembly, by symmetry each unordered pair of near
        # points once (about 6 rule points per DoF in 2D, 24 in 3D), 60 operations each
        per_dof = {1: 3, 2: 6, 3: 24}[i["d"]]
        evals = (0.5 * i["near_entries"] * per_dof ** 2 + i["rho_near_pairs"] + i["rho_far_blocks"] * k * k
                 + 0.5 * i["far_blocks"] * k * k + i["sing_points"])
        # iterations of a solve, nominal: about 3 sqrt(N), preconditioned 40
        its = 40.0 if case["precond"] == "two_level" else 3.0 * math.sqrt(N)
        if case["task"] == "apply":
            b, f = op_bytes + 16.0 * N * nrhs, 2.0 * entries * nrhs
        elif case["task"] in ("solve", "mixed"):
            b, f = op_bytes + 16.0 * N * nrhs, 2.0 * entries * nrhs * its
        elif case["task"] == "step":
            b, f = op_bytes + 24.0 * i["n_q"] + 16.0 * N, 60.0 * evals + 2.0 * entries * its
        else:
            b, f = op_bytes + 48.0 * i["n_q"] + 16.0 * N, 180.0 * evals + 4.0 * entries * its
        total["bytes"] += b
        total["flops"] += f
    return total


# ----------------------------------------------------------------------------
# the same in 64 bits with plain torch: the quadrature-discretised operator
# without H^2 approximations, as a dense matrix
# ----------------------------------------------------------------------------
EXACT_MAX_DOFS, EXACT_MAX_POINTS = 6000, 130000   # a dense assembly and a direct solve in some seconds


class _Dense:
    """A = B + K + M and rho on one mesh for point functions fs, fk of
    (points, vertex ids, barycentrics)."""

    def __init__(self, mesh, geom, fs, fk, tail):
        self.d, X, T, inside = geom
        dev = "cuda"
        dof, self.N = vfd.vfd_mesh_dofs(mesh)   # the numbering of the outputs
        self.dof = torch.tensor(dof.astype(np.int64), device=dev)
        self.X = torch.tensor(X, device=dev)
        order = np.concatenate([np.nonzero(inside)[0], np.nonzero(inside == 0)[0]])
        self.T = torch.tensor(T[order].astype(np.int64), device=dev)
        self.nint, self.C, self.tail = int(inside.sum()), len(T), tail
        self.fs, self.fk = fs, fk
        d, nv = self.d, self.d + 1
        if d == 1:
            g = 0.5 * math.sqrt(0.6)
            t = np.array([0.5 - g, 0.5, 0.5 + g])
            bary, w = np.stack([1.0 - t, t], 1), np.array([5.0, 8.0, 5.0]) / 18.0
        elif d == 2:
            bary, w = np.full((3, 3), 1 / 6) + 0.5 * np.eye(3), np.full(3, 1 / 3)
        else:
            a, b = (5.0 + 3.0 * math.sqrt(5.0)) / 20.0, (5.0 - math.sqrt(5.0)) / 20.0
            bary, w = np.full((4, 4), b) + (a - b) * np.eye(4), np.full(4, 0.25)
        self.nq = len(w)
        bary, w = torch.tensor(bary, device=dev), torch.tensor(w, device=dev)
        P = self.X[self.T]
        e = P[:, 1:] - P[:, :1]
        self.meas = torch.linalg.det(e).abs() / math.factorial(d)
        self.q = (bary @ P).reshape(-1, d)
        self.w = (self.meas[:, None] * w).reshape(-1)
        self.bary = bary.expand(self.C, -1, -1).reshape(-1, nv)
        self.vid = self.T.repeat_interleave(self.nq, 0)
        # touching cell pairs (first, second), both orders
        inc = [[] for _ in range(len(X))]
        for c, vs in enumerate(self.T.cpu().tolist()):
            for v in vs:
                inc[v].append(c)
        pr = np.unique(np.concatenate([np.stack([a.ravel() for a in np.meshgrid(l, l)], 1) for l in inc if l]), axis=0)
        self.touch = torch.tensor(pr, device=dev)
        # psi: (interior points) x (DoFs), quadrature weights not included
        nqi = self.nint * self.nq
        col = self.dof[self.vid[:nqi]]
        row = torch.arange(nqi, device=dev)[:, None].expand_as(col)
        on = col >= 0
        self.psi = torch.sparse_coo_tensor(torch.stack([row[on], col[on]]), self.bary[:nqi][on], (nqi, self.N)).coalesce()
        self.order = order

    def point_fields(self):
        return self.fs(self.q, self.vid, self.bary), self.fk(self.q, self.vid, self.bary)

    def chunks(self, s, k):
        """(first point, gamma of a run of interior points against all points, 0 where cells touch)."""
        step = max(1, 60_000_000 // (self.C * self.nq * self.nq))
        for c0 in range(0, self.nint, step):
            c1 = min(self.nint, c0 + step)
            i0, i1 = c0 * self.nq, c1 * self.nq
            r2 = sum((self.q[i0:i1, None, j] - self.q[None, :, j]) ** 2 for j in range(self.d))
            sel = self.touch[(self.touch[:, 0] >= c0) & (self.touch[:, 0] < c1)]
            mask = torch.zeros((c1 - c0, self.C), dtype=torch.bool, device="cuda")
            mask[sel[:, 0] - c0, sel[:, 1]] = True
            mask = mask.repeat_interleave(self.nq, 0).repeat_interleave(self.nq, 1)
            r2 = torch.where(mask, 1.0, r2)
            g = torch.exp(0.5 * (k[i0:i1, None] + k[None]) - 0.5 * (self.d + s[i0:i1, None] + s[None]) * torch.log(r2))
            yield i0, torch.where(mask, 0.0, g)

    def tail_density(self, s, k):
        nqi = self.nint * self.nq
        if not self.tail:
            return torch.zeros(nqi, dtype=torch.float64, device="cuda")
        x, a, t = self.q[:nqi, 0], torch.exp(k[:nqi]), 2.0 * s[:nqi]
        return a * ((TAIL_R - x) ** -t + (TAIL_R + x) ** -t) / t

    def singular(self):
        """(local vertex ids, local matrices) per kind of touching pair; none in 3D."""
        if self.d == 3:
            return
        t = self.touch[(self.touch[:, 0] < self.nint)]
        orig = torch.tensor(self.order, device="cuda")
        first, second = t[:, 0], t[:, 1]
        both = second < self.nint
        keep = torch.where(both, orig[first] <= orig[second], True)
        first, second = first[keep], second[keep]
        V1, V2 = self.T[first], self.T[second]
        same = V1[:, :, None] == V2[:, None, :]
        shared = same.any(2).sum(1)
        nv = self.d + 1
        gx, gw = np.polynomial.legendre.leggauss(3)
        gx, gw = torch.tensor(0.5 * (gx + 1.0), device="cuda"), torch.tensor(0.5 * gw, device="cuda")
        for n in range(1, nv + 1):
            at = shared == n
            if not at.any():
                continue
            in1, in2 = same[at].any(2), same[at].any(1)
            rank = torch.arange(nv, device="cuda")
            o1 = torch.argsort(torch.where(in1, 0, 10) + rank, 1)
            p = V1[at].gather(1, o1)
            if n == nv:
                q, loc = p, p
            else:
                o2 = torch.argsort(torch.where(in2, 0, 10) + rank, 1)
                q = torch.cat([p[:, :n], V2[at].gather(1, o2)[:, n:]], 1)
                loc = torch.cat([p, q[:, n:]], 1)
            rule = self._rules1 if self.d == 1 else self._rules2
            yield loc, rule(n, p, q, gx, gw) * (1.0 if n == nv else 2.0)

    def _value(self, p, xh):
        """Points, s and log kappa at reference coordinates xh (points, d) of cells p."""
        P = self.X[p]
        if self.d == 1:
            b = torch.stack([1.0 - xh[:, 0], xh[:, 0]], 1)
        else:
            b = torch.stack([1.0 - xh[:, 0], xh[:, 0] - xh[:, 1], xh[:, 1]], 1)
        x = torch.einsum("qa,nad->nqd", b, P)
        v, bb = p[:, None].expand(-1, len(b), -1), b[None].expand(len(p), -1, -1)
        return self.fs(x, v, bb), self.fk(x, v, bb)

    def _rules1(self, n, p, q, gx, gw):
        z, t = (a.ravel() for a in torch.meshgrid(gx, gx, indexing="ij"))
        w = (gw[:, None] * gw[None]).ravel()
        JP, JQ = ((self.X[v[:, 1], 0] - self.X[v[:, 0], 0])[:, None] for v in (p, q))
        if n == 2:
            c = 2.0 - 2.0 * S_BAR
            xi = z ** (1.0 / c)
            yh = (1.0 - xi) * t
            sx, kx = self._value(p, (yh + xi)[:, None])
            sy, ky = self._value(p, yh[:, None])
            S = sx + sy
            g = (w * (1.0 - xi) * 2.0 / c * JP ** 2
                 * torch.exp((2.0 * S_BAR - S) / c * torch.log(z) + 0.5 * (kx + ky) - (1.0 + S) * torch.log(JP.abs())))
            f = torch.stack([-torch.ones_like(z), torch.ones_like(z)], 1)
            return torch.einsum("nq,qi,qj->nij", g, f, f)
        c, L = 3.0 - 2.0 * S_BAR, 0.0
        xi = z ** (1.0 / c)
        one = torch.ones_like(t)
        for a, b in ((one, t), (t, one)):
            sx, kx = self._value(p, (xi * a)[:, None])
            sy, ky = self._value(q, (xi * b)[:, None])
            S = sx + sy
            g = (w / c * JP.abs() * JQ.abs()
                 * torch.exp((2.0 * S_BAR - S) / c * torch.log(z) + 0.5 * (kx + ky)
                             - (1.0 + S) * torch.log((JP * a - JQ * b).abs())))
            f = torch.stack([b - a, a, -b], 1)
            L = L + torch.einsum("nq,qi,qj->nij", g, f, f)
        return L

    def _rules2(self, n, p, q, gx, gw):
        z, e1, e2, e3 = (a.ravel() for a in torch.meshgrid(gx, gx, gx, gx, indexing="ij"))
        w = torch.einsum("a,b,c,d->abcd", gw, gw, gw, gw).ravel()
        P, Q = self.X[p], self.X[q]
        JP, JQ = (torch.stack([V[:, 1] - V[:, 0], V[:, 2] - V[:, 1]], 2) for V in (P, Q))
        det = (torch.linalg.det(JP).abs() * torch.linalg.det(JQ).abs())[:, None]
        c, c2, one, L = 4.0 - 2.0 * S_BAR, 2.0 - 2.0 * S_BAR, torch.ones_like(z), 0.0
        xi, lz = z ** (1.0 / c), torch.log(z)
        if n == 1:
            maps = [((one, e1), (e2, e2 * e3), e2), ((e2, e2 * e3), (one, e1), e2)]
        elif n == 2:
            A, B = (1 - e1 * e2 * e3, e1 * e2 * (1 - e3)), (1 - e1 * e2, e1 * (1 - e2))
            maps = [((one, e1 * e3), B, e1 * e1), ((one, e1), A, e1 * e1 * e2), (B, (one, e1 * e2 * e3), e1 * e1 * e2),
                    (A, (one, e1), e1 * e1 * e2), ((A[0], e1 * (1 - e2 * e3)), (one, e1 * e2), e1 * e1 * e2)]
        else:
            t, e2 = e2, e2 ** (1.0 / c2)
            maps = [((one, 1 - e1 + e1 * e2), (1 - e1 * e2 * e3, 1 - e1), (e3, one)),
                    ((one, e1 * (1 - e2 + e2 * e3)), (1 - e1 * e2, e1 * (1 - e2)), (one, e3)),
                    ((1 - e1 * e2 * e3, e1 * (1 - e2 * e3)), (one, e1 * (1 - e2)), (-e3, 1 - e3))]
        for m in maps:
            a, b = torch.stack(m[0], 1), torch.stack(m[1], 1)
            sx, kx = self._value(p, xi[:, None] * a)
            sy, ky = self._value(q, xi[:, None] * b)
            S = sx + sy
            if n < 3:
                D = torch.einsum("nij,qj->nqi", JP, a) - torch.einsum("nij,qj->nqi", JQ, b)
                scale, extra = m[2] / c, (2.0 * S_BAR - S) / c * lz
                if n == 1:
                    f = [b[:, 0] - a[:, 0], a[:, 0] - a[:, 1], a[:, 1], b[:, 1] - b[:, 0], -b[:, 1]]
                else:
                    f = [b[:, 0] - a[:, 0], a[:, 0] - a[:, 1] - b[:, 0] + b[:, 1], a[:, 1], -b[:, 1]]
            else:
                r = torch.stack(m[2], 1)
                D = torch.einsum("nij,qj->nqi", JP, r)
                scale = 2.0 / (c * c2)
                extra = (2.0 * S_BAR - S) * (lz / c + torch.log(t) / c2) + (2.0 - S) * torch.log(e1)
                f = [-r[:, 0], r[:, 0] - r[:, 1], r[:, 1]]
            g = det * w * scale * torch.exp(extra + 0.5 * (kx + ky) - 0.5 * (2.0 + S) * torch.log((D ** 2).sum(2)))
            f = torch.stack(f, 1)
            L = L + torch.einsum("nq,qi,qj->nij", g, f, f)
        return L

    def matrix(self):
        """(A, rho)."""
        s, k = self.point_fields()
        nqi = self.nint * self.nq
        cw = torch.sparse_coo_tensor(self.psi.indices(), self.psi.values() * self.w[self.psi.indices()[0]],
                                     self.psi.shape).coalesce()
        cwt = cw.t().to_sparse_csr()
        A = torch.zeros((self.N, self.N), dtype=torch.float64, device="cuda")
        rho = self.tail_density(s, k)
        for i0, g in self.chunks(s, k):
            n = len(g)
            rho[i0:i0 + n] += g @ self.w
            row = torch.sparse.mm(cwt, g[:, :nqi].t().contiguous()).t()   # points x DoFs
            idx = cw.indices()
            on = (idx[0] >= i0) & (idx[0] < i0 + n)
            part = torch.sparse_coo_tensor(torch.stack([idx[1, on], idx[0, on] - i0]), cw.values()[on], (self.N, n))
            A -= 2.0 * torch.sparse.mm(part.coalesce().to_sparse_csr(), row.contiguous())
        col, val = self.dof[self.vid[:nqi]], 2.0 * (self.w[:nqi] * rho)[:, None, None]
        self._scatter(A, col, val * self.bary[:nqi, :, None] * self.bary[:nqi, None, :])
        for loc, L in self.singular():
            self._scatter(A, self.dof[loc], L)
        return A, rho

    @staticmethod
    def _scatter(A, col, L):
        i, j = col[:, :, None].expand_as(L), col[:, None, :].expand_as(L)
        on = (i >= 0) & (j >= 0)
        A.index_put_((i[on], j[on]), L[on], accumulate=True)


def exact(case, seed):
    geoms = [_geometry(*g) for g in _geometries(case)]
    meshes = _meshes(case)
    if max(m.n_dof for m in meshes) > EXACT_MAX_DOFS or max(len(g[2]) * (4 if g[0] == 3 else 3) for g in geoms) > EXACT_MAX_POINTS:
        return None
    task, outs = case["task"], []
    for i, (m, geom) in enumerate(zip(meshes, geoms)):
        s, k = _fields(case, geom[0], geom[1], seed + 100 * i)
        if task == "gradient":
            fs, fk = ((lambda x, v, b, n=f.nodal: (n[v] * b).sum(-1)) for f in (s, k))
        else:
            fs, fk = ((lambda x, v, b, f=f: _evaluate(f, x)) for f in (s, k))
        D = _Dense(m, geom, fs, fk, case["mesh"] == "interval")
        A, rho = D.matrix()
        if task == "apply":
            return _rhs(case, m, 0, seed) @ A.T
        if task in ("solve", "mixed"):
            F = _rhs(case, m, i, seed)
            outs.append(torch.linalg.solve(A, F.reshape(-1, m.n_dof).T).T.reshape(F.shape).contiguous())
            continue
        st = prepare(case, seed)   # the inputs alone are taken from it
        if task == "step":
            F = torch.zeros(m.n_dof, dtype=torch.float64, device="cuda")
            fv, nv = st.f[D.T], D.d + 1
            local = D.meas[:, None] / ((nv) * (nv + 1)) * (fv.sum(1, keepdim=True) + fv)
            col = D.dof[D.T]
            F.index_put_((col[col >= 0],), local[col >= 0], accumulate=True)
            return {"U": torch.linalg.solve(A, F), "rho": rho}
        U = torch.linalg.solve(A, st.F)
        Lam = torch.linalg.solve(A, 2.0 * st.mass * (U - st.u_obs))
        # the far field's sensitivities belong to the vertices next to the Chebyshev
        # nodes of the H^2 blocks: no value per vertex without them
        return {"U": U, "g_s": None, "g_logkappa": None, "g_F": Lam}
    return outs[0] if len(outs) == 1 else outs
