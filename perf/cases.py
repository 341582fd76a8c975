"""The calls whose speed matters to a user of this library, over the range in which they are made.

A user analyzes a sparsity pattern once and then factors and solves for every new set of values
on it (time steps, Newton steps, parameter sweeps). A case is one such call sequence:

* ``step``: new values, numeric factorization, solve (``sym_factor`` + ``sym_solve_multi``);
* ``solve``: new right-hand sides on a factor that is kept (``sym_solve_multi``);
* ``sparse``: the forward solve of a sparse right-hand side over its reach set
  (``sym_solve_lower_sparse``) on a factor that is kept;
* ``batch``: many value sets on one pattern (``sym_factor_batch`` + ``sym_solve_batch``).

``prepare`` makes the values on the GPU and the handle (pattern analyzed); a first call's graph
capture belongs to ``run``. Every case takes the library's default options except the precision
and, for graphs without a geometric ordering, the inspector's own ordering.

The right-hand sides are made from a known solution. Matrix values lie on a grid of 2^-20 (2^-12
for the vector problem) and solutions on one of 2^-16 (2^-10), so that every product and sum of
b = A x is exact in FP64 whatever its order, and the known x is the exact solution of the system
that the library is given.
"""
from __future__ import annotations

import functools
import itertools
import math

import numpy as np
import torch

import paper_1705_06575_gb300 as S

DEV = "cuda"


def listed():
    return [
        # One new right-hand side on a small 2D grid: the smallest call, all latency (the inner
        # loop of an explicit time stepper).
        dict(name="grid2d_64_solve", op="solve", problem="grid2d5", size=64, nrhs=1, precision="fp64"),
        # Factor and solve of the same grid: the smallest refactorization.
        dict(name="grid2d_64_step", op="step", problem="grid2d5", size=64, nrhs=1, precision="fp64"),
        # A sparse graph without geometry (circuit- or network-like), ordered by the inspector.
        dict(name="graph_3001_step", op="step", problem="graph", size=3001, degree=6, nrhs=1, precision="fp64"),
        # A medium 3D grid of odd side: ragged tiles everywhere.
        dict(name="grid3d_31_step", op="step", problem="grid3d7", size=31, nrhs=1, precision="fp64"),
        # A 27-point 3D grid (finite elements): wide supernodes on a medium problem.
        dict(name="grid3d27_40_step", op="step", problem="grid3d27", size=40, nrhs=1, precision="fp64"),
        # The library's headline workload and the largest case.
        dict(name="grid3d_64_step", op="step", problem="grid3d7", size=64, nrhs=4, precision="fp64"),
        # Many right-hand sides on a kept 3D factor (sources of an inverse problem).
        dict(name="grid3d_48_solve16", op="solve", problem="grid3d7", size=48, nrhs=16, precision="fp64"),
        # The headline workload in mixed precision: FP32 factor, refined to FP64 accuracy.
        dict(name="grid3d_64_mixed", op="step", problem="grid3d7", size=64, nrhs=4, precision="mixed"),
        # Elasticity-like: three unknowns per node, coefficient jumps, mixed precision.
        dict(name="vector_20_mixed", op="step", problem="vector27", size=20, nrhs=1, precision="mixed"),
        # A parameter sweep: 512 value sets on one 2D pattern.
        dict(name="batch_512x128", op="batch", problem="grid2d9", size=128, count=512, nrhs=1, precision="fp64"),
        # Domain decomposition: many subdomains of uneven size factored as one block-diagonal matrix.
        dict(name="union_48_step", op="step", problem="union", size=128, count=48, nrhs=1, precision="fp64"),
        # A column of A as right-hand side (one impulse): forward solve over its reach set.
        dict(name="sparse_48_forward", op="sparse", problem="grid3d7", size=48, nrhs=1, precision="fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed ones' ranges: sizes of the library's own pattern suites and configurations."""
    kind = rng.choice(["grid2d", "grid3d", "grid3d27", "solve2d", "solve3d", "mixed", "vector", "batch", "union", "graph", "sparse"])
    nrhs = rng.choice([1, 1, 2, 3, 4])
    fp64 = dict(nrhs=nrhs, precision="fp64")
    if kind == "grid2d":
        return dict(op="step", problem=rng.choice(["grid2d5", "grid2d9"]), size=_log_int(rng, 24, 160), **fp64)
    if kind == "grid3d":
        return dict(op="step", problem="grid3d7", size=_log_int(rng, 8, 56), **fp64)
    if kind == "grid3d27":
        return dict(op="step", problem="grid3d27", size=_log_int(rng, 8, 32), **fp64)
    if kind == "solve2d":
        return dict(op="solve", problem=rng.choice(["grid2d5", "grid2d9"]), size=_log_int(rng, 24, 160), **fp64)
    if kind == "solve3d":
        return dict(op="solve", problem="grid3d7", size=_log_int(rng, 12, 48), nrhs=rng.choice([1, 3, 5, 8, 16]), precision="fp64")
    if kind == "mixed":
        return dict(op="step", problem=rng.choice(["grid3d7", "grid3d27"]), size=_log_int(rng, 12, 40), nrhs=nrhs, precision="mixed")
    if kind == "vector":
        return dict(op="step", problem="vector27", size=_log_int(rng, 5, 20), nrhs=nrhs, precision=rng.choice(["fp64", "mixed"]))
    if kind == "batch":
        side = _log_int(rng, 16, 128)
        most = max(2, min(512, 512 * 128 * 128 // (2 * side * side)))
        return dict(op="batch", problem=rng.choice(["grid2d5", "grid2d9"]), size=side, count=_log_int(rng, 2, most), **fp64)
    if kind == "union":
        return dict(op="step", problem="union", size=_log_int(rng, 40, 128), count=_log_int(rng, 6, 48), **fp64)
    if kind == "graph":
        return dict(op="step", problem="graph", size=_log_int(rng, 800, 4000), degree=rng.randint(4, 12), **fp64)
    return dict(op="sparse", problem="grid3d7", size=_log_int(rng, 12, 48), nrhs=1, precision="fp64")


# ---- patterns ------------------------------------------------------------------------------


class Pattern:
    """A symmetric pattern as edges (u, v), its lower-triangle CSC form and an ordering."""

    def __init__(self, n, u, v, perm, dof=1, **more):
        self.n, self.perm, self.dof = int(n), perm, dof
        r, c = np.maximum(u, v), np.minimum(u, v)
        d = np.arange(n, dtype=np.int64)
        key = np.concatenate([d * n + d, c * n + r])
        order = np.argsort(key, kind="stable")
        key = key[order]
        self.Ap = np.zeros(n + 1, dtype=np.int64)
        np.cumsum(np.bincount(key // n, minlength=n), out=self.Ap[1:])
        self.Ai = (key % n).astype(np.int32)
        self.nnz = key.size
        self.u, self.v = u, v
        self.order = order  # CSC entry k holds value order[k] of [diagonal, edges]
        self.more = more
        self.at = {}

    def dev(self, name, make):
        if name not in self.at:
            self.at[name] = torch.as_tensor(make()).to(DEV)
        return self.at[name]


def _edges(dims, box):
    """Undirected edges of a star (5/7-point) or box (9/27-point) stencil, and their directions."""
    ids = np.arange(int(np.prod(dims)), dtype=np.int64).reshape(dims)
    us, vs, ds = [], [], []
    for o in itertools.product((-1, 0, 1), repeat=len(dims)):
        if o <= (0,) * len(dims) or (not box and sum(map(abs, o)) != 1):
            continue
        a = ids[tuple(slice(max(0, -k), d - max(0, k)) for k, d in zip(o, dims))].ravel()
        b = ids[tuple(slice(max(0, k), d - max(0, -k)) for k, d in zip(o, dims))].ravel()
        us.append(a)
        vs.append(b)
        ds.append(np.tile(np.asarray(o, dtype=np.float64) / math.sqrt(sum(k * k for k in o)), (a.size, 1)))
    return np.concatenate(us), np.concatenate(vs), np.concatenate(ds)


def _dissection(dims, dof=1):
    """Geometric nested dissection: halves of the longest side first, the plane between them last."""
    ids = np.arange(int(np.prod(dims)), dtype=np.int64).reshape(dims)
    out = []

    def cut(box):
        ext = [hi - lo for lo, hi in box]
        if min(ext) <= 0:
            return
        if max(ext) <= 2 or math.prod(ext) <= 8:
            out.append(ids[tuple(slice(lo, hi) for lo, hi in box)].ravel())
            return
        d = ext.index(max(ext))
        lo, hi = box[d]
        m = (lo + hi) // 2
        cut(box[:d] + [(lo, m)] + box[d + 1:])
        cut(box[:d] + [(m + 1, hi)] + box[d + 1:])
        out.append(ids[tuple(slice(a, b) for a, b in box[:d] + [(m, m + 1)] + box[d + 1:])].ravel())

    cut([(0, d) for d in dims])
    p = np.concatenate(out)
    return (p[:, None] * dof + np.arange(dof)).ravel().astype(np.int32)


@functools.lru_cache(maxsize=4)
def _pattern(problem, size, extra):
    if problem in ("grid2d5", "grid2d9", "grid3d7", "grid3d27"):
        dims = (size,) * int(problem[4])
        u, v, _ = _edges(dims, problem in ("grid2d9", "grid3d27"))
        return Pattern(math.prod(dims), u, v, _dissection(dims))
    if problem == "vector27":
        dims = (size,) * 3
        nu, nv, d = _edges(dims, True)
        blk = np.round((np.eye(3) + d[:, :, None] * d[:, None, :]) * 4096.0) / 4096.0
        a, b = np.meshgrid(np.arange(3), np.arange(3), indexing="ij")
        nodes = np.arange(size ** 3, dtype=np.int64)[:, None]
        u = np.concatenate([(3 * nu[:, None, None] + a).ravel(), (3 * nodes + [1, 2, 2]).ravel()])
        v = np.concatenate([(3 * nv[:, None, None] + b).ravel(), (3 * nodes + [0, 0, 1]).ravel()])
        return Pattern(3 * size ** 3, u, v, _dissection(dims, 3), dof=3, nu=nu, nv=nv, blk=blk, side=size)
    if problem == "union":
        sides = np.random.default_rng(extra).integers(32, size + 1, size=extra)
        us, vs, ps, n = [], [], [], 0
        for s in sides:
            u, v, _ = _edges((int(s), int(s)), False)
            us.append(u + n)
            vs.append(v + n)
            ps.append(_dissection((int(s), int(s))) + n)
            n += int(s) * int(s)
        return Pattern(n, np.concatenate(us), np.concatenate(vs), np.concatenate(ps).astype(np.int32))
    rng = np.random.default_rng(size)
    e = rng.integers(0, size, size=(size * extra // 2, 2))
    key = np.unique(e.min(1)[e[:, 0] != e[:, 1]] * size + e.max(1)[e[:, 0] != e[:, 1]])
    return Pattern(size, key // size, key % size, None)


def _of(case):
    return _pattern(case["problem"], case["size"], case.get("count" if case["problem"] == "union" else "degree", 0))


# ---- values --------------------------------------------------------------------------------


def _on(x, bits):
    return torch.round(x * 2.0 ** bits) / 2.0 ** bits


def _incident(P, w):
    """Sum of the edges' values at both ends of each edge; w is (..., edges)."""
    u, v = P.dev("u", lambda: P.u), P.dev("v", lambda: P.v)
    s = torch.zeros(w.shape[:-1] + (P.n,), dtype=torch.float64, device=DEV)
    return s.index_add_(-1, u, w).index_add_(-1, v, w)


def _values(case, P, gen):
    """(diagonal, edge values), each (count, .) for a batch."""
    problem, m = case["problem"], P.u.size
    lead = (case["count"],) if case["op"] == "batch" else ()
    uniform = lambda lo, hi, k: _on(lo + (hi - lo) * torch.rand(lead + (k,), dtype=torch.float64, device=DEV, generator=gen), 20)  # noqa: E731
    if problem in ("grid2d5", "union"):  # Laplacian with perturbed coefficients
        return 4.0 + uniform(0.0, 0.1, P.n), -uniform(0.9, 1.1, m)
    if problem == "vector27":  # coefficients 1, 1e2 and 1e4 by subdomain
        sub = 5
        k = -(-P.more["side"] // sub)
        c = torch.tensor([1.0, 1e2, 1e4], dtype=torch.float64, device=DEV)[torch.randint(0, 3, (k, k, k), device=DEV, generator=gen)]
        g = P.dev("g", lambda: np.arange(P.more["side"]) // sub)
        c = c[g[:, None, None], g[None, :, None], g[None, None, :]].reshape(-1)
        nu, nv = P.dev("nu", lambda: P.more["nu"]), P.dev("nv", lambda: P.more["nv"])
        blk = torch.minimum(c[nu], c[nv])[:, None, None] * P.dev("blk", lambda: P.more["blk"])
        D = torch.zeros((c.numel(), 3, 3), dtype=torch.float64, device=DEV).index_add_(0, nu, blk).index_add_(0, nv, blk)
        diag = torch.diagonal(D, dim1=1, dim2=2) + (2.0 ** -10 * c)[:, None]
        inner = torch.stack([D[:, 1, 0], D[:, 2, 0], D[:, 2, 1]], dim=1)
        return diag.reshape(-1), torch.cat([-blk.reshape(-1), inner.reshape(-1)])
    w = uniform(0.5, 2.0, m)
    s = _incident(P, w)
    if problem == "grid2d9":
        return _on(1.05 * s, 20), -w
    if problem == "graph":
        return _on(1.25 * s, 20) + (s == 0), -w
    return s + _on(torch.tensor(1e-3, dtype=torch.float64), 20).item(), -w  # conductivity


def _solution(case, P, gen):
    lead = (case["count"],) if case["op"] == "batch" else ()
    return _on(torch.randn(lead + (case["nrhs"], P.n), dtype=torch.float64, device=DEV, generator=gen), 10 if case["problem"] == "vector27" else 16)


def _inputs(case, seed):
    P = _of(case)
    gen = torch.Generator(device=DEV).manual_seed(int(seed))
    diag, w = _values(case, P, gen)
    Ax = torch.cat([diag, w], dim=-1).index_select(-1, P.dev("order", lambda: P.order)).contiguous()
    return P, diag, w, Ax, gen


def _product(P, diag, w, x):
    """A x for x (..., nrhs, n), exact on the grids above."""
    u, v = P.dev("u", lambda: P.u), P.dev("v", lambda: P.v)
    b = diag[..., None, :] * x
    for k in range(x.shape[-2]):
        b[..., k, :].index_add_(-1, u, w * x[..., k, :].index_select(-1, v))
        b[..., k, :].index_add_(-1, v, w * x[..., k, :].index_select(-1, u))
    return b


def _solver(case, P):
    return S.Solver(P.n, P.Ap, P.Ai, P.perm, precision=case["precision"], ordering="auto" if P.perm is None else None)


def prepare(case, seed):
    P, diag, w, Ax, gen = _inputs(case, seed)
    st = dict(case=case, n=P.n, nnz=P.nnz, Ax=Ax, solver=_solver(case, P))
    if case["op"] == "sparse":  # one column of A: its rows in the lower triangle and their values
        j = P.n // 3 + case["size"] // 2
        lo, hi = int(P.Ap[j]), int(P.Ap[j + 1])
        st["solver"].factor(Ax)
        st["reach"] = S.Reach(st["solver"].h, P.Ai[lo:hi])
        st["b"] = Ax[lo:hi].clone()
        st["x"] = torch.empty(st["reach"].size(), dtype=torch.float64, device=DEV)
        return st
    st["b"] = _product(P, diag, w, _solution(case, P, gen))
    if case["op"] == "solve":
        st["solver"].factor(Ax)
    if case["op"] == "batch":
        st["x"] = torch.empty_like(st["b"])
    return st


def run(st):
    case, s = st["case"], st["solver"]
    if case["op"] == "sparse":
        st["reach"].solve(st["b"], st["x"])
        return st["x"]
    if case["op"] == "solve":
        return s.solve(st["b"])
    if case["op"] == "batch":
        n, nb, nrhs = st["n"], case["count"], case["nrhs"]
        S.sym_factor_batch(s.h, nb, st["Ax"], st["nnz"])
        S.sym_solve_batch(s.h, nb, nrhs, st["b"], n, n * nrhs, st["x"], n, n * nrhs)
        return st["x"]
    s.factor(st["Ax"])
    return s.solve(st["b"])


def exact(case, seed):
    """The known solution that the right-hand sides were made from (none for the forward solve
    alone, whose exact value needs the factor)."""
    if case["op"] == "sparse":
        return None
    P, _, _, _, gen = _inputs(case, seed)
    return _solution(case, P, gen)


@functools.lru_cache(maxsize=32)
def _counts(problem, size, extra):
    P = _pattern(problem, size, extra)
    i = S.Solver(P.n, P.Ap, P.Ai, P.perm, host_only=True, ordering="auto" if P.perm is None else None).info()
    return P.n, P.nnz, i.nnz_l, i.flops


def work(case):
    """Each value of A, b and x once, and each entry of the exact pattern of L once: written by a
    factorization, read by a solve. Factor flops are sum c_j^2, a solve takes 4 per entry of L and
    right-hand side."""
    n, nnz, nnz_l, flops = _counts(case["problem"], case["size"], case.get("count" if case["problem"] == "union" else "degree", 0))
    k, many = case["nrhs"], case.get("count", 1) if case["op"] == "batch" else 1
    if case["op"] == "sparse":  # a column's reach is a path of the tree: about the top separators
        top = case["size"] ** 2
        return {"bytes": 8.0 * top * top / 2, "flops": float(top * top)}
    if case["op"] == "solve":
        return {"bytes": 8.0 * nnz_l + 16.0 * n * k, "flops": 4.0 * nnz_l * k}
    return {"bytes": many * (8.0 * nnz + 8.0 * nnz_l + 16.0 * n * k), "flops": many * (flops + 4.0 * nnz_l * k)}
