"""What a user has this library do, as cases that can be timed and checked.

A case is a dict of plain values; its "kind" says which public entry point it
goes through:

  solve     Problem.solve: Algorithm 1, 2 or 3 on one SDP or on a batch, for a
            fixed number of iterations from the cold start (eps = 0), with the
            solution and the residual history read back
  project   psd_project: the batched projection on its own, orders 1..128
  large     psd_project_large: the projection of blocks above order 128
  grad      unrolled_primal forward and backward: gradients through Algorithm 1
  complete  Problem.complete: the maximum-determinant completion

`prepare` makes the inputs from the seed and sets up the handle that a program
keeps (preprocessing, workspace, upload); `run` is one call.  A solve in the
FP32-projection form keeps its clique state in float32, so its solution, and
the gradients of an unrolled FP32 solve, are handed on in float32; the FP64
form's and the completion's stay float64.  `exact` restates each path in
float64 numpy.  Sizes are those of paper_1707_05058_gb300/workloads.py and of
the tests, or ranges around them.
"""
from __future__ import annotations

import math
import os
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

from paper_1707_05058_gb300 import cdsdp, workloads

SOLVE = dict(kind="solve", family="arrow", count=1, form="primal", precision="fp32", iters=64, adaptive=1, scale=-1,
             shapes=0, density=0.05)


def listed():
    return [
        # the smallest problem a user solves (n = 55, five cliques of order 15): launches and latency
        dict(SOLVE, name="solve_small", l=5, d=10, h=5, m=30, density=1.0, iters=200, adaptive=0),
        # one banded SDP, n = 2000: 1990 small cliques of order 11, everything in L2
        dict(SOLVE, name="solve_banded", family="band", n=2000, w=10, m=500, iters=120),
        # a batch of uneven block-arrow SDPs in one call, each with its own penalty: 800 cliques of order 20..60
        dict(SOLVE, name="solve_batch", count=16, shapes=3707, iters=48),
        # Algorithm 2 with every A_i dense on the pattern (the affine step of the paper's Section 7.4 table)
        dict(SOLVE, name="solve_dual_dense", form="dual", l=100, d=10, h=20, m=409, density=1.0),
        # Algorithm 3 on a batch scaled SDP by SDP: the form that also answers infeasible problems
        dict(SOLVE, name="solve_hsde_batch", form="hsde", count=8, shapes=3707, scale=4, adaptive=0,
             iters=48),
        # the FP64 form, for users who need more digits: four banded SDPs of order-9 cliques
        dict(SOLVE, name="solve_fp64", family="band", count=4, n=500, w=8, m=200, precision="fp64"),
        # MaxCut on a random graph: fill, merged cliques, one clique of about 0.36 n on the tensor cores
        dict(SOLVE, name="solve_maxcut", family="maxcut", n=2500, iters=12, adaptive=0, shapes=4706),
        # projection of a ragged batch of small blocks, the cliques of a sparse problem
        dict(kind="project", name="project_small", p=4096, lo=1, hi=32, shapes=11, precision="fp32"),
        # projection of mid-size blocks, one thread block each
        dict(kind="project", name="project_mid", p=600, lo=33, hi=64, shapes=12, precision="fp32"),
        # projection of a few large blocks, the clique orders of the paper's non-chordal problems and above
        dict(kind="large", name="project_large", p=4, lo=129, hi=1500, shapes=13),
        # gradients through 50 iterations on a batch of banded SDPs
        dict(kind="grad", name="grad_banded", family="band", count=16, n=500, w=8, m=200, iters=50, every=10),
        # completion of a partial matrix on a band, dense n x n result
        dict(kind="complete", name="complete_banded", family="band", count=1, n=2000, w=10),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _band(rng, n, w, m):
    """A band with at most a quarter as many constraints as entries (A has to
    have full row rank, and every A_i an entry)."""
    ne = n * (w + 1) - w * (w + 1) // 2
    return dict(family="band", n=n, w=w, m=max(1, min(m, ne // 4 if ne > 400 else ne // 40)))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["project"] * 3 + ["large", "grad", "complete"])
    shapes = rng.randrange(1, 1 << 20)
    if kind == "project":
        lo, hi = rng.choice([(1, 8), (1, 16), (5, 32), (11, 11), (20, 60), (33, 48), (33, 64), (50, 128)])
        precision = rng.choice(["fp32", "fp32", "fp64"]) if hi <= 32 else "fp32"
        p = _log(rng, 1, 4096 if hi <= 16 else 2048 if hi <= 32 else 400 if hi <= 64 else 100)
        return dict(kind=kind, p=p, lo=lo, hi=hi, shapes=shapes, precision=precision)
    if kind == "large":
        return dict(kind=kind, p=rng.randrange(1, 5), lo=129, hi=_log(rng, 150, 1400), shapes=shapes)
    if kind == "grad":
        return dict(_band(rng, _log(rng, 100, 500), rng.randrange(3, 13), _log(rng, 10, 150)), kind=kind,
                    count=rng.randrange(1, 13), iters=rng.randrange(10, 50), every=rng.randrange(5, 20))
    if kind == "complete":
        if rng.random() < 0.5:
            return dict(kind=kind, family="band", count=_log(rng, 1, 16), n=_log(rng, 60, 1000), w=rng.randrange(1, 21))
        return dict(kind=kind, family="arrow", count=_log(rng, 1, 12), l=rng.randrange(5, 60), d=rng.randrange(4, 21),
                    h=rng.randrange(2, 21))
    form = rng.choice(["primal", "primal", "dual", "hsde"])
    precision = rng.choice(["fp32", "fp32", "fp32", "fp64"])
    base = dict(SOLVE, form=form, precision=precision, shapes=shapes, iters=rng.randrange(20, 48),
                adaptive=0 if form == "hsde" else rng.randrange(2), scale=4 if form == "hsde" else -1)
    family = rng.choice(["band", "band", "arrow", "batch", "maxcut"])
    if family == "band":
        return dict(base, count=_log(rng, 1, 6), **_band(rng, _log(rng, 100, 900), rng.randrange(3, 15),
                                                         _log(rng, 10, 300)))
    if family == "maxcut":
        return dict(base, family="maxcut", form="primal", precision="fp32", scale=-1, adaptive=0,
                    n=_log(rng, 300, 2000), iters=rng.randrange(6, 12))
    if family == "arrow":
        l, d, h = rng.randrange(3, 40), rng.randrange(4, 21), rng.randrange(2, 13)
        ne = l * d * (d + 1) // 2
        return dict(base, l=l, d=d, h=h, m=_log(rng, 10, min(200, max(12, ne // 4))),
                    density=rng.choice([0.05, 0.2, 1.0]) if ne > 400 else 1.0)
    return dict(base, precision="fp32", count=rng.randrange(2, 7 if form == "hsde" else 11))


# ---- inputs ------------------------------------------------------------------

def _sdp_shapes(case):
    """(l, d, h, m) of every block-arrow SDP of the case; a batch has the
    batched workload's ranges."""
    if "l" in case:
        return [(case["l"], case["d"], case["h"], case.get("m", 1))] * case["count"]
    rng = np.random.default_rng(case["shapes"])
    r = lambda lo, hi: int(rng.integers(lo, hi + 1))  # noqa: E731
    return [(r(10, 100), r(10, 40), r(10, 20), r(50, 400)) for _ in range(case["count"])]


def _problems(case, seed):
    s0 = 1000 * int(seed) + 1
    if case["family"] == "maxcut":
        return [_reweighted(workloads.maxcut(case["n"], 6, 1 + case["shapes"]), s0)]
    if case["family"] == "band":
        return [workloads.banded(case["n"], case["w"], case["m"], s0 + i) for i in range(case["count"])]
    density = None if case["density"] >= 1.0 else case["density"]
    return [workloads.block_arrow(l, d, h, m, s0 + i, density=density)
            for i, (l, d, h, m) in enumerate(_sdp_shapes(case))]


def _reweighted(p, seed):
    """The same graph (the case's) with U(0, 1) edge weights of this seed: C = -L / 4."""
    edge = p.C_row != p.C_col
    er, ec = p.C_row[edge], p.C_col[edge]
    wts = np.random.default_rng(seed).random(er.size).astype(np.float32).astype(np.float64)
    deg = np.bincount(er, weights=wts, minlength=p.n) + np.bincount(ec, weights=wts, minlength=p.n)
    p.C_val = np.where(edge, 0.0, -deg[p.C_row] / 4.0)
    p.C_val[edge] = wts / 4.0
    return p


def _pattern_problems(case):
    """SDPs that carry only a pattern (m = 1), for the completion."""
    if case["family"] == "band":
        return [workloads.banded(case["n"], case["w"], 1, 7 + i) for i in range(case["count"])]
    return [workloads.block_arrow(l, d, h, 1, 7 + i) for i, (l, d, h, _) in enumerate(_sdp_shapes(case))]


def _orders(case):
    """Block orders, log-uniform over the case's range; the largest occurs."""
    rng = np.random.default_rng(case["shapes"])
    s = np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"] + 1), case["p"])).astype(np.int64)
    s = np.clip(s, case["lo"], case["hi"])
    s[0] = case["hi"]
    return s


def _blocks(case, seed):
    """Packed random symmetric blocks with a spread-out spectrum of both signs
    (what a projection meets: a positive part and a negative part), float32
    values."""
    sizes = _orders(case)
    off = np.concatenate([[0], np.cumsum(sizes * (sizes + 1) // 2)])
    rng = np.random.default_rng(int(seed) + 17)
    return rng.standard_normal(int(off[-1])).astype(np.float32), off, sizes


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        ps = _problems(case, seed)
        scale = case["scale"] if case["scale"] >= 0 else None
        if case["family"] == "maxcut":
            P = cdsdp.Problem(ps[0], merge_cliques=True)
        elif len(ps) == 1:
            P = cdsdp.Problem(ps[0], scale_passes=scale)
        else:
            P = cdsdp.Problem.batch(ps, scale_passes=scale)
        P.bind(max_iter=case["iters"])
        return dict(kind=kind, P=P, form=case["form"],
                    opts=dict(eps=0.0, max_iter=case["iters"], precision=case["precision"],
                              adaptive_rho=case["adaptive"]))
    if kind == "project":
        W, off, sizes = _blocks(case, seed)
        dt = torch.float64 if case["precision"] == "fp64" else torch.float32
        return dict(kind=kind, W=torch.tensor(W, dtype=dt, device="cuda"),
                    off=torch.tensor(off, dtype=torch.int32, device="cuda"),
                    sizes=torch.tensor(sizes, dtype=torch.int32, device="cuda"))
    if kind == "large":
        W, off, sizes = _blocks(case, seed)
        return dict(kind=kind, W=torch.tensor(W, device="cuda"), sizes=sizes.astype(np.int32))
    if kind == "grad":
        ps = _problems(case, seed)
        P = cdsdp.Problem(workloads.direct_sum(ps)).bind(max_iter=case["every"])
        c, b = P.problem_data()
        return dict(kind=kind, P=P, c=c.requires_grad_(), b=b.requires_grad_(),
                    g=torch.tensor(_cotangent(c.numel(), seed), device="cuda"), iters=case["iters"],
                    every=case["every"])
    ps = _pattern_problems(case)
    P = cdsdp.Problem(ps[0]) if len(ps) == 1 else cdsdp.Problem.batch(ps)
    scratch, elems, _ = P.completion_sizes()
    X = np.concatenate([_partial(p, seed, i) for i, p in enumerate(ps)])
    return dict(kind=kind, P=P, X=torch.tensor(X, device="cuda"),
                scratch=torch.empty(scratch, dtype=torch.uint8, device="cuda"),
                out=torch.empty(elems, dtype=torch.float64, device="cuda"))


def _cotangent(n, seed):
    return np.random.default_rng(int(seed) + 5).standard_normal(n)


def _partial(p, seed, i):
    """Values on the pattern of p (column by column) of a positive definite matrix."""
    r, c = _entries(p)
    return workloads.pd_on_pattern(p.n, r, c, 1000 * int(seed) + i)


def run(state):
    kind = state["kind"]
    if kind == "solve":
        out = state["P"].solve(state["form"], **state["opts"])
        res = {k: out[k] for k in ("X", "y", "Z", "hist")}
        if state["opts"]["precision"] == "fp32":
            res = {k: v.astype(np.float32) for k, v in res.items()}
        return res
    if kind == "project":
        return cdsdp.psd_project(state["W"], state["off"], state["sizes"])
    if kind == "large":
        return cdsdp.psd_project_large(state["W"], state["sizes"])
    if kind == "grad":
        x = cdsdp.unrolled_primal(state["P"], state["c"], state["b"], iters=state["iters"], ckpt_every=state["every"])
        cbar, bbar = torch.autograd.grad(x, (state["c"], state["b"]), state["g"])
        return {"x": x.detach().float(), "cbar": cbar.float(), "bbar": bbar.float()}
    W, logdet = state["P"].complete(state["X"], scratch=state["scratch"], out=state["out"])
    return {"W": W, "logdet": logdet}


# ---- work ----------------------------------------------------------------------

def _sizes(case):
    """Per SDP (cliques, clique order, pattern entries, nonzeros of A, m)."""
    if case["family"] == "maxcut":  # the merged extension's largest clique is about 0.36 n; it dominates
        s = int(0.36 * case["n"])
        return [(1, s, s * (s + 1) // 2, case["n"], case["n"])]
    if case["family"] == "band":
        n, w = case["n"], case["w"]
        ne = n * (w + 1) - w * (w + 1) // 2
        m = case.get("m", 1)
        return [(n - w, w + 1, ne, 0.05 * m * ne, m)] * case["count"]
    out = []
    for l, d, h, m in _sdp_shapes(case):
        ne = l * d * (d + 1) // 2 + h * (h + 1) // 2 + h * l * d
        out.append((l, d + h, ne, case.get("density", 1.0) * m * ne, m))
    return out


def work(case):
    """Bytes and operations of one call.  A projection of order s is counted
    as 10 s^3 (9 s^3 for the eigendecomposition, s^3 for the product).  An
    iteration has to go over A twice (A t, then A^T y, 12 B a nonzero), over
    the cached inverse (not for MaxCut, where it is diagonal) and over the
    clique state and the pattern vectors (read and written once)."""
    kind = case["kind"]
    if kind in ("project", "large"):
        s = _orders(case).astype(float)
        item = 8 if case.get("precision") == "fp64" else 4
        return {"bytes": float(2 * item * np.sum(s * (s + 1) / 2)), "flops": float(np.sum(10 * s ** 3))}
    if kind == "complete":
        ns = [case["n"]] * case["count"] if case["family"] == "band" else [l * d + h for l, d, h, _ in _sdp_shapes(case)]
        b = sum(8.0 * n * n for n in ns) + sum(8.0 * ne for _, _, ne, _, _ in _sizes(case))
        f = sum(float(n) * n * (s - 1) for n, (_, s, _, _, _) in zip(ns, _sizes(case)))
        return {"bytes": b, "flops": f}
    item = 8 if case.get("precision") == "fp64" else 4
    b = f = 0.0
    for p, s, ne, nnz, m in _sizes(case):
        inv = 0 if case["family"] == "maxcut" else m * m
        b += 24 * nnz + 8 * inv + p * s * (s + 1) / 2 * item * 4 + 8 * 4 * ne
        f += p * 10.0 * s ** 3 + 4 * nnz + 2 * inv
    passes = case["iters"] * (3 if kind == "grad" else 1)  # forward, replay, reverse
    return {"bytes": b * passes, "flops": f * passes}


# ---- the same paths in float64 numpy -------------------------------------------

def _entries(p):
    """Rows and columns of the pattern, lower triangle, column by column."""
    o = np.lexsort((p.C_row, p.C_col))
    return p.C_row[o].astype(np.int64), p.C_col[o].astype(np.int64)


def _cliques(case, k):
    """Vertices of every maximal clique of SDP k, one row each."""
    if case["family"] == "band":
        return np.arange(case["n"] - case["w"])[:, None] + np.arange(case["w"] + 1)[None, :]
    l, d, h, _ = _sdp_shapes(case)[k]
    head = np.broadcast_to(l * d + np.arange(h), (l, h))
    return np.concatenate([np.arange(l * d).reshape(l, d), head], axis=1)


_THREADS = max(1, min(16, os.cpu_count() or 1))


def _each(f, items):
    """[f(x) for x in items], several at a time."""
    with ThreadPoolExecutor(_THREADS) as pool:
        return list(pool.map(f, items))


def _eigh(B):
    """Eigenvalues and eigenvectors of a stack of symmetric matrices (large stacks in parts, several at a time)."""
    if len(B) < 512:
        return np.linalg.eigh(B)
    res = _each(np.linalg.eigh, np.array_split(B, 16))
    return np.concatenate([r[0] for r in res]), np.concatenate([r[1] for r in res])


def _psd(B):
    lam, V = _eigh(B)
    return np.matmul(V * np.maximum(lam, 0.0)[:, None, :], np.swapaxes(V, 1, 2))


class _Plain:
    """One SDP on its lower pattern: clique blocks as full symmetric matrices."""

    def __init__(self, p, cliques, scale):
        self.n, self.m = p.n, p.m
        r, c = _entries(p)
        self.ne = r.size
        key = c * p.n + r
        ent = lambda a, b: np.searchsorted(key, np.minimum(a, b) * p.n + np.maximum(a, b))  # noqa: E731
        self.A = np.zeros((p.m, self.ne))
        self.A[p.A_con, ent(p.A_row.astype(np.int64), p.A_col.astype(np.int64))] = p.A_val
        self.c = np.zeros(self.ne)
        self.c[ent(p.C_row.astype(np.int64), p.C_col.astype(np.int64))] = p.C_val
        self.b = p.b.astype(float).copy()
        self.w = np.where(r == c, 1.0, 2.0)
        self.dd, self.e, self.tau, self.sigma = np.ones(self.ne), np.ones(p.m), 1.0, 1.0
        if scale >= 0:
            self._scale(r, c, scale)
        self.g = ent(cliques[:, :, None].astype(np.int64), cliques[:, None, :].astype(np.int64))
        s = cliques.shape[1]
        self.low = np.tril(np.ones((s, s), bool))
        self.D = self.scatter(np.ones(self.g.shape))
        # products with A W, A and A^T: sparse rows where that is less to read
        self.mul_aw, self.mul_a, self.mul_at = (self._product(M) for M in (self.A * self.w, self.A, self.A.T))

    @staticmethod
    def _product(M):
        if np.count_nonzero(M) > 0.2 * M.size:
            return lambda v: M @ v
        rows, cols = np.nonzero(M)
        vals, full = M[rows, cols], np.unique(rows)
        at = np.searchsorted(rows, full)

        def mul(v):
            out = np.zeros(M.shape[0])
            if full.size:
                out[full] = np.add.reduceat(vals * v[cols], at)
            return out
        return mul

    def _scale(self, r, c, passes):
        d, e = np.ones(self.n), np.ones(self.m)
        for _ in range(passes):
            a = e[:, None] * (d[r] * d[c]) * self.A
            nrm = np.sqrt((a * a) @ self.w)
            e = np.clip(e / np.sqrt(np.where(nrm > 0, nrm, 1.0)), 1e-4, 1e4)
            col = np.abs(e[:, None] * self.A).max(axis=0) * d[r] * d[c]
            top = np.zeros(self.n)
            np.maximum.at(top, r, col)
            np.maximum.at(top, c, col)
            d = np.clip(d / np.sqrt(np.where(top > 0, top, 1.0)), 1e-4, 1e4)
        self.dd, self.e = d[r] * d[c], e
        nb = np.linalg.norm(e * self.b)
        nc = math.sqrt(float(self.w @ (self.dd * self.c) ** 2))
        self.tau, self.sigma = 1.0 / nb if nb > 0 else 1.0, 1.0 / nc if nc > 0 else 1.0
        self.A = e[:, None] * self.dd * self.A
        self.b = self.tau * e * self.b
        self.c = self.sigma * self.dd * self.c

    def scatter(self, B):
        """Sum of the cliques' lower triangles on the pattern."""
        return np.bincount(self.g[:, self.low].ravel(), weights=B[:, self.low].ravel(), minlength=self.ne)

    def unscale(self, X, y, Z):
        return X * self.dd / self.tau, y * self.e / self.sigma, Z / (self.dd * self.sigma)

    def first_order(self, form, iters, adapt):
        """Algorithms 1 and 2; returns X, y, Z and the per-iteration
        (eps_c, eps_lambda, rho, <C, X>, b^T y)."""
        b, c, g = self.b, self.c, self.g
        di = 1.0 / self.D
        inv = np.linalg.inv((self.A * (self.w * di)) @ self.A.T)
        nrm = np.linalg.norm
        zero = np.zeros(g.shape)
        rho, hist = 1.0, []
        xk, lam, v = zero, zero, zero
        for it in range(iters):
            if form == "dual":
                old, xk = xk, _psd(v - lam / rho)
                t = di * (c - self.scatter(xk + lam / rho))
                y = inv @ (self.mul_aw(t) + b / rho)
                x = t - di * self.mul_at(y)
                v = xk + lam / rho + x[g]
                lam = lam + rho * (xk - v)
                other, cx, by = v, -rho * float((self.w * c) @ x), float(b @ y)
            else:
                t = di * (self.scatter(xk + lam / rho) - c / rho)
                y = inv @ (self.mul_aw(t) - b)
                x = t - di * self.mul_at(y)
                hx = x[g]
                old, xk = xk, _psd(hx - lam / rho)
                lam = lam + rho * (xk - hx)
                other, cx, by = hx, float((self.w * c) @ x), -rho * float(b @ y)
            ec = nrm(xk - other) / max(nrm(xk), nrm(other), 1e-300)
            el = rho * nrm(xk - old) / max(nrm(lam), 1e-300)
            hist.append((ec, el, rho, 0.0, cx, by, 0.0, 0.0))
            if adapt and it + 1 < iters:
                rho = rho * 2.0 if ec >= 10.0 * el else rho / 2.0 if el >= 10.0 * ec else rho
        if form == "dual":
            return (*self.unscale(-rho * x, y, self.scatter(xk)), np.array(hist))
        return (*self.unscale(x, -rho * y, self.scatter(lam)), np.array(hist))

    def hsde(self, iters):
        """Algorithm 3; returns X, y, Z and the per-iteration
        (eps_p, eps_d, eps_g, eps_c, <C, X>, b^T y, tau, kappa)."""
        b, c, g, w = self.b, self.c, self.g, self.w
        pi = 1.0 / (1.0 + 0.5 * self.D)
        inv = np.linalg.inv(np.eye(self.m) + (self.A * (w * pi)) @ self.A.T)
        nrm = np.linalg.norm

        def solve(n11, n21, half):
            q = (n11 + self.mul_at(n21) + half) * pi
            s11 = q - pi * self.mul_at(inv @ self.mul_aw(q))
            as11 = self.mul_aw(s11)
            return s11, n21 - as11, as11
        zx, zy, azx = solve(c, -b, 0.0)
        z0 = float((w * c) @ zx) - float(b @ zy)
        zx, zy, azx = zx / (1 + z0), zy / (1 + z0), azx / (1 + z0)
        us = vz = ut = np.zeros(g.shape)
        ux, uy, tau, kappa, hist = np.zeros(self.ne), np.zeros(self.m), 1.0, 1.0, []
        nb, nc = nrm(b), math.sqrt(float(w @ c ** 2))
        for _ in range(iters):
            w2 = tau + kappa
            s11, s21, as11 = solve(ux - w2 * c, uy + w2 * b, 0.5 * self.scatter(us + vz + ut))
            gam = float((w * c) @ s11) - float(b @ s21)
            hat = w2 + gam * (1.0 - z0 / (1 + z0))
            tau_new = max(0.0, hat - kappa)
            tau, kappa = tau_new, kappa - hat + tau_new
            hs, zs = s11[g], 0.5 * zx[g]
            s12 = 0.5 * (us + vz - ut + hs)
            uh, ut = s12 - gam * zs, ut - hs + s12 + gam * zs
            us = _psd(uh - vz)
            vz = vz - uh + us
            ux, uy = s11 - gam * zx, s21 - gam * zy
            hux = ux[g]
            rp = nrm(as11 - gam * azx - tau * b)
            rd = math.sqrt(float(w @ (self.mul_at(uy) + self.scatter(vz) - tau * c) ** 2))
            cx, by = float((w * c) @ ux), float(b @ uy)
            if tau > 0:
                cx, by = cx / tau, by / tau
                ec = max(nrm(us - hux) / max(nrm(us), nrm(hux), 1e-300),
                         nrm(vz - ut) / max(nrm(vz), nrm(ut), 1e-300))
                hist.append((rp / tau / (1 + nb), rd / tau / (1 + nc), abs(cx - by) / (1 + abs(cx) + abs(by)), ec,
                             cx, by, tau, kappa))
            else:
                hist.append((rd, rp, by, cx, 0.0, 0.0, tau, kappa))
        k = tau if tau > 0 else 1.0
        return (*self.unscale(ux / k, uy / k, self.scatter(vz) / k), np.array(hist))

    def unrolled(self, iters, gout):
        """x_N of Algorithm 1 with rho = 1 and the gradients of <gout, x_N>
        with respect to c and b (Daleckii-Krein adjoint of the projections)."""
        b, c, g = self.b, self.c, self.g
        di = 1.0 / self.D
        inv = np.linalg.inv((self.A * (self.w * di)) @ self.A.T)
        xk = lam = np.zeros(g.shape)
        tape = []
        for _ in range(iters):
            t = di * (self.scatter(xk + lam) - c)
            x = t - di * self.mul_at(inv @ (self.mul_aw(t) - b))
            hx = x[g]
            L, V = _eigh(hx - lam)
            tape.append((L, V))
            xk = np.matmul(V * np.maximum(L, 0.0)[:, None, :], np.swapaxes(V, 1, 2))
            lam = lam + xk - hx
        s = g.shape[1]
        wp = np.where(np.eye(s, dtype=bool), 1.0, 2.0)
        xb = lb = np.zeros(g.shape)  # packed adjoints, kept on both triangles
        cb, bb = np.zeros(self.ne), np.zeros(self.m)
        for n in range(iters - 1, -1, -1):
            L, V = tape[n]
            f = np.maximum(L, 0.0)
            dl = L[:, :, None] - L[:, None, :]
            tie = np.where(L > 0, 1.0, np.where(L < 0, 0.0, 0.5))
            gam = np.where(dl == 0, np.broadcast_to(tie[:, :, None], dl.shape),
                           (f[:, :, None] - f[:, None, :]) / np.where(dl == 0, 1.0, dl))
            Vt = np.swapaxes(V, 1, 2)
            G = (xb + lb) / wp
            wb = wp * np.matmul(V, np.matmul(gam * np.matmul(Vt, np.matmul(G, V)), Vt))
            xbar = self.scatter(wb - lb) + (gout if n == iters - 1 else 0.0)
            prev = lb - wb
            rb = inv @ -self.mul_a(xbar * di)
            bb -= rb
            sb = (xbar + self.w * self.mul_at(rb)) * di
            cb -= sb
            xb, lb = sb[g], prev + sb[g]
        return x, cb, bb


def _complete(p, cliques, X):
    """Dense maximum-determinant completion along the natural vertex order
    (perfect for bands and block-arrows) and its log det."""
    r, c = _entries(p)
    W = np.zeros((p.n, p.n))
    W[r, c] = X
    W[c, r] = X
    order = np.argsort(c, kind="stable")
    start = np.searchsorted(c[order], np.arange(p.n + 1))
    logdet = 0.0
    for k in range(p.n - 1, -1, -1):
        N = r[start[k]:start[k + 1]][1:]
        if N.size == 0:
            logdet += math.log(W[k, k])
            continue
        t = np.linalg.solve(W[np.ix_(N, N)], W[N, k])
        logdet += math.log(W[k, k] - W[k, N] @ t)
        free = np.ones(p.n, bool)
        free[:k + 1] = False
        free[N] = False
        W[free, k] = W[np.ix_(free, N)] @ t
        W[k, free] = W[free, k]
    return W, logdet


def exact(case, seed):
    kind = case["kind"]
    if kind in ("project", "large"):
        W, off, sizes = _blocks(case, seed)
        out = np.empty(W.size)
        for s in np.unique(sizes):
            ks = np.flatnonzero(sizes == s)
            i, j = np.tril_indices(s)
            i, j = i[np.lexsort((i, j))], j[np.lexsort((i, j))]
            idx = off[ks][:, None] + np.arange(i.size)[None, :]
            B = np.zeros((ks.size, s, s))
            B[:, i, j] = W[idx]
            B[:, j, i] = W[idx]
            out[idx] = _psd(B)[:, i, j]
        return out
    if kind == "complete":
        res = [_complete(p, _cliques(case, k), _partial(p, seed, k)) for k, p in enumerate(_pattern_problems(case))]
        return {"W": np.concatenate([r[0].ravel() for r in res]), "logdet": np.array([r[1] for r in res])}
    if case["family"] == "maxcut":
        return None  # the iterates depend on which chordal extension and merged cliques are taken
    ps = _problems(case, seed)
    if kind == "grad":
        offs = np.cumsum([0] + [p.C_val.size for p in ps])
        g = _cotangent(int(offs[-1]), seed)
        res = _each(lambda k: _Plain(ps[k], _cliques(case, k), -1).unrolled(case["iters"], g[offs[k]:offs[k + 1]]),
                    range(len(ps)))
        return {n: np.concatenate([r[q] for r in res]) for q, n in enumerate(("x", "cbar", "bbar"))}
    def one(k):
        q = _Plain(ps[k], _cliques(case, k), case["scale"])
        if case["form"] == "hsde":
            return q.hsde(case["iters"])
        return q.first_order(case["form"], case["iters"], case["adaptive"])

    res = _each(one, range(len(ps)))
    hist = res[0][3]
    if len(ps) > 1:  # a batch reports the largest residuals, the summed objectives and the SDPs still running
        h = np.stack([r[3] for r in res])
        hist = np.zeros((case["iters"], 8))
        hist[:, 0], hist[:, 1] = h[:, :, 0].max(axis=0), h[:, :, 1].max(axis=0)
        hist[:, 4], hist[:, 5] = h[:, :, 4].sum(axis=0), h[:, :, 5].sum(axis=0)
        hist[:-1, 6] = len(ps)
    return {"X": np.concatenate([r[0] for r in res]), "y": np.concatenate([r[1] for r in res]),
            "Z": np.concatenate([r[2] for r in res]), "hist": hist}
