"""What a user of this package has it do, as cases that can be timed and compared.

Each case is one call, or the few calls that belong together, through the public functions of
``kchol`` and ``batch``, on seeded synthetic points shaped like the package's own workloads: uniform
points and jittered grids in the square, uniform points in the cube, swiss rolls in R^20, batches of
uneven sets.  Sizes run from a set of a few thousand points to the 1024 x 1024 grid of ``bench.py``.

``kind`` says which call; the other entries are its sizes and options:

  path        a small point set from raw points to the solution: ordering, pattern, schedule, factor, solve
  order       the maximin ordering
  pattern     pattern S_rho and its schedule, from ordered points
  factor      the factor on a scheduled pattern
  factorsolve a factor and a solve with it
  solve       both triangular solves with a factor in hand
  matvec      L L^T v with a factor in hand
  refine      conjugate gradients on the dense matrix, preconditioned by the factor
  batch       one launch of a batch's factor plan
  supernodal  the supernodal order and pattern from the maximin ones, and the block factor on it
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1706_02205_gb300 import kchol as kc
from paper_1706_02205_gb300.batch import BatchFactor


def listed():
    return [
        # a first experiment: 2000 uniform points (the smallest workload of the package), where launches,
        # allocations and waits count rather than kernels
        dict(name="path_2000_f64", kind="path", points="uniform", N=2000, d=2, rho=3.0, nu=0.5, ell=0.2, nugget=0.0,
             prec="f64", nrhs=1),
        # the headline workload's three stages before the solve, on the 1024 x 1024 jittered grid
        dict(name="order_grid1024", kind="order", points="grid", N=1 << 20, d=2),
        dict(name="pattern_grid1024", kind="pattern", points="grid", N=1 << 20, d=2, rho=3.0),
        dict(name="factor_grid1024_f32", kind="factor", points="grid", N=1 << 20, d=2, rho=3.0, nu=0.5, ell=0.1,
             nugget=0.0, prec="f32"),
        # an ordinary set of odd size in full precision, one right-hand side (kriging one data vector)
        dict(name="factorsolve_100003_f64", kind="factorsolve", points="uniform", N=100003, d=2, rho=3.0, nu=0.5,
             ell=0.1, nugget=0.0, prec="f64", nrhs=1),
        # the 3-D points of the serving mix: long rows, narrow levels
        dict(name="factor_cube_131071_f32", kind="factor", points="uniform", N=131071, d=3, rho=4.0, nu=1.5, ell=0.1,
             nugget=0.0, prec="f32"),
        # the solve of the headline workload: 16 right-hand sides
        dict(name="solve16_grid1024_f32", kind="solve", points="grid", N=1 << 20, d=2, rho=3.0, nu=0.5, ell=0.1,
             nugget=0.0, prec="f32", nrhs=16),
        # products with the factor's approximation of the matrix, 16 vectors at a time (block iterations)
        dict(name="matvec16_grid1024_f32", kind="matvec", points="grid", N=1 << 20, d=2, rho=3.0, nu=0.5, ell=0.1,
             nugget=0.0, prec="f32", nrhs=16),
        # a system solved to 1e-10 with the factor as preconditioner
        dict(name="refine_grid128_f32", kind="refine", points="grid", N=128 * 128, d=2, rho=3.0, nu=0.5, ell=0.1,
             nugget=0.0, prec="f32", nrhs=16),
        # many uneven sets in one launch (their plan made once): three of four in the square, the fourth in the cube
        dict(name="batch_128_f32", kind="batch", sets=128, n_min=2000, n_max=50000, rho=3.0, nu=1.5, prec="f32"),
        # the front end of a serving request on a 2-D sheet in 20 dimensions, an odd size
        dict(name="swiss_250007", kind="pattern", points="swiss", N=250007, d=20, rho=3.0, order=True),
        # the supernodal order of the headline points and the block factor on it
        dict(name="supernodal_grid1024_f32", kind="supernodal", points="grid", N=1 << 20, d=2, rho=3.0, nu=0.5,
             ell=0.1, nugget=0.0, prec="f32"),
    ]


def _between(rng, lo, hi):
    """A whole number between lo and hi, even over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["path", "order", "pattern", "factor", "factor3", "factorsolve", "solve", "matvec", "refine",
                       "batch", "swiss", "supernodal"])
    grid = rng.random() < 0.5
    prec = rng.choice(["f32", "f64"])
    ell = round(rng.uniform(0.05, 0.3), 3)

    def points(lo, hi):
        n = _between(rng, lo, hi)
        if grid:
            side = max(2, int(round(math.sqrt(n))))
            return dict(points="grid", N=side * side, d=2)
        return dict(points="uniform", N=n, d=2)

    kern = dict(nu=0.5, ell=ell, nugget=0.0, prec=prec)
    if kind == "path":
        return dict(kind="path", **points(1000, 20000), rho=rng.choice([2.0, 3.0]), **kern, nrhs=rng.randint(1, 8))
    if kind == "order":
        return dict(kind="order", **points(2000, 1 << 20))
    if kind == "pattern":
        return dict(kind="pattern", **points(2000, 1 << 20), rho=rng.choice([2.0, 3.0]))
    if kind == "factor":
        return dict(kind="factor", **points(10000, 1 << 20), rho=rng.choice([2.0, 3.0]), **kern)
    if kind == "factor3":
        return dict(kind="factor", points="uniform", N=_between(rng, 10000, 131071), d=3, rho=rng.choice([3.0, 4.0]),
                    nu=rng.choice([0.5, 1.5]), ell=0.1, nugget=0.0, prec="f32")
    if kind == "factorsolve":
        return dict(kind="factorsolve", **points(10000, 400000), rho=rng.choice([2.0, 3.0]), **kern,
                    nrhs=rng.randint(1, 16))
    if kind == "solve":
        return dict(kind="solve", **points(10000, 1 << 20), rho=rng.choice([2.0, 3.0]), **kern, nrhs=rng.randint(1, 16))
    if kind == "matvec":
        return dict(kind="matvec", **points(10000, 1 << 20), rho=rng.choice([2.0, 3.0]), **kern, nrhs=rng.randint(1, 16))
    if kind == "refine":
        return dict(kind="refine", **points(2000, 20000), rho=3.0, **kern, nrhs=rng.randint(1, 16))
    if kind == "batch":
        return dict(kind="batch", sets=rng.randint(16, 128), n_min=2000, n_max=_between(rng, 10000, 50000), rho=3.0,
                    nu=rng.choice([0.5, 1.5]), prec="f32")
    if kind == "swiss":
        return dict(kind="pattern", points="swiss", N=_between(rng, 10000, 400000), d=20, rho=rng.choice([3.0, 4.0]),
                    order=True)
    return dict(kind="supernodal", **points(20000, 1 << 20), rho=rng.choice([2.0, 3.0]), nu=0.5, ell=ell, nugget=0.0,
                prec="f32")


# ------------------------------------------------------------------ inputs

def _gen(seed, stream=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 16 + stream)
    return g


def _rand(g, *shape):
    return torch.rand(shape, dtype=torch.float64, device="cuda", generator=g)


def _randn(g, *shape):
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)


def _points(case, seed):
    N, d, g = case["N"], case["d"], _gen(seed)
    if case["points"] == "uniform":
        return _rand(g, N, d)
    if case["points"] == "grid":  # cell centres, jittered by a quarter of a cell, in random order
        side = int(round(math.sqrt(N)))
        c = torch.arange(side, dtype=torch.float64, device="cuda")
        base = torch.stack(torch.meshgrid(c, c, indexing="ij"), -1).reshape(-1, 2)
        x = (base + 0.5 + 0.5 * (_rand(g, N, 2) - 0.5)) / side
        return x[torch.randperm(N, device="cuda", generator=g)].contiguous()
    # a swiss roll (a 2-D sheet) turned into R^d, with a little noise
    t = math.pi * (1.5 + 3.0 * _rand(g, N))
    y = torch.stack([t * torch.cos(t), 10.0 * _rand(g, N), t * torch.sin(t)], 1) / (4.5 * math.pi)
    q, _ = np.linalg.qr(np.random.Generator(np.random.PCG64(seed)).standard_normal((d, 3)))
    return (y @ torch.from_numpy(q.T.copy()).cuda() + 1e-3 * _randn(g, N, d)).contiguous()


def _vectors(case, seed):
    return _randn(_gen(seed, 1), case["nrhs"], case["N"])


def _kernel(case):
    return kc.Kernel(nu=case["nu"], ell=case["ell"], sigma2=1.0, nugget=case["nugget"])


def _prec(case):
    return kc.FP64 if case["prec"] == "f64" else kc.FP32_FORM


def _batch_sizes(case):
    """(size, dimension) of every set: sizes even over their logarithm, uneven neighbours, every fourth set in
    the cube, the others in the square."""
    S, a, b = case["sets"], math.log(case["n_min"]), math.log(case["n_max"])
    return [(int(math.exp(a + (b - a) * ((s * 0.6180339887498949) % 1.0))), 3 if s % 4 == 3 else 2) for s in range(S)]


def _batch_sets(case, seed):
    r, g = np.random.Generator(np.random.PCG64(seed)), _gen(seed)
    sizes = _batch_sizes(case)
    return [_rand(g, n, d) for n, d in sizes], [kc.Kernel(nu=case["nu"], ell=float(r.uniform(0.05, 0.3))) for _ in sizes]


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        xs, kerns = _batch_sets(case, seed)
        return dict(kind=kind, share=_share(case), b=BatchFactor(xs, kerns, case["rho"], _prec(case)))
    x = _points(case, seed)
    s = dict(kind=kind, share=_share(case), x=x, rho=case.get("rho"), order=case.get("order", False))
    if kind == "order" or s["order"]:
        return s
    if "nu" in case:
        s.update(kern=_kernel(case), prec=_prec(case))
    if kind in ("path", "factorsolve", "solve", "matvec", "refine"):
        s["b"] = _vectors(case, seed)
    if kind == "path":
        return s
    s["perm"], s["l"], s["xo"] = kc.order_points(x)
    if kind == "pattern":
        return s
    s["pat"] = kc.build_pattern(s["xo"], s["l"], case["rho"])
    if kind in ("solve", "matvec", "refine"):
        s["val"], s["diag"], _ = kc.factor(s["pat"], s["xo"], s["kern"], s["prec"])
    return s


# ------------------------------------------------------------------ one pass

def _row(points, N, d, rho):
    """Entries of a row of L on average: measured at these sizes, linear in log N between them."""
    L = math.log2(N)
    if points == "swiss":
        at, v = (13.29, 15.61, 17.93, 18.61), {3.0: (102.5, 135.7, 188.6, 215.1), 4.0: (159.3, 217.1, 312.3, 360.7)}
    elif d == 3:
        at, v = (10.97, 12.29, 13.29, 15.29, 17.0), {3.0: (139.0, 183.8, 221.5, 303.8, 379.9),
                                                     4.0: (226.9, 317.7, 396.5, 571.9, 740.5)}
    else:
        at, v = (10.0, 12.0, 14.0, 16.0, 18.0, 20.0), {2.0: (32.8, 43.7, 54.7, 66.0, 77.4, 88.8),
                                                       3.0: (56.4, 79.1, 103.1, 127.9, 153.2, 178.7)}
    return float(np.interp(L, at, v[rho]))


def _nnz(case):
    """Entries of the pattern, within some per cent (the points decide)."""
    if case["kind"] == "batch":
        return sum(n * _row("uniform", n, d, case["rho"]) for n, d in _batch_sizes(case))
    return case["N"] * _row(case["points"], case["N"], case["d"], case["rho"])


def _share(case):
    """How many of the entries _whole() puts in each of its two parts: fewer than there are, more than half."""
    if case["kind"] == "order":
        return 0
    more = (1.12 if case["rho"] == 2.0 else 1.28) if case["kind"] == "supernodal" else 1.0
    return int(0.8 * more * _nnz(case))


def _whole(t, m):
    """All values of t, whose length depends on the points, as two overlapping views whose length does not."""
    if not m <= t.shape[0] <= 2 * m:
        raise ValueError(f"{t.shape[0]} entries are not between {m} and {2 * m}")
    return t[:m], t[t.shape[0] - m:]


def _pattern_out(p, m):
    return dict(rowptr=p.rowptr[:-1], col=_whole(p.col, m), colptr=p.colptr[:-1], rowidx=_whole(p.rowidx, m),
                slot=_whole(p.slot, m), level=p.level, order=p.order, depth=p.depth, nnz=p.nnz)


def run(s):
    kind, m = s["kind"], s["share"]
    if kind == "path":
        r = kc.pipeline(s["x"], s["rho"], s["kern"], s["prec"])
        x = kc.solve(r["pat"], s["prec"], r["val"], r["diag"], s["kern"], r["perm"], s["b"])
        return dict(perm=r["perm"], l=r["l"], pattern=_pattern_out(r["pat"], m), val=_whole(r["val"], m),
                    diag=r["diag"], zero_pivots=r["zero_pivots"], x=x)
    if kind == "order":
        perm, l, xo = kc.order_points(s["x"])
        return dict(perm=perm, l=l, xo=xo)
    if kind == "pattern":
        if s["order"]:
            perm, l, xo = kc.order_points(s["x"])
            return dict(perm=perm, l=l, pattern=_pattern_out(kc.build_pattern(xo, l, s["rho"]), m))
        return _pattern_out(kc.build_pattern(s["xo"], s["l"], s["rho"]), m)
    if kind == "factor":
        val, diag, zero = kc.factor(s["pat"], s["xo"], s["kern"], s["prec"])
        return dict(val=_whole(val, m), diag=diag, zero_pivots=zero)
    if kind == "factorsolve":
        val, diag, zero = kc.factor(s["pat"], s["xo"], s["kern"], s["prec"])
        x = kc.solve(s["pat"], s["prec"], val, diag, s["kern"], s["perm"], s["b"])
        return dict(val=_whole(val, m), diag=diag, zero_pivots=zero, x=x)
    if kind == "solve":
        return kc.solve(s["pat"], s["prec"], s["val"], s["diag"], s["kern"], s["perm"], s["b"])
    if kind == "matvec":
        return kc.llt_matvec(s["pat"], s["prec"], s["val"], s["diag"], s["perm"], s["b"])
    if kind == "refine":  # the residuals it reports are rounding at 1e-11 of the right-hand side: left out
        x, iters, _, status = kc.refine(s["pat"], s["xo"], s["kern"], s["prec"], s["val"], s["diag"], s["perm"],
                                        s["b"], rtol=1e-10)
        return dict(x=x, iters=iters, status=status)
    if kind == "batch":
        zero = s["b"].factor()
        return dict(val=_whole(s["b"].val, m), diag=s["b"].diag, zero_pivots=zero)
    sn = kc.supernodal(s["xo"], s["l"], s["rho"], s["pat"])
    val, diag, zero = kc.factor_blocked(sn["pat"], sn["x_new"], s["kern"], s["prec"])
    return dict(newm=sn["newm"], level=sn["level"], node=sn["node"], color=sn["color"], x_new=sn["x_new"],
                pattern=_pattern_out(sn["pat"], m), val=_whole(val, m), diag=diag, zero_pivots=zero)


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    kind = case["kind"]
    s = 8 if case.get("prec") == "f64" else 4
    if kind == "batch":
        by = fl = 0.0
        for n, d in _batch_sizes(case):
            r = _row("uniform", n, d, case["rho"])
            by += n * (r * (4 + s) + 8 * d + 16)
            fl += n * r * r * 0.6
        return dict(bytes=by, flops=fl)
    N, d = case["N"], case["d"]
    by = fl = 0.0
    if kind in ("path", "order") or case.get("order"):
        by += N * (16.0 * d + 12)  # points in, points and order and length scales out
    if kind == "order":
        return dict(bytes=by, flops=N * 3.0 * d * 8)
    nnz = _nnz(case)
    r = nnz / N
    if kind in ("path", "pattern"):
        by += N * (8.0 * d + 8) + nnz * 20 + N * 24  # points; col, rowidx, slot; rowptr, colptr, level, order
        fl += nnz * 3.0 * d
    if kind in ("path", "factor", "factorsolve"):
        by += nnz * (4 + s) + N * (8.0 * d + 16)  # columns in, values out, points, pivots
        fl += nnz * r * 0.6  # a product and a sum where two rows share a column: about 0.6 of the prefix entries
    if kind in ("path", "factorsolve", "solve"):
        by += 2 * nnz * (4 + s) + N * (28.0 + 16.0 * case["nrhs"])  # L read by each solve; vectors in and out
        fl += 4.0 * nnz * case["nrhs"]
    if kind == "matvec":
        by += 2 * nnz * (4 + s) + N * (28.0 + 16.0 * case["nrhs"])
        fl += 4.0 * nnz * case["nrhs"]
    if kind == "refine":  # nine products with the dense matrix, whose entries are evaluated, not stored
        by += 9 * (2 * nnz * (4 + s) + N * (16.0 * case["nrhs"] + 8 * d))
        fl += 9.0 * N * N * (2.0 * case["nrhs"] + 3 * d + 20)
    if kind == "supernodal":
        by += nnz * 4 + 1.29 * nnz * (20 + 4 + 2 * s) + N * (24.0 * d + 60)
        fl += 1.29 * nnz * r * 0.6
    return dict(bytes=by, flops=fl)


# ------------------------------------------------------------------ the same in plain 64-bit NumPy, for small sets

def _maximin(x):
    N = x.shape[0]
    perm, l2 = np.empty(N, np.int64), np.empty(N)
    best = np.full(N, np.inf)
    k = 0
    for p in range(N):
        perm[p], l2[p] = k, best[k]
        diff = x - x[k]
        d2 = diff[:, 0] * diff[:, 0]
        for t in range(1, x.shape[1]):
            d2 = d2 + diff[:, t] * diff[:, t]
        best = np.minimum(best, d2)
        best[k] = -1.0
        k = int(np.argmax(best))
    return perm, np.sqrt(l2)


def _matern(r, nu, ell):
    t = math.sqrt(2.0 * nu) * r / ell
    return np.exp(-t) if nu == 0.5 else (1.0 + t) * np.exp(-t)


def _exact_factor(x, case):
    """Order, scales, the mask of S and the dense ICHOL(0) factor, by their definitions."""
    perm, l = _maximin(x)
    xo = x[perm]
    r = np.sqrt(sum((xo[:, None, t] - xo[None, :, t]) ** 2 for t in range(x.shape[1])))
    mask = np.tril(r <= case["rho"] * l[None, :])
    np.fill_diagonal(mask, True)
    A = np.where(mask, _matern(r, case["nu"], case["ell"]), 0.0)
    A[np.diag_indices_from(A)] += case["nugget"]
    for k in range(A.shape[0]):
        rows = k + np.flatnonzero(mask[k:, k])
        p = A[k, k]
        if not p > 0.0:
            A[rows, k] = 0.0
            continue
        A[k, k] = math.sqrt(p)
        rows = rows[1:]
        c = A[rows, k] / A[k, k]
        A[rows, k] = c
        at = np.ix_(rows, rows)
        A[at] -= np.where(mask[at], np.outer(c, c), 0.0)
    return perm, l, mask, A


def _solve_lower(L, b):
    return torch.linalg.solve_triangular(torch.from_numpy(L), torch.from_numpy(b), upper=False).numpy()


def _solve_upper(L, b):
    return torch.linalg.solve_triangular(torch.from_numpy(L.T.copy()), torch.from_numpy(b), upper=True).numpy()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "supernodal", "pattern"):
        return None  # the orders and patterns are whole numbers; the others would take minutes
    N = case["N"]
    if kind == "refine" and N <= 20000:  # the dense system, solved directly
        x = _points(case, seed)
        r = torch.cdist(x, x, compute_mode="donot_use_mm_for_euclid_dist")
        A = torch.exp(-math.sqrt(2.0 * case["nu"]) * r / case["ell"])
        del r
        return dict(x=torch.linalg.solve(A, _vectors(case, seed).T).T.contiguous(), iters=None, status=None)
    if N > 5000:
        return None
    x = _points(case, seed).cpu().numpy()
    if kind == "order":
        perm, l = _maximin(x)
        return dict(perm=None, l=l, xo=x[perm])
    perm, l, mask, L = _exact_factor(x, case)
    diag = np.diag(L).copy()
    res = dict(val=_whole(L[mask], _share(case)), diag=diag, zero_pivots=None)  # row by row, columns ascending
    if kind in ("path", "factorsolve", "solve", "matvec"):
        b = _vectors(case, seed).cpu().numpy()[:, perm].T
        S = L.copy()
        at = np.flatnonzero(diag <= 0.0)
        S[at, at] = math.sqrt(1.0 + case["nugget"])
        y = L @ (L.T @ b) if kind == "matvec" else _solve_upper(S, _solve_lower(S, b))
        out = np.empty_like(y)
        out[perm] = y
        out = np.ascontiguousarray(out.T)
        if kind in ("solve", "matvec"):
            return out
        res["x"] = out
    if kind == "path":
        res.update(perm=None, l=l, pattern=None)
    return res
