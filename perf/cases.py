"""Performance cases of the framework: what its users run, through its public entry points.

A case names one call of one family (`kind`) and its size.  The graphs are made on the GPU
from the seed alone: R-MAT (the power-law graphs of the paper's suite), uniform random, and
grid graphs (road networks), with any vertex count.  Matrices are CSR with sorted columns;
a PageRank matrix holds 1/outdeg(source) at (destination, source).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2605_07391_gb300 as mb
from paper_2605_07391_gb300 import autograd as ag

DEV = "cuda"
F32, F64 = torch.float32, torch.float64
DTYPES = {"f32": F32, "f64": F64, "bf16": torch.bfloat16, "f16": torch.float16}
ALPHA = 0.85


def listed():
    return [
        # the smallest call: one product of a 1,024-vertex graph, where the launch is the cost
        {"name": "spmv_f32_tiny", "kind": "spmv", "graph": "rmat", "n": 1 << 10, "degree": 16, "dtype": "f32"},
        # the headline: one f32 product of a 16.8 M-vertex graph (263 M nonzeros)
        {"name": "spmv_f32_large", "kind": "spmv", "graph": "rmat", "n": 1 << 24, "degree": 16, "dtype": "f32"},
        # double precision, 30 % of the rows empty
        {"name": "spmv_f64_empty_rows", "kind": "spmv", "graph": "empty", "n": 1 << 22, "degree": 16, "dtype": "f64"},
        # batched products: a wide block of right-hand sides, and a ragged one (odd k, odd n)
        {"name": "spmm_k32", "kind": "spmm", "graph": "rmat", "n": 1 << 21, "degree": 16, "k": 32},
        {"name": "spmm_k13_ragged", "kind": "spmm", "graph": "rmat", "n": 1_000_003, "degree": 12, "k": 13},
        # personalised PageRank of eight seeds
        {"name": "ppr_k8", "kind": "ppr", "graph": "rmat", "n": 1 << 20, "degree": 16, "k": 8},
        # PageRank: 100 updates of a small graph (launch latency), and the mixed-precision
        # refinement (bf16 sweeps, f64 residuals) to 1e-10 on a large one
        {"name": "pagerank_f32_small", "kind": "pagerank", "graph": "rmat", "n": 1 << 14, "degree": 16,
         "mode": "plain", "dtype": "f32", "updates": 100},
        {"name": "pagerank_ir_bf16", "kind": "pagerank", "graph": "rmat", "n": 1 << 22, "degree": 16,
         "mode": "ir_bf16", "dtype": "f64", "updates": 0},
        # training: forward and backward of y = A x (gradients of the values and of x)
        {"name": "spmv_train_f32", "kind": "train", "graph": "rmat", "n": 1 << 20, "degree": 16, "dtype": "f32"},
        # a new pattern made ready for training: its plan, its transpose and the transpose's plan
        {"name": "new_pattern", "kind": "pattern", "graph": "rmat", "n": 1 << 20, "degree": 16, "dtype": "f32"},
        # PageRank of 64 graphs of very different sizes in one call
        {"name": "batch_f64", "kind": "batch", "graphs": 64, "lo": 10, "hi": 18, "dtype": "f64"},
        # a linear solve on a road network (two to three neighbours per vertex)
        {"name": "bicgstab_road", "kind": "bicgstab", "n": 3_000_000, "keep": 0.55},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same families: sizes log-uniform, odd ones included."""
    kind = rng.choice(["spmv", "spmv", "spmm", "ppr", "pagerank", "train", "pattern", "batch", "bicgstab"])
    graph = rng.choice(["rmat", "rmat", "empty", "hubs", "uniform"])
    degree = rng.randint(4, 32)
    if kind == "spmv":
        return {"kind": kind, "graph": graph, "n": _log(rng, 300, 5_000_000), "degree": degree,
                "dtype": rng.choice(["f32", "f32", "f64", "bf16", "f16"])}
    if kind == "spmm":
        return {"kind": kind, "graph": graph, "n": _log(rng, 300, 1_500_000), "degree": degree,
                "k": _log(rng, 2, 40)}
    if kind == "ppr":
        return {"kind": kind, "graph": "rmat", "n": _log(rng, 1000, 1_000_000), "degree": degree,
                "k": rng.choice([1, 4, 7, 8, 16, 32])}
    if kind == "pagerank":
        mode = rng.choice(["plain", "plain", "ir_bf16", "ir_f16", "ir_f32"])
        dtype = rng.choice(["f32", "f64"]) if mode == "plain" else "f64"
        return {"kind": kind, "graph": "rmat", "n": _log(rng, 1000, 4_000_000), "degree": degree, "mode": mode,
                "dtype": dtype, "updates": rng.randint(20, 100) if dtype == "f32" else 0}
    if kind in ("train", "pattern"):
        return {"kind": kind, "graph": graph, "n": _log(rng, 1000, 2_000_000), "degree": degree,
                "dtype": rng.choice(["f32", "f64"])}
    if kind == "batch":
        lo = rng.randint(6, 12)
        return {"kind": kind, "graphs": _log(rng, 3, 100), "lo": lo, "hi": rng.randint(lo + 1, 17),
                "dtype": rng.choice(["f32", "f64"])}
    return {"kind": kind, "n": _log(rng, 2000, 4_000_000), "keep": rng.uniform(0.5, 0.9)}


# ---------------------------------------------------------------------------- graphs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _rmat_ids(scale, count, gen):
    """Sources and destinations of `count` R-MAT edges (0.57, 0.19, 0.19, 0.05).  `scale` is
    a number, or a tensor with the scale of each edge."""
    top = scale if isinstance(scale, int) else int(scale.max())
    src = torch.zeros(count, dtype=torch.int64, device=DEV)
    dst = torch.zeros_like(src)
    for level in range(top):
        u = torch.rand(count, generator=gen, device=DEV)
        sb = u >= 0.76
        db = ((u >= 0.57) & ~sb) | (u >= 0.95)
        if isinstance(scale, int):
            src.mul_(2).add_(sb)
            dst.mul_(2).add_(db)
        else:
            on = level < scale
            src = torch.where(on, src * 2 + sb, src)
            dst = torch.where(on, dst * 2 + db, dst)
    return src, dst


def _csr(rows, cols, n):
    """Sorted CSR without repeated entries."""
    key = torch.unique(rows * n + cols)
    row = key // n
    col = (key - row * n).to(torch.int32)
    row_ptr = torch.zeros(n + 1, dtype=torch.int32, device=DEV)
    row_ptr[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return row_ptr, col


def _graph(case, gen, turn=()):
    """A graph of the case's family; `turn`: how far its rows and columns are rotated."""
    n, edges = case["n"], case["n"] * case["degree"]
    if case["graph"] == "uniform":
        src = torch.randint(0, n, (edges,), generator=gen, device=DEV)
        dst = torch.randint(0, n, (edges,), generator=gen, device=DEV)
    else:
        scale = max(1, (n - 1).bit_length())
        src, dst = _rmat_ids(scale, edges, gen)
        if n != 1 << scale:
            src, dst = (src * n) >> scale, (dst * n) >> scale
    ok = src != dst
    if case["graph"] == "empty":
        ok &= (torch.rand(n, generator=gen, device=DEV) >= 0.3)[dst]
    src, dst = src[ok], dst[ok]
    if case["graph"] == "hubs":
        # four rows that reach a quarter of the columns
        hub = torch.randint(0, n, (4,), generator=gen, device=DEV)
        reach = torch.rand(4, n, generator=gen, device=DEV) < 0.25
        h, c = reach.nonzero(as_tuple=True)
        src, dst = torch.cat([src, c]), torch.cat([dst, hub[h]])
    return _csr((dst + turn[0]) % n, (src + turn[1]) % n, n) if turn else _csr(dst, src, n)


def _rows(row_ptr):
    n = row_ptr.numel() - 1
    return torch.repeat_interleave(torch.arange(n, device=DEV), (row_ptr[1:] - row_ptr[:-1]).long())


def _transition(col, n):
    """1/outdeg(source) in f64."""
    return 1.0 / torch.bincount(col, minlength=n).double()[col.long()]


def _uniform_values(count, gen):
    return 1.0 - torch.rand(count, generator=gen, device=DEV, dtype=F64)


def _batch_scales(case, seed):
    rng = np.random.default_rng(seed if case["graphs"] < 8 else 42)
    return rng.integers(case["lo"], case["hi"] + 1, case["graphs"]), rng.integers(8, 33, case["graphs"])


def _batch_graph(case, seed, gen):
    """The graphs as the diagonal blocks of one CSR, and the first vertex of each."""
    scales, degrees = _batch_scales(case, seed)
    off = np.zeros(case["graphs"] + 1, np.int64)
    np.cumsum(1 << scales.astype(np.int64), out=off[1:])
    edges = torch.tensor(degrees * (1 << scales.astype(np.int64)), device=DEV)
    scale = torch.repeat_interleave(torch.tensor(scales, device=DEV), edges)
    base = torch.repeat_interleave(torch.tensor(off[:-1], device=DEV), edges)
    src, dst = _rmat_ids(scale, scale.numel(), gen)
    ok = src != dst
    row_ptr, col = _csr((dst + base)[ok], (src + base)[ok], int(off[-1]))
    return row_ptr, col, off


def _road_system(case, gen):
    """Laplacian of a grid graph that keeps each edge with probability `keep`, plus 1/2 on
    the diagonal."""
    nx = max(2, int(math.isqrt(case["n"])))
    n = nx * nx
    v = torch.arange(n, device=DEV)
    right, down = v[v % nx != nx - 1], v[: n - nx]
    a = torch.cat([right, down])
    b = torch.cat([right + 1, down + nx])
    keep = torch.rand(a.numel(), generator=gen, device=DEV) < case["keep"]
    a, b = a[keep], b[keep]
    degree = torch.bincount(torch.cat([a, b]), minlength=n).double()
    row_ptr, col = _csr(torch.cat([a, b, v]), torch.cat([b, a, v]), n)
    row = _rows(row_ptr)
    return row_ptr, col, torch.where(row == col, degree[row] + 0.5, -1.0)


# ---------------------------------------------------------------------------- the calls

def _inputs(case, seed):
    """Every array of the call; on the GPU, from the seed alone."""
    gen = _gen(seed)
    kind = case["kind"]
    s = {}
    if kind == "batch":
        s["row_ptr"], s["col"], s["off"] = _batch_graph(case, seed, gen)
        s["vals"] = _transition(s["col"], int(s["off"][-1])).to(DTYPES[case["dtype"]])
        return s
    if kind == "bicgstab":
        s["row_ptr"], s["col"], s["vals"] = _road_system(case, gen)
        s["b"] = torch.rand(s["row_ptr"].numel() - 1, generator=gen, device=DEV, dtype=F64)
        return s
    if kind in ("train", "pattern"):
        # results of one shape whatever the seed (they have an entry per nonzero): one graph,
        # its vertices relabelled
        s["row_ptr"], s["col"] = _graph(case, _gen(7), torch.randint(0, case["n"], (2,), generator=gen, device=DEV).tolist())
    else:
        s["row_ptr"], s["col"] = _graph(case, gen)
    n, nnz = case["n"], s["col"].numel()
    if kind in ("ppr", "pagerank"):
        v = _transition(s["col"], n)
        s["vals"] = v.to(F32 if kind == "ppr" else DTYPES[case["dtype"]])
        if kind == "ppr":
            has_out = torch.bincount(s["col"], minlength=n) > 0
            pick = torch.where(has_out, torch.rand(n, generator=gen, device=DEV), -1.0)
            s["seeds"] = torch.topk(pick, case["k"]).indices.to(torch.int32).cpu().numpy()
        return s
    dtype = DTYPES[case.get("dtype", "f32")]
    s["vals"] = _uniform_values(nnz, gen).to(dtype)
    xt = F64 if dtype == F64 else F32
    if kind == "spmv":
        s["x"] = torch.rand(n, generator=gen, device=DEV, dtype=xt)
    elif kind == "spmm":
        s["X"] = torch.rand(n, case["k"], generator=gen, device=DEV, dtype=F32)
    elif kind == "train":
        s["x"] = torch.rand(n, generator=gen, device=DEV, dtype=xt)
        s["g"] = torch.randn(n, generator=gen, device=DEV, dtype=xt)
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    if kind == "train":
        s["A"] = ag.Matrix(s["row_ptr"], s["col"])
        s["A"].transposed()
    elif kind == "batch":
        s["batch"] = mb.Batch(s["row_ptr"], s["col"], s["off"])
        s["pi"] = torch.empty(int(s["off"][-1]), dtype=s["vals"].dtype, device=DEV)
    elif kind != "pattern":
        s["plan"] = mb.plan(s["row_ptr"], s["col"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "spmv":
        return mb.spmv(s["plan"], s["vals"], s["x"])
    if kind == "spmm":
        return mb.spmm(s["plan"], s["vals"], s["X"])
    if kind == "ppr":
        return mb.ppr(s["plan"], s["vals"], s["seeds"], ALPHA, tol=1e-6)["pi"]
    if kind == "pagerank":
        if case["updates"]:
            return mb.pagerank(s["plan"], s["vals"], ALPHA, tol=0.0, max_iter=case["updates"])[0]
        if case["mode"] == "plain":
            return mb.pagerank(s["plan"], s["vals"], ALPHA, tol=1e-10)[0]
        sweeps, inner = {"ir_bf16": (12, 2.0 ** -4), "ir_f16": (6, 2.0 ** -11), "ir_f32": (6, 2.0 ** -10)}[case["mode"]]
        return mb.pagerank(s["plan"], s["vals"], ALPHA, tol=1e-10, max_iter=60, mode=case["mode"],
                           inner_sweeps=sweeps, inner_tol=inner)[0]
    if kind == "train":
        vals, x = s["vals"].detach().requires_grad_(), s["x"].detach().requires_grad_()
        y = ag.spmv(s["A"], vals, x)
        gv, gx = torch.autograd.grad(y, (vals, x), s["g"])
        return {"y": y.detach(), "gvals": gv, "gx": gx}
    if kind == "pattern":
        A = ag.Matrix(s["row_ptr"], s["col"])
        t, _ = A.transposed()
        return {"row_ptr_t": t.row_ptr_t, "col_t": t.col_t, "perm": t.perm,
                "vals_t": A.transposed_values(s["vals"])}
    if kind == "batch":
        pi, info = s["batch"].pagerank(s["vals"], ALPHA, tol=1e-8 if case["dtype"] == "f64" else 1e-5, pi=s["pi"])
        return {"pi": pi, "iters": info["iters"]}
    return mb.bicgstab(s["plan"], s["vals"], s["b"], tol=1e-11, max_iter=200)[0]


# ---------------------------------------------------------------------------- exact results

def _mul(row, col, vals, x):
    """A x in 64 bits (x: n or n x k)."""
    n = x.shape[0]
    p = vals[:, None] * x[col] if x.dim() == 2 else vals * x[col]
    return torch.zeros_like(x[:n]).index_add_(0, row, p)


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    row, col = _rows(s["row_ptr"]), s["col"].long()
    vals = s["vals"].double()
    n = s["row_ptr"].numel() - 1
    if kind == "spmv":
        return _mul(row, col, vals, s["x"].double())
    if kind == "spmm":
        X = s["X"].double()
        return torch.cat([_mul(row, col, vals, X[:, c:c + 4].contiguous()) for c in range(0, case["k"], 4)], 1)
    if kind == "train":
        x, g = s["x"].double(), s["g"].double()
        return {"y": _mul(row, col, vals, x), "gvals": g[row] * x[col], "gx": _mul(col, row, vals, g)}
    if kind == "pattern":
        perm = torch.argsort(col, stable=True)
        return {"row_ptr_t": None, "col_t": None, "perm": None, "vals_t": vals[perm]}
    if kind == "bicgstab":
        # conjugate gradients (the system is symmetric and positive definite)
        x = torch.zeros(n, dtype=F64, device=DEV)
        r = s["b"].clone()
        p, rr = r.clone(), r @ r
        stop = 1e-15 * rr.sqrt()
        for _ in range(400):
            q = _mul(row, col, vals, p)
            a = rr / (p @ q)
            x += a * p
            r -= a * q
            old, rr = rr, r @ r
            if rr.sqrt() < stop:
                break
            p = r + (rr / old) * p
        return x
    dangling = torch.bincount(col, minlength=n) == 0
    if kind == "ppr":
        seeds = torch.tensor(s["seeds"], dtype=torch.int64, device=DEV)
        at = torch.zeros(n, case["k"], dtype=F64, device=DEV)
        at[seeds, torch.arange(case["k"], device=DEV)] = 1.0
        pi = at.clone()
        for _ in range(60):
            mass = ALPHA * pi[dangling].sum(0) + 1.0 - ALPHA
            new = torch.cat([_mul(row, col, vals, pi[:, c:c + 8].contiguous()) for c in range(0, case["k"], 8)], 1)
            pi = ALPHA * new + at * mass
        return pi
    if kind == "pagerank":
        if s["vals"].dtype == F32:
            vals = _transition(s["col"], n)
        pi = torch.full((n,), 1.0 / n, dtype=F64, device=DEV)
        for _ in range(case["updates"] or 200):
            pi = ALPHA * _mul(row, col, vals, pi) + (ALPHA * pi[dangling].sum() + 1.0 - ALPHA) / n
        return pi
    off = torch.tensor(s["off"], device=DEV)
    size = off[1:] - off[:-1]
    graph = torch.repeat_interleave(torch.arange(case["graphs"], device=DEV), size)
    vals = _transition(s["col"], n)
    inv = 1.0 / size.double()
    pi = inv[graph]
    for _ in range(150):
        mass = torch.zeros(case["graphs"], dtype=F64, device=DEV).index_add_(0, graph[dangling], pi[dangling])
        pi = ALPHA * _mul(row, col, vals, pi) + ((ALPHA * mass + 1.0 - ALPHA) * inv)[graph]
    return {"pi": pi, "iters": None}


# ---------------------------------------------------------------------------- work

def _nnz(n, degree, graph):
    """Nonzeros left of n * degree edges: R-MAT draws repeat edges (13 % of 16 * 2^14, 2.8 %
    of 16 * 2^22, 1.9 % of 16 * 2^24)."""
    m = n * degree
    if graph != "uniform":
        m *= 1.0 - min(0.5, 0.13 * degree / 16.0 * 2.0 ** (-0.277 * (math.log2(n) - 14.0)))
    return m * 0.7 if graph == "empty" else m + n if graph == "hubs" else m


def work(case):
    """Bytes and operations of the mathematics: matrix, vectors and results, once each per
    product; solves count the updates that these inputs take."""
    kind = case["kind"]
    if kind == "batch":
        scales, degrees = _batch_scales(case, 0)
        n = float((1 << scales.astype(np.int64)).sum())
        m = 0.9 * float((degrees * (1 << scales.astype(np.int64))).sum())
        e = 8 if case["dtype"] == "f64" else 4
        rounds = 20 if case["dtype"] == "f64" else 10
        return {"bytes": rounds * (m * (4 + e) + 2 * n * e), "flops": rounds * 2.0 * m}
    n = case["n"]
    if kind == "bicgstab":
        m = n * (1 + 4 * case["keep"])
        # an iteration: two products, and ten vectors read or written by the rest
        return {"bytes": 37 * (2 * (12 * m + 16 * n) + 80 * n), "flops": 37 * (4 * m + 20 * n)}
    m = _nnz(n, case["degree"], case["graph"])
    if kind == "spmv":
        v = {"f32": 4, "f64": 8}.get(case["dtype"], 2)
        return {"bytes": m * (4 + v) + 2 * n * max(v, 4), "flops": 2.0 * m}
    if kind == "spmm":
        return {"bytes": 8 * m + 8 * n * case["k"], "flops": 2.0 * m * case["k"]}
    if kind == "ppr":
        return {"bytes": 13 * (8 * m + 8 * n * case["k"]), "flops": 13 * 2.0 * m * case["k"]}
    if kind == "pagerank":
        e = 4 if case["dtype"] == "f32" else 8
        if case["updates"]:
            return {"bytes": case["updates"] * (m * (4 + e) + 2 * n * e), "flops": case["updates"] * 2.0 * m}
        if case["mode"] == "plain":
            return {"bytes": 31 * (12 * m + 16 * n), "flops": 31 * 2.0 * m}
        v = 4 if case["mode"] == "ir_f32" else 2
        steps, sweeps = {"ir_bf16": (8, 68), "ir_f16": (10, 61), "ir_f32": (5, 31)}[case["mode"]]
        return {"bytes": sweeps * (m * (4 + v) + 12 * n) + steps * (12 * m + 16 * n), "flops": 2.0 * m * (steps + sweeps)}
    e = 4 if case["dtype"] == "f32" else 8
    if kind == "train":
        # forward, value gradient, transposed values, transposed product
        return {"bytes": m * (4 + e) + 2 * n * e + m * (4 + e) + 2 * n * e + m * (4 + 2 * e) + m * (4 + e) + 2 * n * e,
                "flops": 5.0 * m}
    # pattern: columns in; transposed columns, permutation and values out
    return {"bytes": 4 * m + 8 * n + 8 * m + 2 * e * m, "flops": 0.0}
