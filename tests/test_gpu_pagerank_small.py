"""Plain PageRank of graphs that fit the SMs' shared memory (one cooperative launch) and of the
ones just too large for it, against the float64 oracle: tile counts at the edges of the CTAs and of
the rule, hub rows over many tiles, long runs of empty rows, other sigma, and the stop test."""
import numpy as np
import pytest
import torch

import inputs
import oracle
import paper_2605_07391_gb300 as mb
from tests.gpu_helpers import as_f64

pytestmark = pytest.mark.gpu
ALPHA = 0.85


def _graph(n, nnz, seed, hub=0):
    """About nnz edges into the first two thirds of n vertices, `hub` of them into vertex 3."""
    rng = np.random.default_rng(seed)
    dst = np.concatenate([(rng.random(nnz) ** 2 * (2 * n / 3)).astype(np.int64), np.full(hub, 3)])
    src = rng.integers(0, n, dst.size)
    key = np.unique(dst * n + src)
    dst, src = key // n, key % n
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(dst, minlength=n), out=row_ptr[1:])
    deg = np.bincount(src, minlength=n)
    return inputs.CSR(n, n, row_ptr.astype(np.int32), src.astype(np.int32), 1.0 / deg[src], f"g{n}_{nnz}")


def _updates(a, k):
    pi = np.full(a.n_rows, 1.0 / a.n_rows)
    dang = np.bincount(a.col, minlength=a.n_cols) == 0
    for _ in range(k):
        y, _ = oracle.spmv(a.row_ptr, a.col, a.val, pi)
        pi = ALPHA * y + (ALPHA * pi[dang].sum() + 1.0 - ALPHA) / a.n_rows
    return pi


# steps (vertices + edges) of 448 a tile: 1, 4 and 5 tiles, 608 (four a CTA) and 609, 2,432 (16 a
# CTA) and a few more
@pytest.mark.parametrize("n,nnz,hub,sigma", [(40, 100, 0, 14), (700, 1000, 0, 14), (900, 1300, 0, 14),
                                             (100_000, 172_000, 0, 14), (100_100, 173_000, 60_000, 14),
                                             (400_000, 690_000, 0, 14), (400_000, 700_000, 0, 14),
                                             (30_000, 300_000, 20_000, 14), (9_000, 40_000, 3_000, 7),
                                             (1_000, 9_000, 500, 1)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_updates(cuda_device, n, nnz, hub, sigma, dtype):
    a = _graph(n, nnz, n, hub)
    rp, col = torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col).cuda()
    p = mb.plan(rp, col, sigma=sigma)
    v = torch.from_numpy(a.val).to("cuda", dtype)
    # an update's rounding is at most a few units of the type, and shrinks by alpha per update
    tol = 20 * torch.finfo(dtype).eps / (1 - ALPHA)
    for k in (1, 2, 9):
        pi, info = mb.pagerank(p, v, ALPHA, tol=0.0, max_iter=k, history=True)
        ref = _updates(a, k)
        assert info["iters"] == k and len(info["hist"]) == k
        assert np.abs(as_f64(pi) - ref).max() <= tol * ref.max()
        assert abs(as_f64(pi).sum() - 1.0) <= tol
        prev = _updates(a, k - 1)
        assert abs(info["resid"] - np.abs(ref - prev).sum()) <= tol
    if dtype == torch.float64:
        pi, info = mb.pagerank(p, v, ALPHA, tol=1e-11)
        assert info["converged"] and info["resid"] < 1e-11
        assert oracle.pagerank_residual(a.row_ptr, a.col, a.val, as_f64(pi), ALPHA) < 1.1e-11
    # the plan's other products still find its state clean
    x = torch.rand(n, device="cuda", dtype=dtype)
    y_ref, d = oracle.spmv(a.row_ptr, a.col, as_f64(v), as_f64(x))
    err = oracle.relative_errors(as_f64(mb.spmv(p, v, x)), y_ref, d)
    assert err.max() <= (1e-5 if dtype == torch.float32 else 1e-12)
