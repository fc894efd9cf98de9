"""Batches at the limit of the graph table that a product keeps in shared memory (256 graphs), and
graphs whose row counts straddle the spans of the reduction's warps (1,024 rows, 32 lanes x 8)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2605_07391_gb300 as mb
from tests.gpu_helpers import as_f64

pytestmark = pytest.mark.gpu

ALPHA = 0.85
TOL = 1e-10


def _graph(n, rng):
    """A P^T with 3 n random links among n vertices; vertices without out-links are dangling."""
    row = rng.integers(0, n, 3 * n)
    col = rng.integers(0, max(1, n - n // 5), 3 * n)
    order = np.argsort(row, kind="stable")
    row, col = row[order], col[order]
    val = 1.0 / np.bincount(col, minlength=n)[col]
    return np.concatenate([[0], np.cumsum(np.bincount(row, minlength=n))]), col, val


@pytest.mark.parametrize("sizes", [
    [1 + g % 40 for g in range(256)],
    [1 + g % 40 for g in range(257)],
    [255, 1, 256, 257, 1023, 1024, 1025, 31, 32, 33, 5000],
    [3000],
], ids=["256_graphs", "257_graphs", "straddling", "one_graph"])
def test_batch_sizes(cuda_device, sizes):
    rng = np.random.default_rng(len(sizes))
    parts = [_graph(n, rng) for n in sizes]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    nnz = np.concatenate([[0], np.cumsum([p[1].size for p in parts])])
    rp = np.concatenate([p[0][:-1] + k for p, k in zip(parts, nnz)] + [nnz[-1:]]).astype(np.int32)
    col = np.concatenate([p[1] + o for p, o in zip(parts, off)]).astype(np.int32)
    val = np.concatenate([p[2] for p in parts])
    b = mb.Batch(torch.from_numpy(rp).cuda(), torch.from_numpy(col).cuda(), off)
    pi, info = b.pagerank(torch.from_numpy(val).cuda(), ALPHA, tol=TOL, max_iter=500)
    assert info["converged"]
    got = as_f64(pi)
    # the power method's error is at most its last step's size times alpha / (1 - alpha)
    bound = TOL * ALPHA / (1 - ALPHA) * 1.01 + 1e-13
    for g, (prp, pcol, pval) in enumerate(parts):
        ref = oracle.pagerank(prp.astype(np.int32), pcol.astype(np.int32), pval, ALPHA, tol=TOL,
                              max_iter=500)
        assert abs(int(info["iters"][g]) - ref["iters"]) <= 1, g
        exact = oracle.pagerank(prp.astype(np.int32), pcol.astype(np.int32), pval, ALPHA,
                                tol=1e-15, max_iter=5000)["pi"]
        assert np.abs(got[off[g]:off[g + 1]] - exact).sum() <= bound, g
    b.destroy()
