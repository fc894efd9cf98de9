"""The one-launch PageRank at every width of a CTA up to its largest, and the first size past it.
Sizes follow the device's SMs, and the plan's tile count is checked: a warp holds one tile, a CTA up
to 16, and an SM one CTA."""
import numpy as np
import pytest
import torch

import inputs
import oracle
import paper_2605_07391_gb300 as mb
from tests.gpu_helpers import as_f64

pytestmark = pytest.mark.gpu
ALPHA = 0.85
STEPS = 14 * 32                      # vertices and edges of a tile at sigma 14


def _graph(tiles, seed, hub, empty):
    """A graph of exactly `tiles` tiles: a third of the steps are vertices, `empty` of the vertices
    lie in one run without in-edges, and vertex 3 takes every third edge when `hub`."""
    steps = tiles * STEPS - seed % 7
    n = steps // 3
    nnz = steps - n
    rng = np.random.default_rng(seed)
    live = np.concatenate([np.arange(n // 4), np.arange(n // 4 + int(n * empty), n)])
    dst = live[(rng.random(nnz) ** 2 * live.size).astype(np.int64)]
    if hub:
        dst[::3] = 3
    src = rng.integers(0, n, nnz)
    order = np.lexsort((src, dst))
    dst, src = dst[order], src[order]
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(dst, minlength=n), out=row_ptr[1:])
    deg = np.bincount(src, minlength=n)
    return inputs.CSR(n, n, row_ptr.astype(np.int32), src.astype(np.int32), 1.0 / deg[src], f"resident{tiles}")


def _updates(a, k):
    pi = np.full(a.n_rows, 1.0 / a.n_rows)
    dang = np.bincount(a.col, minlength=a.n_cols) == 0
    for _ in range(k):
        y, _ = oracle.spmv(a.row_ptr, a.col, a.val, pi)
        pi = ALPHA * y + (ALPHA * pi[dang].sum() + 1.0 - ALPHA) / a.n_rows
    return pi


@pytest.mark.parametrize("per_sm,more,hub,empty", [(7, 0, False, 0.3), (8, 0, True, 0.0), (12, 0, False, 0.0),
                                                   (15, 0, True, 0.3), (16, -1, False, 0.3), (16, 0, True, 0.3),
                                                   (16, 1, True, 0.0)])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_widths(cuda_device, per_sm, more, hub, empty, dtype):
    sms = torch.cuda.get_device_properties(cuda_device).multi_processor_count
    tiles = per_sm * sms + more
    a = _graph(tiles, 10 * per_sm + more, hub, empty)
    rp, col = torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col).cuda()
    p = mb.plan(rp, col)
    assert p.info().tile_num == tiles
    v = torch.from_numpy(a.val).to("cuda", dtype)
    # an update's rounding is at most a few units of the type, and shrinks by alpha per update;
    # 12 updates take the barriers' count past its wrap
    tol = 20 * torch.finfo(dtype).eps / (1 - ALPHA)
    for k in (1, 12):
        pi, info = mb.pagerank(p, v, ALPHA, tol=0.0, max_iter=k)
        ref = _updates(a, k)
        assert info["iters"] == k
        assert np.abs(as_f64(pi) - ref).max() <= tol * ref.max()
        assert abs(as_f64(pi).sum() - 1.0) <= tol
    if dtype == torch.float64:
        pi, info = mb.pagerank(p, v, ALPHA, tol=1e-11)
        assert info["converged"]
        assert oracle.pagerank_residual(a.row_ptr, a.col, a.val, as_f64(pi), ALPHA) < 1.1e-11
