"""Captured products with an unaligned X take the padded copy like the others, and keep it."""
import numpy as np
import pytest
import torch

import inputs
import oracle
import paper_2605_07391_gb300 as mb
from tests.gpu_helpers import TOL, as_f64, check_rel, upload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [2, 5, 13, 33])
@pytest.mark.parametrize("warm", [True, False])
def test_captured_unaligned_product(cuda_device, k, warm):
    a = inputs.rmat_transition(13, 16, 3)
    rp, col, vals = upload(a)
    p = mb.plan(rp, col)
    X = torch.from_numpy(np.random.default_rng(k).random((a.n_cols, k)).astype(np.float32)).cuda()
    Y = torch.empty(a.n_rows, k, device="cuda")
    other = torch.rand(a.n_cols, 65, device="cuda")
    # the plan has its accumulators; with `warm`, also a copy of the chunk's width
    mb.spmm(p, vals, X if warm else torch.rand(a.n_cols, 8, device="cuda"))
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode="thread_local"):
        mb.spmm(p, vals, X, Y)
    # a wider product takes a copy of its own; the replay still finds its
    mb.spmm(p, vals, other)
    X.copy_(torch.rand(a.n_cols, k, device="cuda"))
    Y.fill_(float("nan"))
    g.replay()
    torch.cuda.synchronize()
    Y_ref, d = oracle.spmm(a.row_ptr, a.col, as_f64(vals), as_f64(X))
    for c in range(k):
        check_rel(as_f64(Y)[:, c], Y_ref[:, c], d[:, c], TOL[torch.float32], f"captured, k={k}, column {c}")
    # the same kernels as outside a capture: the same sums (rows between units are added by atomics)
    assert (Y != mb.spmm(p, vals, X)).float().mean().item() < 0.01
