"""The streaming pass of a personalised PageRank update at the widths where its sums take another
route: one segment of rows per block or several (2 k against the block's threads), 16-byte and
scalar columns, one row of more than 256 threads; on graphs smaller and larger than a block's rows."""
import numpy as np
import pytest
import torch

import inputs
import oracle
import paper_2605_07391_gb300 as mb
from tests.gpu_helpers import as_f64

pytestmark = pytest.mark.gpu

ALPHA = 0.85


@pytest.mark.parametrize("scale", [3, 12])
@pytest.mark.parametrize("k", [2, 4, 16, 63, 64, 65, 127, 128, 256, 257, 1024])
def test_ppr_widths(cuda_device, k, scale):
    a = inputs.rmat_transition(scale, 8, 3)
    rng = np.random.default_rng(k)
    seeds = rng.integers(0, a.n_rows, k).astype(np.int32)
    p = mb.plan(torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col).cuda())
    vals = torch.from_numpy(a.val).to("cuda", torch.float32)
    r = mb.ppr(p, vals, seeds, ALPHA, tol=0.0, max_iter=6)
    some = np.unique(np.concatenate([[0, k - 1], rng.integers(0, k, 6)]))
    ref = oracle.personalized_pagerank(a.row_ptr, a.col, a.val, seeds[some], ALPHA, fixed_iters=6)
    # six f32 updates of vectors that sum to 1: each adds at most a few 2^-24 per entry's row
    assert np.abs(as_f64(r["pi"])[:, some] - ref["pi"]).sum(axis=0).max() < 2e-5
    np.testing.assert_allclose(np.asarray(r["resid"])[some], ref["last"], rtol=1e-3, atol=1e-6)
    # the history holds the largest column residual of every update
    assert abs(r["hist"][-1] - np.max(r["resid"])) <= 1e-12
