"""BiCGSTAB at the edges of the vector passes' chunks (1,024 rows: 256 threads x 4) and on more
chunks than CTAs: the solution of a diagonally dominant banded system, and the count of iterations
when max_iter ends the loop."""
import numpy as np
import pytest
import torch

import paper_2605_07391_gb300 as mb
from tests.gpu_helpers import as_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset", [0, 1], ids=["aligned", "odd_x"])
@pytest.mark.parametrize("n", [1, 2, 255, 257, 1023, 1024, 1025, 3 * 1024 + 769, 700_001])
def test_bicgstab_sizes(cuda_device, n, offset):
    rng = np.random.default_rng(n)
    lo, hi = rng.uniform(-1, 1, n), rng.uniform(-1, 1, n)
    i = np.arange(n)
    col = np.stack([i - 1, i, i + 1], 1)
    val = np.stack([lo, np.full(n, 4.0), hi], 1)
    keep = (col >= 0) & (col < n)
    rp = np.concatenate([[0], np.cumsum(keep.sum(1))]).astype(np.int32)
    ref = rng.standard_normal(n)
    lower = np.concatenate([[0.0], ref[:-1]])
    upper = np.concatenate([ref[1:], [0.0]])
    b = 4.0 * ref + lo * lower + hi * upper
    p = mb.plan(torch.from_numpy(rp).cuda(), torch.from_numpy(col[keep].astype(np.int32)).cuda(), n, n)
    vals = torch.from_numpy(val[keep]).cuda()
    rhs = torch.from_numpy(b).cuda()
    x = torch.zeros(n + 1, dtype=torch.float64, device="cuda")[offset:n + offset]
    x, info = mb.bicgstab(p, vals, rhs, x, tol=1e-11, max_iter=200)
    assert info["converged"]
    # every eigenvalue's distance from 4 is at most 2 (Gershgorin): ||A^-1||_2 <= 1 / (4 - 2), the
    # symmetric part's smallest eigenvalue being at least 2; a factor 2 for the recursive residual
    assert np.linalg.norm(as_f64(x) - ref) <= 2 * 1e-11 * np.linalg.norm(b) / 2 + 1e-14 * n ** 0.5
    if n > 1000:
        x.zero_()
        _, info = mb.bicgstab(p, vals, rhs, x, tol=0.0, max_iter=3)
        assert info["iters"] == 3 and not info["converged"]
