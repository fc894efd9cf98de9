"""Per-nonzero products at every small sigma (a thread per lane below 3 or 4, a warp per tile from there
on), at sizes around a CTA's and a tile's, with empty and long rows."""
import numpy as np
import pytest
import torch

import inputs
import paper_2605_07391_gb300 as mb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("sigma", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("lens", [[1], [0, 31, 0], [255, 0, 1, 256, 257], [0] * 700 + [3000] + [0] * 300 + [2] * 999])
def test_values(cuda_device, sigma, dtype, lens):
    a = inputs.row_lengths_csr(lens, 4000, 2)
    p = mb.plan(torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col).cuda(), a.n_rows, a.n_cols, sigma=sigma)
    rng = np.random.default_rng(sigma)
    np_t = np.float32 if dtype == torch.float32 else np.float64
    g, x = rng.standard_normal(a.n_rows).astype(np_t), rng.standard_normal(a.n_cols).astype(np_t)
    out = mb.sddmm(p, torch.from_numpy(g).cuda(), torch.from_numpy(x).cuda(), 0.75)
    rows = np.repeat(np.arange(a.n_rows), np.diff(a.row_ptr))
    assert np.array_equal(out.cpu().numpy(), (np_t(0.75) * g)[rows] * x[a.col])


def test_time_at_sigma_1(cuda_device):
    """A tile of 32 steps is too little for a warp (3.7 times the time of sigma 14 that way)."""
    a = inputs.rmat_transition(18, 16, 1)
    rp, col = torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col).cuda()
    g, x = torch.rand(a.n_rows, device="cuda"), torch.rand(a.n_cols, device="cuda")
    out = torch.empty(a.nnz, device="cuda")

    def time(sigma):
        p = mb.plan(rp, col, sigma=sigma)
        ms = []
        for _ in range(9):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(20):
                mb.sddmm(p, g, x, 1.0, out)
            e1.record()
            torch.cuda.synchronize()
            ms.append(e0.elapsed_time(e1))
        return sorted(ms)[4]

    assert time(1) < 2.7 * time(14)
