"""Products around the number of unit boundaries up to which the kernel's last CTA finishes them."""
import numpy as np
import pytest
import torch

import inputs
import oracle
import paper_2605_07391_gb300 as mb
from tests.gpu_helpers import TOL, as_f64, check_rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles", [1022, 1023, 1024, 1438, 1439, 1440, 1441])   # boundaries: one more
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_product_and_solve(cuda_device, tiles, dtype):
    n = tiles * 448 // 4                         # three nonzeros a row; the rest in one row
    lens = np.full(n, 3, np.int64)
    lens[::5] = 0
    lens[n // 3] += tiles * 448 - n - int(lens.sum())
    a = inputs.row_lengths_csr(lens.tolist(), n, 2)
    rp, col = torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col).cuda()
    p = mb.plan(rp, col, a.n_rows, a.n_cols)
    assert p.info().tile_num == tiles
    v = torch.from_numpy(a.val).to("cuda", dtype)
    x = torch.from_numpy(inputs.uniform_vector(a.n_cols, 3)).to("cuda", dtype)
    for _ in range(2):                           # the second finds the accumulators clear
        y = mb.spmv(p, v, x)
        y_ref, d = oracle.spmv(a.row_ptr, a.col, as_f64(v), as_f64(x))
        check_rel(as_f64(y), y_ref, d, TOL[dtype], f"{tiles} tiles")
