"""The lane-walk kernel's tile buffers filled to their last byte: tiles of nonzeros alone and of one
row fewer, rows and nonzeros in every ratio, starting at every offset from a 16-byte boundary."""
import numpy as np
import pytest
import torch

import inputs
import oracle
import paper_2605_07391_gb300 as mb
from tests.gpu_helpers import TOL, as_f64, check_rel

pytestmark = pytest.mark.gpu

COLS = 1500


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64, torch.bfloat16, torch.float16])
@pytest.mark.parametrize("sigma", [1, 7, 13, 14])
@pytest.mark.parametrize("shift", range(8))
def test_full_buffers(cuda_device, shift, sigma, dtype):
    step = 32 * sigma
    lengths = [shift]
    lengths += [step - 1] * 4                           # a tile of one row
    lengths += [3 * step + 5]                           # tiles of nonzeros alone
    lengths += [0] * (step + 3)                         # a tile of rows alone
    lengths += [1] * step + [2] * step                  # half and a third of the steps are rows
    lengths += [step - 2, 0] * 3 + [step // 2 + 1] * 5
    a = inputs.row_lengths_csr(lengths, COLS, shift, "buffers")
    xt = torch.float64 if dtype == torch.float64 else torch.float32
    rng = np.random.default_rng(shift)
    x = torch.from_numpy(rng.uniform(-1, 1, COLS)).to("cuda", xt)
    vals = torch.from_numpy(a.val).to("cuda", dtype)
    p = mb.plan(torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col).cuda(), a.n_rows, COLS, sigma=sigma)
    y = mb.spmv(p, vals, x)
    y_ref, d = oracle.spmv(a.row_ptr, a.col, as_f64(vals), as_f64(x))[:2]
    check_rel(as_f64(y), y_ref, d, TOL[xt], f"{dtype} sigma={sigma} shift={shift}")
