"""SpMM at the sigmas around where the unrolled steps change (7 and 10), of every kind of X."""
import numpy as np
import pytest
import torch

import inputs
import oracle
import paper_2605_07391_gb300 as mb
from tests.gpu_helpers import TOL, as_f64, check_rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [1, 2, 6, 7, 8, 10, 11, 13])
@pytest.mark.parametrize("k", [4, 8, 13, 32])
@pytest.mark.parametrize("sparse", [False, True])      # sparse: unaligned X is gathered column by column
def test_against_the_oracle(cuda_device, sigma, k, sparse):
    if sparse:
        a = inputs.row_lengths_csr([2, 0, 3, 1, 900, 0] * 300, 200_000, 2)
    else:
        a = inputs.add_hubs(inputs.rmat_uniform(10, 8, 3, 3), 2, 600, 1500, 5)
    p = mb.plan(torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col).cuda(), a.n_rows, a.n_cols, sigma=sigma)
    vals = torch.from_numpy(a.val).cuda().float()
    X = torch.from_numpy(np.random.default_rng(k).random((a.n_cols, k)).astype(np.float32)).cuda()
    Y = mb.spmm(p, vals, X)
    p.sync()
    Y_ref, d = oracle.spmm(a.row_ptr, a.col, as_f64(vals), as_f64(X))
    for c in range(k):
        check_rel(as_f64(Y)[:, c], Y_ref[:, c], d[:, c], TOL[torch.float32], f"sigma {sigma}, k {k}, column {c}")
