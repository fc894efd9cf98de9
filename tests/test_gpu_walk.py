"""The lane-walk SpMV kernel (the automatic choice) against the float64 oracle where it can go
wrong: the array's last nonzeros (short of a 16-byte unit) for every value width, tile edges,
rows over many units, every unit length, and its bounded waits."""
import numpy as np
import pytest
import torch

import inputs
import oracle
import paper_2605_07391_gb300 as mb
from tests.gpu_helpers import TOL, as_f64, check_rel

pytestmark = pytest.mark.gpu
DTYPES = [torch.float32, torch.float64, torch.bfloat16, torch.float16]


def _check(a, dtype, sigma=14, W=8, calls=2):
    rp, col = torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col).cuda()
    p = mb.plan(rp, col, a.n_rows, a.n_cols, sigma=sigma, tiles_per_block=W)
    vals = torch.from_numpy(a.val).to("cuda", dtype)
    xt = torch.float64 if dtype == torch.float64 else torch.float32
    x = torch.from_numpy(inputs.uniform_vector(a.n_cols, 2)).to("cuda", xt)
    y_ref, d = oracle.spmv(a.row_ptr, a.col, as_f64(vals), as_f64(x))
    y = torch.full((a.n_rows,), float("nan"), dtype=xt, device="cuda")
    for _ in range(calls):
        mb.spmv(p, vals, x, y)
    p.sync()
    check_rel(as_f64(y), y_ref, d, TOL[xt], f"{a.name} {dtype} sigma={sigma} W={W}")


@pytest.mark.parametrize("dtype", DTYPES)
def test_array_ends_and_tile_edges(cuda_device, dtype):
    for tail in range(9):                      # nnz mod 8 takes every value
        _check(inputs.row_lengths_csr([3, 0, 400, 14 + tail], 500, tail, f"tail{tail}"), dtype)
    for extra in (-1, 0, 1):                   # paths that end just before, at and after a tile
        _check(inputs.row_lengths_csr([446 + extra], 500, 1, f"edge{extra}"), dtype)
        _check(inputs.row_lengths_csr([1] * (224 * 3) + [extra + 1], 500, 2, f"rows{extra}"), dtype, sigma=14)
    _check(inputs.row_lengths_csr([0] * 2000 + [20000, 0, 5] + [0] * 999, 30000, 3, "hub_between_empties"), dtype)


@pytest.mark.parametrize("W", [4, 8, 16])
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("n", [1_000_003, 2_100_001, 4_200_003, 8_400_001])
def test_every_unit_length(cuda_device, n, dtype, W):
    """Four nonzeros a row (one row has 300,001): from n = 1.3 M rows on a warp takes units
    of 1, 2, 4 or 8 tiles, as W allows."""
    lens = np.full(n, 4, np.int64)
    lens[1::7] = 0
    lens[n // 2] = 300_001
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    rng = np.random.default_rng(n)
    col = rng.integers(0, n, nnz).astype(np.int32)
    a = inputs.CSR(n, n, row_ptr.astype(np.int32), col, 1.0 - rng.random(nnz), f"units{n}")
    _check(a, dtype, W=W)


@pytest.mark.parametrize("mode", ["plain", "ir_bf16"])
def test_expired_wait_then_recovery(cuda_device, mode):
    a = inputs.rmat_transition(15, 16, 2)
    rp, col = torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col).cuda()
    p = mb.plan(rp, col, a.n_rows, a.n_cols)
    v = torch.from_numpy(a.val).cuda()
    p.set_wait_limit(0)
    with pytest.raises(mb.MerbitError) as e:
        mb.pagerank(p, v, 0.85, tol=1e-10, mode=mode, inner_sweeps=8, max_iter=40)
    assert e.value.status == 6
    p.set_wait_limit(-1)
    pi, info = mb.pagerank(p, v, 0.85, tol=1e-10, mode=mode, inner_sweeps=12, max_iter=60)
    assert info["converged"]
    assert oracle.pagerank_residual(a.row_ptr, a.col, a.val, as_f64(pi), 0.85) < 1.1e-10
