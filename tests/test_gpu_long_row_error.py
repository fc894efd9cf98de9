"""Rows of a few tiles: an f32 product's error is that of sums within a tile and one rounding.

Products of width 1 to 32 walk a tile in different orders, and a warp takes up to four tiles; the
error must not grow with either.  The yardstick is a float32 model of the narrowest order: 14
products a lane in turn, the 32 lanes of a tile pairwise, the tiles in 64 bits, one rounding.  A
wider order has a few roundings more a tile: its root mean square may be 1.3 times the model's."""
import numpy as np
import pytest
import torch

import paper_2605_07391_gb300 as mb

pytestmark = pytest.mark.gpu
ROWS, LEN, COLS = 6000, 1700, 200_000        # 22,800 tiles: units of four tiles


def _model(prod):
    """Row sums of float32 products (rows x LEN) in the order described above."""
    rows = prod.shape[0]
    pad = np.zeros((rows, -(-LEN // 448) * 448), np.float32)
    pad[:, :LEN] = prod
    lanes = np.zeros((rows, pad.shape[1] // 14), np.float32)
    for k in range(14):
        lanes += pad.reshape(rows, -1, 14)[:, :, k]
    t = lanes.reshape(rows, -1, 32)
    while t.shape[2] > 1:
        t = t[:, :, ::2] + t[:, :, 1::2]
    return t[:, :, 0].astype(np.float64).sum(1).astype(np.float32)


def _rms(y, y64):
    return float((((y.double() - y64) / y64) ** 2).mean().sqrt())


@pytest.mark.parametrize("k", [1, 4, 8, 13, 16, 32])
def test_error_of_long_rows(cuda_device, k):
    rng = np.random.default_rng(7)
    row_ptr = torch.arange(0, ROWS * LEN + 1, LEN, dtype=torch.int32, device="cuda")
    col = torch.from_numpy(rng.integers(0, COLS, ROWS * LEN).astype(np.int32)).cuda()
    vals = torch.from_numpy(rng.random(ROWS * LEN).astype(np.float32)).cuda()
    X = torch.from_numpy(rng.random((COLS, k)).astype(np.float32)).cuda()
    p = mb.plan(row_ptr, col, ROWS, COLS)
    y = mb.spmm(p, vals, X)
    y64 = torch.stack([(vals.double() * X[:, c].double()[col.long()]).view(ROWS, LEN).sum(1) for c in range(k)], 1)
    v, x, c0 = vals.cpu().numpy(), X[:, 0].cpu().numpy(), col.cpu().numpy()
    prod = (v * x[c0]).reshape(ROWS, LEN)
    model = _rms(torch.from_numpy(_model(prod)), torch.from_numpy(prod.astype(np.float64).sum(1)))
    assert _rms(y, y64) <= 1.3 * model


@pytest.mark.parametrize("k,dtype", [(1, torch.float32), (1, torch.bfloat16), (1, torch.float64), (8, torch.float32),
                                     (32, torch.float32)])
def test_tiles_of_a_long_row_add_up_in_64_bits(cuda_device, k, dtype):
    """Rows of 20 tiles: 2^25 in one tile and -2^25 in another, 2^-6 elsewhere.  Every tile's sum is
    exact in f32, so the row is exact if the tiles are added up without rounding (units of four
    tiles: 40,000 tiles; both large terms lie seven tiles from the row's ends)."""
    rows, length = 2000, 448 * 20
    v = np.full(length, 2.0 ** -6, np.float64)
    for at, sign in ((8 * 448, 1.0), (12 * 448, -1.0)):
        v[at - 448:at + 448] = 0.0               # the large term's tile holds nothing else
        v[at] = sign * 2.0 ** 25
    row_ptr = torch.arange(0, rows * length + 1, length, dtype=torch.int32, device="cuda")
    vals = torch.from_numpy(np.tile(v, rows)).to("cuda", dtype)
    col = torch.zeros(rows * length, dtype=torch.int32, device="cuda")
    p = mb.plan(row_ptr, col, rows, 4)
    xt = torch.float64 if dtype == torch.float64 else torch.float32
    if k == 1:
        y = mb.spmv(p, vals, torch.ones(4, dtype=xt, device="cuda"))
    else:
        y = mb.spmm(p, vals, torch.ones(4, k, device="cuda"))
    assert (y == float(v.sum())).all()


@pytest.mark.parametrize("k", [1, 8, 32])
@pytest.mark.parametrize("what", ["inf", "both", "nan", "overflow"])
def test_long_rows_that_are_not_finite(cuda_device, k, what):
    """Rows of 20 tiles with an infinity, both, a NaN, or finite terms whose sum overflows."""
    rows, length = 2000, 448 * 20
    v = np.ones(length, np.float32)
    at = 8 * 448
    if what in ("inf", "both"):
        v[at] = np.inf
    if what == "both":
        v[at + 2000] = -np.inf
    if what == "nan":
        v[at] = np.nan
    if what == "overflow":
        v[:] = 3e38 / 4000
    row_ptr = torch.arange(0, rows * length + 1, length, dtype=torch.int32, device="cuda")
    vals = torch.from_numpy(np.tile(v, rows)).cuda()
    p = mb.plan(row_ptr, torch.zeros(rows * length, dtype=torch.int32, device="cuda"), rows, 4)
    y = mb.spmv(p, vals, torch.ones(4, device="cuda")) if k == 1 else mb.spmm(p, vals, torch.ones(4, k, device="cuda"))
    assert (torch.isnan(y) if what in ("both", "nan") else y == float("inf")).all()
