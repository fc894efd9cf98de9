"""The transpose's radix sort against a stable argsort, bit for bit, where its plan changes: one,
two and three passes (column counts at the edges of the digit widths), tiles that are not full,
long rows, runs of empty rows across tiles, and repeated, unsorted columns."""
import numpy as np
import pytest
import torch

import paper_2605_07391_gb300 as mb

pytestmark = pytest.mark.gpu


def _check(lens, col, n_cols):
    n, nnz = len(lens), int(np.sum(lens))
    row_ptr = np.zeros(n + 1, np.int64)
    np.cumsum(lens, out=row_ptr[1:])
    t = mb.transpose(torch.from_numpy(row_ptr.astype(np.int32)).cuda(), torch.from_numpy(col.astype(np.int32)).cuda(), n, n_cols)
    perm = np.argsort(col, kind="stable")
    rows = np.repeat(np.arange(n), lens)
    ptr = np.searchsorted(col[perm], np.arange(n_cols + 1), side="left")
    assert np.array_equal(t.perm.cpu().numpy(), perm)
    assert np.array_equal(t.col_t.cpu().numpy(), rows[perm])
    assert np.array_equal(t.row_ptr_t.cpu().numpy(), ptr)
    assert ptr[-1] == nnz


@pytest.mark.parametrize("n_cols", [1, 2, 3, 255, 256, 257, 2047, 2048, 2049, 1 << 18, (1 << 20) + 1, 1 << 22, (1 << 22) + 1])
def test_passes(cuda_device, n_cols):
    rng = np.random.default_rng(n_cols)
    for nnz in (1, 6143, 6144, 6145, 40_001):
        lens = rng.multinomial(nnz, np.full(777, 1 / 777))
        lens[100:400] = 0
        lens[5] += nnz - lens.sum()
        col = rng.integers(0, n_cols, nnz) if nnz % 2 else (n_cols * rng.random(nnz) ** 4).astype(np.int64)
        col[-1] = n_cols - 1
        _check(lens, col, n_cols)


def test_rows_across_tiles(cuda_device):
    rng = np.random.default_rng(1)
    lens = np.zeros(60_000, np.int64)
    lens[[0, 3, 40_000, 59_999]] = [30_000, 1, 7_000, 3]
    lens[30_000:30_020] = 613
    _check(lens, rng.integers(0, 5000, lens.sum()), 5000)


def test_dropped_transposes_give_their_memory_back(cuda_device):
    """A transpose whose object and views are gone frees its arrays (they stay while a view lives)."""
    n, nnz = 1000, 4_000_000
    row_ptr = torch.arange(n + 1, dtype=torch.int32, device="cuda") * (nnz // n)
    col = torch.randint(0, n, (nnz,), dtype=torch.int32, device="cuda")
    first = mb.transpose(row_ptr, col).perm               # a view alone keeps the arrays
    want = first.cpu()
    for _ in range(3):
        mb.transpose(row_ptr, col)
    free = torch.cuda.mem_get_info()[0]
    for _ in range(50):                                   # 32 MB each
        t = mb.transpose(row_ptr, col)
        view = t.col_t
        del t, view
    assert free - torch.cuda.mem_get_info()[0] < 200 << 20
    assert torch.equal(first.cpu(), want)
