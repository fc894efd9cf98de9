"""Transposes with long runs of empty rows: a tile of the sort (6,144 nonzeros) walks the rows that
start in it up to 12,288, and searches beyond that."""
import numpy as np
import pytest
import torch

import paper_2605_07391_gb300 as mb

pytestmark = pytest.mark.gpu
WALKED = 2 * 6144


def _matrix(counts, n_cols, seed):
    row_ptr = np.zeros(counts.size + 1, np.int64)
    np.cumsum(counts, out=row_ptr[1:])
    col = np.random.default_rng(seed).integers(0, n_cols, int(row_ptr[-1]))
    return row_ptr.astype(np.int32), col.astype(np.int32)


def _check(row_ptr, col, n_cols):
    n_rows = row_ptr.size - 1
    t = mb.transpose(torch.from_numpy(row_ptr).cuda(), torch.from_numpy(col).cuda(), n_rows, n_cols)
    perm = np.argsort(col, kind="stable")
    rows = np.repeat(np.arange(n_rows), np.diff(row_ptr))
    assert np.array_equal(t.perm.cpu().numpy(), perm)
    assert np.array_equal(t.col_t.cpu().numpy(), rows[perm])
    assert np.array_equal(t.row_ptr_t.cpu().numpy(), np.searchsorted(col[perm], np.arange(n_cols + 1)))


@pytest.mark.parametrize("run", [WALKED - 7000, WALKED - 1, WALKED, WALKED + 1, 3 * WALKED, 1_000_003])
@pytest.mark.parametrize("where", ["middle", "edge", "first", "last"])
@pytest.mark.parametrize("n_cols", [300, 5000])                # one digit, two
def test_run_of_empty_rows(cuda_device, run, where, n_cols):
    before = {"middle": 3000, "edge": 6144, "first": 0, "last": 9000}[where]
    after = 0 if where == "last" else 9000
    counts = np.concatenate([np.ones(before, np.int64), np.zeros(run, np.int64), np.ones(after, np.int64)])
    row_ptr, col = _matrix(counts, n_cols, run)
    _check(row_ptr, col, n_cols)


@pytest.mark.parametrize("every", [2, 3, 100, 4096])
def test_sparse_rows(cuda_device, every):
    counts = np.zeros(2_000_000, np.int64)
    counts[::every] = np.random.default_rng(every).integers(0, 12, counts[::every].size)
    row_ptr, col = _matrix(counts, 5000, every)
    _check(row_ptr, col, 5000)


def test_time_of_a_long_run(cuda_device):
    """2^24 empty rows between two dense ones: the rows are not walked by one CTA (15 ms)."""
    counts = np.zeros(1 << 24, np.int64)
    counts[0] = counts[-1] = 3000
    row_ptr, col = (torch.from_numpy(x).cuda() for x in _matrix(counts, 4096, 1))
    times = []
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        t = mb.transpose(row_ptr, col, 1 << 24, 4096)
        e1.record()
        torch.cuda.synchronize()
        times.append(e0.elapsed_time(e1))
        t.destroy()
    assert sorted(times)[2] < 3.0, times
