"""The SpMM where its routes differ, every row of every column against the float64 oracle: rows
of X off 16-byte boundaries (padded copies, or one-column slices when the matrix has few
nonzeros or the stream is captured), Y off them, one contiguous column (the plain product), and
rows over several warps' units."""
import numpy as np
import pytest
import torch

import inputs
import oracle
import paper_2605_07391_gb300 as mb
from tests.gpu_helpers import TOL, as_f64, check_rel, make_plan

pytestmark = pytest.mark.gpu


def _check(a, vals, X, Y, what):
    x64 = as_f64(X)
    for c in range(X.shape[1]):
        ref, d = oracle.spmv(a.row_ptr, a.col, as_f64(vals), x64[:, c])
        check_rel(as_f64(Y[:, c]), ref, d, TOL[torch.float32], f"{what} column {c}")


MATRICES = {
    # 2.5 nonzeros per row: no padded copies; then enough of them, with rows of 20,000 and 70,000
    "sparse": lambda: inputs.row_lengths_csr([0, 5] * 3000, 6000, 1),
    "hubs": lambda: inputs.row_lengths_csr([3, 0, 12, 448, 1] * 1000 + [20000, 0, 70000], 80000, 2),
    "rmat": lambda: inputs.rmat_uniform(13, 16, 3, 3),
}


@pytest.mark.parametrize("k", [1, 2, 3, 5, 13, 33, 36])
@pytest.mark.parametrize("name", sorted(MATRICES))
def test_odd_rows(cuda_device, name, k):
    a = MATRICES[name]()
    p, _ = make_plan(a)
    vals = torch.from_numpy(a.val).to("cuda", torch.float32)
    g = torch.Generator(device="cuda").manual_seed(k)
    for ldx, ldy, off in ((k, k, 0), (k + 3, k + 1, 1), (-(-k // 4) * 4, k, 0), (k, -(-k // 4) * 4, 0)):
        xb = torch.rand(a.n_cols * ldx + off, generator=g, device="cuda")[off:]
        X = xb.view(a.n_cols, ldx)[:, :k]
        Y = torch.full((a.n_rows, ldy), float("nan"), device="cuda")[:, :k]
        for _ in range(2):
            mb.spmm(p, vals, X, Y)
        p.sync()
        _check(a, vals, X, Y, f"{name} k={k} ldx={ldx} ldy={ldy}")


def test_captured_call_keeps_no_buffer(cuda_device):
    """A captured call replays right after wider eager calls have replaced the padded copies."""
    a = MATRICES["rmat"]()
    p, _ = make_plan(a)
    vals = torch.from_numpy(a.val).to("cuda", torch.float32)
    X = torch.rand(a.n_cols, 5, device="cuda")
    Y = torch.empty(a.n_rows, 5, device="cuda")
    mb.spmm(p, vals, X, Y)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        mb.spmm(p, vals, X, Y)
    mb.spmm(p, vals, torch.rand(a.n_cols, 33, device="cuda"))
    torch.cuda.synchronize()
    X.uniform_()
    Y.fill_(float("nan"))
    graph.replay()
    torch.cuda.synchronize()
    _check(a, vals, X, Y, "replay")
