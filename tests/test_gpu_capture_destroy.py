"""Objects destroyed while a stream is being captured: the capture stays whole, and the memory
waits for the work that still uses it."""
import threading

import numpy as np
import pytest
import torch

import inputs
import paper_2605_07391_gb300 as mb
from tests.gpu_helpers import upload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode", ["relaxed", "thread_local", "global"])
@pytest.mark.parametrize("other_thread", [False, True])
def test_destroy_during_a_capture(cuda_device, mode, other_thread):
    a = inputs.rmat_transition(12, 16, 1)
    rp, col, vals = upload(a)
    keep = mb.plan(rp, col)
    x = torch.rand(a.n_cols, device="cuda")
    y, y_ref = torch.empty_like(x), mb.spmv(keep, vals, x)
    t = mb.transpose(rp, col)
    doomed = [mb.plan(rp, col), t, mb.Batch(rp, col, np.array([0, a.n_rows]))]
    src = torch.rand(a.nnz, device="cuda")
    out = torch.empty_like(src)
    torch.cuda.synchronize()
    mb.gather(src, t.perm, out)                # may still read the transpose when it is destroyed

    def destroy():
        torch.cuda.set_device(0)
        for d in doomed:
            d.destroy()

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode=mode):
        mb.spmv(keep, vals, x, y)
        if other_thread:
            th = threading.Thread(target=destroy)
            th.start()
            th.join()
        else:
            destroy()
        mb.spmv(keep, vals, y_ref, y)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, mb.spmv(keep, vals, y_ref))


@pytest.mark.parametrize("kind", ["plan", "transpose"])
def test_destroy_waits_for_other_streams(cuda_device, kind):
    a = inputs.rmat_transition(18, 16, 1)
    rp, col, vals = upload(a)
    p, t = mb.plan(rp, col), mb.transpose(rp, col)
    x, src = torch.rand(a.n_cols, device="cuda"), torch.rand(a.nnz, device="cuda")
    y, out = torch.empty_like(x), torch.empty_like(src)
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        for _ in range(300):
            mb.spmv(p, vals, x, y) if kind == "plan" else mb.gather(src, t.perm, out)
    assert not side.query()
    (p if kind == "plan" else t).destroy()
    assert side.query()
