"""BiCGSTAB and batched PageRank after a solve in which the stage waits gave up (every wait is
bounded): the error is reported, and the next calls are right again."""
import ctypes

import numpy as np
import pytest
import torch

import inputs
import oracle
import paper_2605_07391_gb300 as mb
from tests.gpu_helpers import TOL, as_f64, check_rel

pytestmark = pytest.mark.gpu
EDEVICE = 6
LIMITS = [0, 1]


def _gives_up(call):
    try:
        call()
    except mb.MerbitError as e:
        assert e.status == EDEVICE
        return True
    return False


@pytest.mark.parametrize("scale", [13, 16])          # one launch a product, and two
def test_bicgstab(cuda_device, scale):
    a = inputs.rmat_transition(scale, 16, 2)
    rp, col = torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col).cuda()
    p = mb.plan(rp, col)
    v = torch.from_numpy(a.val).cuda()
    x = torch.from_numpy(inputs.uniform_vector(a.n_cols, 3)).cuda()
    y_ref, d = oracle.spmv(a.row_ptr, a.col, a.val, as_f64(x))
    failed = 0
    for limit in LIMITS:
        p.set_wait_limit(limit)
        failed += _gives_up(lambda: mb.bicgstab(p, v, x, tol=0.0, max_iter=2))
        p.set_wait_limit(-1)
        y = mb.spmv(p, v, x)
        p.sync()
        check_rel(as_f64(y), y_ref, d, TOL[torch.float64], f"after a give-up at {limit} polls")
    assert failed


@pytest.mark.parametrize("scale", [13, 16])
def test_batch(cuda_device, scale):
    a = inputs.rmat_transition(scale, 16, 2)
    rp, col = torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col).cuda()
    v = torch.from_numpy(a.val).cuda()
    off = np.array([0, a.n_rows])
    ref = mb.Batch(rp, col, off).pagerank(v, 0.85, tol=0.0, max_iter=1)[0]
    failed = 0
    for limit in LIMITS:
        b = mb.Batch(rp, col, off)
        lib = mb.merbit.load()
        plan = ctypes.c_void_p(lib.merbit_batch_get_plan(b.handle))
        lib.merbit_plan_set_wait_limit(plan, limit)
        failed += _gives_up(lambda: b.pagerank(v, 0.85, tol=0.0, max_iter=2))
        lib.merbit_plan_set_wait_limit(plan, -1)
        pi = b.pagerank(v, 0.85, tol=0.0, max_iter=1)[0]      # recorded anew: another max_iter
        # one update from 1/n: the rows differ by rounding at most
        assert ((pi - ref).abs() <= 1e-13 * ref).all(), f"after a give-up at {limit} polls"
    assert failed


def test_batch_follows_the_plans_wait_limit(cuda_device):
    """The kept solve is recorded with the plan's wait limit: a new limit records it again."""
    a = inputs.rmat_transition(13, 16, 2)
    rp, col = torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col).cuda()
    v = torch.from_numpy(a.val).cuda()
    b = mb.Batch(rp, col, np.array([0, a.n_rows]))
    pi = torch.empty(a.n_rows, dtype=torch.float64, device="cuda")
    lib = mb.merbit.load()
    plan = ctypes.c_void_p(lib.merbit_batch_get_plan(b.handle))
    for limit, gives_up in ((-1, False), (0, True), (-1, False)):
        lib.merbit_plan_set_wait_limit(plan, limit)
        assert _gives_up(lambda: b.pagerank(v, 0.85, tol=1e-10, pi=pi)) == gives_up, limit
