"""Host-side rules of the library's device memory, against a stand-in CUDA runtime (no GPU)."""
import ctypes

import numpy as np
import pytest

from tests import fake_runtime as fr


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fr.library(str(tmp_path_factory.mktemp("fake")))


@pytest.mark.parametrize("kind", ["plan", "transpose", "batch"])
def test_destroy_waits_for_the_objects_own_device(lib, kind):
    lib.fake_reset()
    h = getattr(fr.Pattern(lib), kind)()       # on device 0
    used = lib.fake_used()
    lib.cudaSetDevice(1)
    lib.fake_busy(0, 1)                        # a product on device 0 is still running
    getattr(lib, f"merbit_{kind}_destroy")(h)
    assert lib.fake_violations() == 0, "memory went back to the pool under running work"
    assert lib.fake_used() < used
    assert lib.fake_device() == 1


@pytest.mark.parametrize("kind", ["plan", "transpose", "batch"])
def test_destroy_during_a_capture(lib, kind):
    lib.fake_reset()
    h = getattr(fr.Pattern(lib), kind)()
    lib.fake_busy(0, 1)
    lib.fake_capture(1)                        # some thread captures a stream
    getattr(lib, f"merbit_{kind}_destroy")(h)
    lib.fake_capture(0)
    assert lib.fake_violations() == 0, "memory went back to the pool under running work"
    assert not lib.fake_broken(), "the capture was broken"


@pytest.mark.parametrize("kind", ["bicgstab", "batch"])
def test_state_is_clear_after_a_give_up(lib, kind):
    """A kernel that gave up may leave sums in the accumulators between units, not the error bit
    alone: both are cleared before the error is reported."""
    lib.fake_reset()
    m = fr.Pattern(lib)
    h = m.batch() if kind == "batch" else m.plan()
    size = ctypes.c_size_t()
    at = lib.fake_first_set(ctypes.byref(size))    # the new plan's state and accumulators
    state = np.ctypeslib.as_array((ctypes.c_ubyte * size.value).from_address(at))
    state[:] = 0xFF
    v = np.zeros(m.nnz + 2)
    v = v[(-v.ctypes.data // 8) % 2:][:m.nnz]      # values on a 16-byte boundary
    b, x = np.zeros(m.n), np.zeros(m.n)
    vp, f64 = ctypes.c_void_p, ctypes.c_double
    if kind == "batch":
        st = lib.merbit_batch_pagerank(h, 1, vp(v.ctypes.data), f64(0.85), f64(0.0), 2, vp(x.ctypes.data), None, None,
                                       None, None)
    else:
        st = lib.merbit_bicgstab(h, vp(v.ctypes.data), vp(b.ctypes.data), vp(x.ctypes.data), f64(0.0), 2, None, None,
                                 None, None, None)
    assert st == 6, lib.merbit_last_error()
    assert not state.any()
    getattr(lib, "merbit_batch_destroy" if kind == "batch" else "merbit_plan_destroy")(h)


@pytest.mark.parametrize("call", ["autotune", "hot", "host_async"])
def test_idle_pool_memory_is_given_back(lib, call):
    """What the pool holds for later does not make another allocation of the library fail."""
    lib.fake_reset()
    m = fr.Pattern(lib)
    h = m.plan()
    for p in [m.plan() for _ in range(12)]:
        lib.merbit_plan_destroy(p)
    assert lib.fake_idle() > 500_000
    lib.fake_limit(100)
    v, x, y = np.zeros(m.nnz), np.zeros(m.n), np.zeros(m.n)
    vp, i64 = ctypes.c_void_p, ctypes.c_int64
    if call == "autotune":
        cand, best = (ctypes.c_int * 1)(14), ctypes.c_int()
        st = lib.merbit_autotune_sigma(*m.args(), 0, vp(v.ctypes.data + -v.ctypes.data % 16), cand, 1, 1, None,
                                       ctypes.byref(best), None)
    elif call == "hot":
        st = lib.merbit_plan_set_hot_columns(h, 64, ctypes.c_double(0.0), None, None, None)
    else:
        st = lib.merbit_spmv_host_async(h, 0, vp(v.ctypes.data + -v.ctypes.data % 16), vp(x.ctypes.data), vp(y.ctypes.data),
                                        None)
    assert st == 0, (st, lib.merbit_last_error())
    lib.merbit_plan_destroy(h)


@pytest.mark.parametrize("k", [1, 8, 13])
def test_first_spmm_of_a_plan_takes_pool_memory(lib, k):
    lib.fake_reset()
    m = fr.Pattern(lib)
    h = m.plan()
    v, X, Y = np.zeros(m.nnz + 4, np.float32), np.zeros(m.n * k + 4, np.float32), np.zeros(m.n * k + 4, np.float32)
    at = [ctypes.c_void_p(t.ctypes.data + -t.ctypes.data % 16) for t in (v, X, Y)]
    before, used = lib.fake_mallocs(), lib.fake_used()
    k64 = ctypes.c_int64(k)
    assert lib.merbit_spmm(h, *at, k64, k64, k64, None) == 0, lib.merbit_last_error()
    assert lib.fake_mallocs() == before
    assert (lib.fake_used() == used) == (k == 1)      # one column needs no accumulators
    lib.merbit_plan_destroy(h)


@pytest.mark.parametrize("call", ["plan", "transpose", "batch", "autotune", "bicgstab"])
def test_a_refused_allocation_is_reported_once(lib, call):
    lib.fake_reset()
    m = fr.Pattern(lib)
    h = m.plan()
    v, x, y = (np.zeros(s + 2) for s in (m.nnz, m.n, m.n))
    vp, out = ctypes.c_void_p, ctypes.c_void_p()
    at = [vp(t.ctypes.data + -t.ctypes.data % 16) for t in (v, x, y)]
    lib.fake_limit(100)
    if call == "plan":
        st = lib.merbit_plan_ex(*m.args(), 14, 8, None, ctypes.byref(out))
    elif call == "transpose":
        st = lib.merbit_transpose(*m.args(), None, ctypes.byref(out))
    elif call == "batch":
        off, (rp, col, n, _, nnz) = np.array([0, m.n], np.int64), m.args()
        st = lib.merbit_batch_plan(rp, col, n, nnz, vp(off.ctypes.data), 1, 14, None, ctypes.byref(out))
    elif call == "autotune":
        cand, best = (ctypes.c_int * 1)(14), ctypes.c_int()
        st = lib.merbit_autotune_sigma(*m.args(), 1, at[0], cand, 1, 1, None, ctypes.byref(best), None)
    else:
        st = lib.merbit_bicgstab(h, *at, ctypes.c_double(0.0), 2, None, None, None, None, None)
    assert st == 3, lib.merbit_last_error()      # ENOMEM
    assert lib.merbit_spmv_ex(h, 1, 1, *at, 0, None) == 0, lib.merbit_last_error()
    lib.merbit_plan_destroy(h)
