"""Host-side rules of the library's device memory, against a stand-in CUDA runtime (no GPU)."""
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
