"""The library linked against tests/fake_cudart.cpp, for tests of its host side without a GPU."""
import ctypes
import os
import shutil
import subprocess

import numpy as np

from paper_2605_07391_gb300 import build as b

HERE = os.path.dirname(os.path.abspath(__file__))


def library(folder):
    """The library's own objects with the stand-in runtime; calls it does not define return 0."""
    b.build()
    objs = [os.path.join(b.BUILD, os.path.basename(s)[:-3] + ".o") for s in b._sources()]
    nvcc = b._nvcc()
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    cxx = shutil.which("g++")
    fake = os.path.join(folder, "fake.o")
    subprocess.run([cxx, "-O1", "-fPIC", "-I", inc, "-c", os.path.join(HERE, "fake_cudart.cpp"), "-o", fake], check=True)

    def symbols(files, flag):
        out = subprocess.run(["nm", flag, *files], check=True, capture_output=True, text=True).stdout
        return {line.split()[-1] for line in out.splitlines() if line.strip() and not line.endswith(":")}

    missing = {s for s in symbols(objs, "-u") if s.startswith(("cuda", "__cuda"))} - symbols([fake], "--defined-only")
    stubs = os.path.join(folder, "stubs.c")
    with open(stubs, "w") as f:
        f.write("".join(f"long {s}() {{ return 0; }}\n" for s in sorted(missing)))
    subprocess.run([shutil.which("gcc"), "-w", "-fno-builtin", "-fPIC", "-c", stubs, "-o", stubs + ".o"], check=True)
    path = os.path.join(folder, "libfake.so")
    subprocess.run([cxx, "-shared", "-Wl,-Bsymbolic", "-o", path, *objs, fake, stubs + ".o"], check=True)
    lib = ctypes.CDLL(path)
    lib.fake_used.restype = lib.fake_idle.restype = ctypes.c_size_t
    lib.fake_first_set.restype = ctypes.c_void_p
    lib.fake_limit.argtypes = [ctypes.c_size_t]
    lib.merbit_last_error.restype = ctypes.c_char_p
    return lib


class Pattern:
    """A CSR pattern in (host) memory and calls of the library on it."""

    def __init__(self, lib, n=1000, degree=4):
        self.lib, self.n, self.nnz = lib, n, n * degree
        self.row_ptr = np.arange(0, self.nnz + 1, degree, dtype=np.int32)
        mem = np.zeros(self.nnz + 4, np.int32)            # col_idx on a 16-byte boundary
        self.col = mem[(-mem.ctypes.data // 4) % 4:][:self.nnz]
        self.col[:] = np.random.default_rng(1).integers(0, n, self.nnz)

    def args(self):
        vp, i64 = ctypes.c_void_p, ctypes.c_int64
        return vp(self.row_ptr.ctypes.data), vp(self.col.ctypes.data), i64(self.n), i64(self.n), i64(self.nnz)

    def plan(self, sigma=14):
        h = ctypes.c_void_p()
        assert self.lib.merbit_plan_ex(*self.args(), sigma, 8, None, ctypes.byref(h)) == 0, self.lib.merbit_last_error()
        return h

    def transpose(self):
        h = ctypes.c_void_p()
        assert self.lib.merbit_transpose(*self.args(), None, ctypes.byref(h)) == 0, self.lib.merbit_last_error()
        return h

    def batch(self):
        h = ctypes.c_void_p()
        off = np.array([0, self.n], np.int64)
        rp, col, n, _, nnz = self.args()
        assert self.lib.merbit_batch_plan(rp, col, n, nnz, ctypes.c_void_p(off.ctypes.data), 1, 14, None,
                                          ctypes.byref(h)) == 0, self.lib.merbit_last_error()
        return h
