"""A kernel launch of a sparse step that fails partway, on the CPU: the host
code of the library runs over a stand-in for the CUDA runtime that logs every
call and refuses chosen ones.  Nothing may be launched after the refused one
(the next kernel would take positions from what it has not written), and the
touched-row map and the dedup's counters must be cleared before another step
counts into them."""
import concurrent.futures
import ctypes
import os
import subprocess

import pytest

from paper_2607_01455_gb300 import build as B

TESTS = os.path.dirname(os.path.abspath(__file__))
LAUNCH, MEMSET = 1, 2
V, D, MAX_N = 5000, 64, 100000
ERR_CUDA = 5


class Entry(ctypes.Structure):
    _fields_ = [("kind", ctypes.c_int), ("ptr", ctypes.c_void_p), ("bytes", ctypes.c_size_t),
                ("stream", ctypes.c_void_p)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = str(tmp_path_factory.mktemp("fake"))
    quick = ["-O0", "-Xcicc", "-O0", "-Xptxas", "-O0"]  # only the host code runs
    flags = [f for f in B.FLAGS if not f.startswith(("-O", "-lineinfo"))]

    def compile_one(src):
        obj = os.path.join(d, os.path.basename(src) + ".o")
        subprocess.run([B.NVCC, *B.ARCH, *flags, *quick, "-c", src, "-o", obj], check=True, capture_output=True)
        return obj

    srcs = B.sources() + [os.path.join(TESTS, "fake_cudart.cpp")]
    with concurrent.futures.ThreadPoolExecutor(len(srcs)) as ex:
        objs = list(ex.map(compile_one, srcs))
    so = os.path.join(d, "libember_fake.so")
    # -Bsymbolic: its own runtime calls, whatever else the process has loaded
    subprocess.run([B.NVCC, *B.ARCH, "-shared", "-cudart", "none", "-Xlinker", "-Bsymbolic", "-o", so, *objs],
                   check=True)
    lib = ctypes.CDLL(so)
    lib.ember_workspace_bytes.restype = ctypes.c_size_t
    lib.ember_workspace_bytes.argtypes = [ctypes.c_void_p, ctypes.c_int64]
    return lib


class Fake:
    P = ctypes.c_void_p
    ADDR = 1 << 30  # never dereferenced

    def __init__(self, lib):
        self.lib = lib
        self.h = self.P()
        assert lib.ember_create(ctypes.c_int64(V), ctypes.c_int64(D), None, 0, ctypes.byref(self.h)) == 0
        n = lib.ember_workspace_bytes(self.h, MAX_N)
        lib.fake_reset(-1, 0, 0)
        assert lib.ember_bind_workspace(self.h, self.P(1 << 32), ctypes.c_size_t(n), ctypes.c_int64(MAX_N),
                                        None) == 0
        scalars, *self.cleared = self.log()  # binding clears the map and the counters last
        assert len(self.cleared) == 2 and self.cleared[0][2] == 4 * V

    def log(self):
        buf = (Entry * 4096)()
        n = self.lib.fake_log(buf)
        return [(e.kind, e.ptr, e.bytes) for e in buf[:n]]

    def call(self, kind, fail=-1, memset_failures=0, capturing=0):
        """(status, log) of one call whose launch number `fail` is refused."""
        self.lib.fake_reset(fail, memset_failures, capturing)
        a = self.P(self.ADDR)
        if kind[0] == "step":
            st = self.lib.ember_step_sparse(self.h, a, a, kind[1], ctypes.c_int64(kind[2]), a, a,
                                            ctypes.c_float(1e-3), ctypes.c_int64(1), None)
        else:
            st = self.lib.ember_sparse_unique(self.h, a, kind[1], ctypes.c_int64(kind[2]), a, a, a, None)
        return st, self.log()


KINDS = [("step", 1, 0), ("step", 1, 100), ("step", 0, 3072), ("step", 1, 5000), ("step", 0, 100000),
         ("unique", 1, 100), ("unique", 0, 70000)]


@pytest.mark.parametrize("kind", KINDS, ids=str)
def test_a_refused_launch_ends_the_call_and_clears(lib, kind):
    f = Fake(lib)
    st, whole = f.call(kind)
    assert st == 0
    kernels = [e for e in whole if e[0] == LAUNCH]
    assert len(kernels) >= 3
    for k in range(len(kernels)):
        st, log = f.call(kind, fail=k)
        assert st == ERR_CUDA
        assert log == kernels[:k] + f.cleared, k
        assert f.call(kind) == (0, whole)  # the next step has nothing left to clear


@pytest.mark.parametrize("kind", KINDS, ids=str)
def test_a_clear_that_fails_is_made_up_for(lib, kind):
    f = Fake(lib)
    _, whole = f.call(kind)
    st, _ = f.call(kind, fail=1, memset_failures=1)
    assert st == ERR_CUDA
    st, log = f.call(kind, memset_failures=1)  # it fails again: nothing is launched
    assert st == ERR_CUDA and not [e for e in log if e[0] == LAUNCH]
    # a clear that is only captured has not happened yet
    assert f.call(kind, capturing=1) == (0, f.cleared + whole)
    assert f.call(kind) == (0, f.cleared + whole)
    assert f.call(kind) == (0, whole)
