"""xeng_set_delays where device memory runs out: the library's host code against a
runtime on host memory (fake_cuda.cpp) whose allocations fail one at a time.  A list
that could not be allocated is an error, whatever else would still fit; only the
history itself is tried again, smaller."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

import paper_1503_06202_gb300 as xe

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
N, F, T, DELAY = 40, 3, 5000, 70  # delayed inputs 1, 17, 18
ROW = 3 * F


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    if shutil.which("g++") is None or not os.path.exists(os.path.join(CUDA, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    so = str(tmp_path_factory.mktemp("fake") / "libxeng_fake.so")
    csrc = os.path.join(ROOT, "paper_1503_06202_gb300", "csrc")
    # -Bsymbolic: its own runtime, whatever libcudart the process holds; the kernels'
    # launchers stay unresolved and are never called
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-x", "c++", os.path.join(csrc, "xeng_api.cu"),
                           os.path.join(ROOT, "tests", "fake_cuda.cpp"), "-I" + CUDA, "-I" + csrc,
                           "-I" + os.path.join(ROOT, "include"), "-Wl,-Bsymbolic", "-Wl,-z,lazy",
                           "-Wl,--unresolved-symbols=ignore-all", "-o", so])
    lib = ctypes.CDLL(so, mode=os.RTLD_LAZY | os.RTLD_LOCAL)
    lib.fake_allocs.argtypes = [ctypes.c_long, ctypes.c_size_t]
    lib.fake_alloc_count.restype = lib.fake_live.restype = ctypes.c_long
    lib.fake_live_bytes.restype = ctypes.c_size_t
    lib.xeng_create.argtypes = [ctypes.c_int32, ctypes.c_int32, ctypes.c_int64, ctypes.POINTER(ctypes.c_void_p)]
    lib.xeng_set_delays.argtypes = [ctypes.c_void_p, ctypes.c_void_p]
    lib.xeng_set_engine.argtypes = [ctypes.c_void_p, ctypes.c_int32]
    lib.xeng_destroy.argtypes = [ctypes.c_void_p]
    return lib


ALL = 2 ** 60


@pytest.fixture
def handle(fake):
    fake.fake_allocs(-1, ALL)
    h = ctypes.c_void_p()
    assert fake.xeng_create(N, F, T, ctypes.byref(h)) == xe.XENG_OK
    yield h
    fake.fake_allocs(-1, ALL)
    fake.xeng_destroy(h)
    assert fake.fake_live() == 0


def delays():
    d = np.zeros(N, np.int32)
    d[[1, 17, 18]] = DELAY, 3, 5
    return d


def shifted(fake, h):
    """The handle holds delays: it then refuses the engine that has none."""
    rc = fake.xeng_set_engine(h, xe.XENG_ENGINE_DP4A)
    assert rc in (xe.XENG_OK, xe.XENG_ERR_UNSUPPORTED)
    fake.xeng_set_engine(h, xe.XENG_ENGINE_TENSOR)
    return rc == xe.XENG_ERR_UNSUPPORTED


def test_each_allocation_failing_alone(fake, handle):
    d = delays()
    live, held = fake.fake_live(), fake.fake_live_bytes()
    assert fake.xeng_set_delays(handle, d.ctypes.data) == xe.XENG_OK and shifted(fake, handle)
    full = fake.fake_live_bytes() - held
    n = fake.fake_live() - live
    assert n == 7  # five lists, the history and where it stands
    again = 0
    for k in range(n):
        fake.fake_allocs(k, ALL)
        rc = fake.xeng_set_delays(handle, d.ctypes.data)
        tried = fake.fake_alloc_count()
        fake.fake_allocs(-1, ALL)
        if rc == xe.XENG_OK:  # the history, made again without a push's own samples
            assert tried == n + 1 and fake.fake_live() - live == n and shifted(fake, handle), k
            assert full - (fake.fake_live_bytes() - held) == T * ROW, k
            again += 1
        else:
            assert rc == xe.XENG_ERR_NOMEM and tried == k + 1, k
            assert fake.fake_live() == live and not shifted(fake, handle), k
    assert again == 1
    assert fake.xeng_set_delays(handle, None) == xe.XENG_OK and fake.fake_live() == live


def test_history_too_large_either_way(fake, handle):
    d = delays()
    fake.fake_allocs(-1, DELAY * ROW)  # room for the delays' samples alone
    assert fake.xeng_set_delays(handle, d.ctypes.data) == xe.XENG_OK and shifted(fake, handle)
    fake.fake_allocs(-1, DELAY * ROW - 1)
    assert fake.xeng_set_delays(handle, d.ctypes.data) == xe.XENG_ERR_NOMEM and not shifted(fake, handle)
