"""The bench names the correlation kernel the default engine runs (and takes
that kernel's DRAM figure for the roofline) from its own copy of the library's
choice between the two single-pass kernels above 256 inputs.  These checks keep
that copy equal to the library's build defaults and to the winners measured on
GB300 (1024 channels, 8192 samples, both kernels forced in turn)."""
import ctypes
import importlib.util
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SINGLE_PASS = os.path.join(ROOT, "paper_1503_06202_gb300", "csrc", "single_pass.cu")


def _bench():
    spec = importlib.util.spec_from_file_location("bench_under_test", os.path.join(ROOT, "bench.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    return mod


def _library_defaults():
    src = open(SINGLE_PASS).read()
    return {k: int(v) for k, v in re.findall(r"#define (XENG_\w+) (\d+)", src)}


def test_bench_copy_equals_library_defaults():
    d, b = _library_defaults(), _bench()
    assert (b.PAIR_COST, b.ONEPASS_COST, b.FUSED_MAX_N) == (
        d["XENG_PAIR_COST"], d["XENG_ONEPASS_COST"], d["XENG_FUSED_MAX_N"])


# the faster kernel per N, measured with each forced (ms, one pass / pair):
# 384 2.29 / 3.29, 512 3.60 / 3.33, 640 5.38 / 6.79, 768 7.54 / 6.82,
# 896 10.76 / 11.17, 1024 12.56 / 11.24, 1152 15.61 / 16.83,
# 1408 22.78 / 23.75, 1664 31.62 / 32.79, 1920 48.64 / 41.55
MEASURED_WINNER = {384: "onepass", 512: "pair", 640: "onepass", 768: "pair", 896: "onepass",
                   1024: "pair", 1152: "onepass", 1408: "onepass", 1664: "onepass", 1920: "pair"}


@pytest.mark.parametrize("N", sorted(MEASURED_WINNER))
def test_choice_matches_measured_winner(N):
    assert ("pair" if _bench().use_pair_kernel(N) else "onepass") == MEASURED_WINNER[N]


def test_pair_when_block_count_is_even_above_384():
    # an even number of 128-input blocks pads nothing at 256: the pair kernel's
    # quarter of the MMA instructions per block wins there
    b = _bench()
    for N in range(512, 3585, 256):
        assert b.use_pair_kernel(N), N


@pytest.mark.parametrize("N,kernel", [(16, "correlate_small"), (256, "correlate_small"),
                                      (272, "correlate_onepass"), (2048, "correlate_pair"),
                                      (3584, "correlate_pair"), (3600, "correlate_tc"),
                                      (4096, "correlate_tc"), (250, "correlate_tc"), (1000, "correlate_tc")])
def test_default_engine_path_by_n(N, kernel):
    # single pass for N a multiple of 16 up to the bound; decoded planes otherwise
    assert _bench().correlate_kernel("tensor", N)[0].startswith(kernel)


# The two build parameters hold for every launch shape: a cost of 0 forces that kernel
@pytest.mark.parametrize("pair,onepass", [(0, 36), (118, 0), (118, 36)])
def test_a_cost_of_zero_forces_a_kernel(pair, onepass, tmp_path):
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if shutil.which("g++") is None or not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, so = tmp_path / "rule.cpp", str(tmp_path / "rule.so")
    src.write_text('#include "launch_rule.h"\nusing namespace xeng;\n'
                   'extern "C" int choice(int N, long nf, long nt, int add, int *cut) {\n'
                   '    const int k = single_pass_by_shape(use_pair_kernel(N) ? kSinglePair : kSingleOnepass, N, nf, nt, add, 152);\n'
                   '    *cut = single_pass_cut(k, N, nf, nt, add, 152);\n    return k;\n}\n')
    subprocess.check_call(["g++", "-std=c++17", "-fPIC", "-shared", "-I" + cuda, "-I" + os.path.dirname(SINGLE_PASS),
                           "-DXENG_PAIR_COST=%d" % pair, "-DXENG_ONEPASS_COST=%d" % onepass, str(src), "-o", so])
    lib = ctypes.CDLL(so)
    lib.choice.argtypes = [ctypes.c_int, ctypes.c_long, ctypes.c_long, ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    seen = set()
    for N in (272, 512, 1024, 2048, 3584):
        for F in (1, 4, 26, 64, 1024):
            for T in (1, 200, 8192, 32768):
                for add in (0, 1):
                    cut = ctypes.c_int()
                    k = lib.choice(N, F, T, add, ctypes.byref(cut))
                    seen.add((k, cut.value > 0))
    # 2: one pass, 3: pair kernel, and whether its last round goes to the one pass
    if pair and onepass:
        assert seen == {(3, False), (3, True), (2, False)}
    else:
        assert seen == {(2 if pair else 3, False)}
