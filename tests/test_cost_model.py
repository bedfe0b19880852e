"""Which kernel takes a launch.  Batches choose by N alone between the two
single-pass kernels above 256 inputs, and the bench counts their launches from its
own copy of that choice: equal to the library's build defaults and to the winners
measured on GB300 (1024 channels, 8192 samples, both kernels forced in turn).
Handles and the streaming service choose by the launch's channels and samples too;
the bench names the kernel (and takes its DRAM figure for the roofline) as the
library says it, checked here against measured winners."""
import ctypes
import importlib.util
import os
import re
import shutil
import subprocess

import pytest

import paper_1503_06202_gb300 as xe

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
                                      (4096, "correlate_tc"), (250, "correlate_small"), (1000, "correlate_pair")])
def test_default_engine_path_by_n(N, kernel):
    # 1024 channels x 8192 samples: single pass for every N up to the bound (rows that
    # TMA cannot address are rearranged first); decoded planes above
    assert _bench().correlate_kernel("tensor", N)[0].startswith(kernel)


# (N, channels, samples) and the faster kernel, us a call with the N-only choice / the
# one pass; 256 x 8 x 4096 the N <= 256 kernel's 24 against 31
MEASURED_SHAPE = [(1024, 4, 32768, "onepass"),   # 322 / 207
                  (512, 256, 256, "onepass"),    # 100 / 65
                  (256, 256, 256, "onepass"),    # 32 / 25
                  (256, 8, 1024, "onepass"),     # 22.3 / 14.3
                  (256, 8, 2048, "onepass"),     # 22.5 / 19.2
                  (256, 8, 4096, "small"),
                  (256, 48, 4096, "onepass"),    # 37.9 / 31.3
                  (160, 2, 256, "onepass"),      # 15.0 / 9.0
                  (128, 152, 4096, "onepass"),   # 39.5 / 27.7
                  (128, 152, 32768, "small"),    # 168 / 191
                  (256, 1024, 32768, "small"), (1024, 1024, 8192, "pair"), (2048, 256, 8192, "pair")]


@pytest.mark.parametrize("N,F,T,kernel", MEASURED_SHAPE)
def test_choice_by_launch_shape_matches_measured_winner(N, F, T, kernel, monkeypatch):
    monkeypatch.delenv("XENG_FUSED_KERNEL", raising=False)
    assert _bench().correlate_kernel("tensor", N, F, T)[0].startswith("correlate_" + kernel)


# Above 256 inputs the last channels may go to the one pass: 1024 x 64 x 8192 is 640
# items on 76 clusters, eight rounds (60 channels) and 40 items
def test_last_round_of_few_items_goes_to_the_one_pass(monkeypatch):
    monkeypatch.delenv("XENG_FUSED_KERNEL", raising=False)
    for accumulate in (False, True):
        assert xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR, 1024, 64, 8192, accumulate) == (xe.XENG_KERNEL_PAIR, 60)
        assert xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR, 2048, 1024, 8192, accumulate) == (xe.XENG_KERNEL_PAIR, 1023)
    # 76 channels: ten whole rounds
    assert xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR, 1024, 76, 8192) == (xe.XENG_KERNEL_PAIR, 76)
    monkeypatch.setenv("XENG_FUSED_KERNEL", "pair")
    assert xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR, 1024, 64, 8192) == (xe.XENG_KERNEL_PAIR, 64)
    assert xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR, 1024, 4, 32768) == (xe.XENG_KERNEL_PAIR, 4)


def test_executed_work_counts_whole_tiles():
    b, useful = _bench(), 512 * 513 / 2  # 1216 channels: 48 whole rounds
    assert b.correlate_kernel("tensor", 512, 1216, 8192)[1] == 3 * 256 ** 2 / useful
    assert b.correlate_kernel("planes", 512)[1] == 10 * 128 ** 2 / useful
    useful = 1024 * 1025 / 2
    assert b.correlate_kernel("tensor", 1024, 64, 8192)[1] == pytest.approx(
        (60 * 10 * 256 ** 2 + 4 * 36 * 128 ** 2) / 64 / useful, rel=1e-12)


def test_choice_argument_checks():
    T = xe.XENG_ENGINE_TENSOR
    assert xe.xeng_kernel_choice(xe.XENG_ENGINE_DP4A, 64, 1, 1)[0] == xe.XENG_ERR_ARG
    for args in ((0, 1, 1), (4097, 1, 1), (64, 0, 1), (64, 1, 0), (64, 1, 32769)):
        assert xe.xeng_kernel_choice(T, *args)[0] == xe.XENG_ERR_RANGE
    assert xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR_PLANES, 64, 1, 1)[0] == xe.XENG_KERNEL_PLANES
    # the single-pass engine above the bound: blocks that TMA reads in place
    assert xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR_FUSED, 4096, 256, 8192)[0] == xe.XENG_KERNEL_PAIR
    assert xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR_FUSED, 4001, 256, 8192)[0] == xe.XENG_KERNEL_PLANES
    assert xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR_FUSED, 3583, 256, 8192)[0] == xe.XENG_KERNEL_PAIR


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
                    if pair and onepass:
                        assert (k, cut.value or F) == xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR, N, F, T, add)
    if pair and onepass:
        assert seen == {(xe.XENG_KERNEL_PAIR, False), (xe.XENG_KERNEL_PAIR, True), (xe.XENG_KERNEL_ONEPASS, False)}
    else:
        assert seen == {(xe.XENG_KERNEL_ONEPASS if pair else xe.XENG_KERNEL_PAIR, False)}
