"""Time shifting (Sec. IV-C-5) through the C ABI: per-input delays applied to
a stream of pushes, bit-exact against the oracle's definition over every
integration window, with ragged inputs, mixed and uniform 16-input chunks,
pushes shorter than the delays, multi-chunk pushes, the maximum delay, host
and device blocks, and the argument checks."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1503_06202_gb300 as xe  # noqa: E402


def run_stream(N, F, t_integ, delays, pushes, dumps_after, seed, host=False):
    """Push blocks of the given sizes, dumping after the listed push indices.
    Returns (stream, [(t_a, t_b, dump)])."""
    rng = np.random.default_rng(seed)
    total = sum(pushes)
    stream = rng.integers(0, 256, size=(total, F, N), dtype=np.uint8)
    eng = xe.XEngine(N, F, t_integ)
    eng.set_delays(delays)
    out = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    got, t, t_a = [], 0, 0
    for k, n in enumerate(pushes):
        blk = stream[t:t + n]
        eng.push(blk if host else torch.from_numpy(blk).cuda(), n)
        t += n
        if k in dumps_after:
            assert eng.dump(out) == t - t_a
            got.append((t_a, t, out.cpu().numpy().astype(np.int64)))
            t_a = t
    eng.close()
    return stream, got


def check(stream, delays, got):
    for t_a, t_b, v in got:
        want = oracle.correlate_shifted(stream, delays, t_a, t_b)
        assert np.array_equal(v, want), (t_a, t_b)


def test_shift_ragged_inputs_short_pushes():
    # N = 200: not a multiple of 16 (every chunk on the byte path); pushes
    # shorter than the larger delays, so early samples come from the history
    N, F = 200, 3
    rng = np.random.default_rng(1)
    delays = rng.integers(0, 300, N).astype(np.int32)
    delays[:50] = 0
    pushes = [100, 37, 256, 1, 500, 129, 300]
    stream, got = run_stream(N, F, 4096, delays, pushes, {1, 2, 4, 6}, seed=2)
    check(stream, delays, got)


def test_shift_uniform_and_mixed_chunks_host_blocks():
    # N = 256: chunks of 16 inputs sharing one delay take the vector loads,
    # one chunk mixes delays; blocks come from host memory
    N, F = 256, 2
    delays = np.zeros(N, np.int32)
    delays[16:32] = 77          # one uniform delayed chunk
    delays[64:80] = 1000        # another, longer than the first push
    delays[130] = 5             # a mixed chunk
    delays[255] = 3
    pushes = [640, 640, 1280, 333]
    stream, got = run_stream(N, F, 8192, delays, pushes, {0, 2, 3}, seed=3, host=True)
    check(stream, delays, got)


def test_shift_tma_decode_ragged_blocks():
    # N = 272 (a multiple of 16: the TMA decode, with a last block of 16
    # inputs): delayed inputs in a mixed chunk, in the last block, and one
    # delayed longer than the pushes; pushes with ragged sample tiles
    N, F = 272, 2
    delays = np.zeros(N, np.int32)
    delays[0] = 2000
    delays[140:144] = 9
    delays[260] = 50
    delays[271] = 1
    pushes = [300, 129, 1000, 64]
    stream, got = run_stream(N, F, 4096, delays, pushes, {1, 3}, seed=6)
    check(stream, delays, got)


def test_shift_multi_chunk_push_and_max_delay():
    # a push longer than one 65,536-sample round, and the largest delay
    N, F = 32, 1
    delays = np.zeros(N, np.int32)
    delays[0] = xe.XENG_MAX_DELAY
    delays[7] = 70000
    delays[8:16] = 12345
    pushes = [150000, 100]
    stream, got = run_stream(N, F, 200000, delays, pushes, {1}, seed=4)
    check(stream, delays, got)


def test_shift_restores_correlation_of_a_delayed_copy():
    # input 1 carries input 0's signal D samples late: delaying input 0 by D
    # makes V_01 equal the autocorrelation over the overlap, as intended
    N, F, T, D = 16, 1, 4096, 300
    rng = np.random.default_rng(5)
    stream = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    stream[D:, :, 1] = stream[:T - D, :, 0]
    delays = np.zeros(N, np.int32)
    delays[0] = D
    eng = xe.XEngine(N, F, T)
    eng.set_delays(delays)
    eng.push(torch.from_numpy(stream).cuda(), T)
    out = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    eng.dump(out)
    v = out.cpu().numpy().astype(np.int64)
    assert np.array_equal(v, oracle.correlate_shifted(stream, delays))
    k01 = int(oracle.triangle_index(0, 1, N))
    x0 = (stream[:T - D, 0, 0].astype(np.int64) >> 4) - 8, (stream[:T - D, 0, 0].astype(np.int64) & 15) - 8
    auto = int((x0[0] ** 2 + x0[1] ** 2).sum())
    assert v[0, k01, 0] == auto and v[0, k01, 1] == 0
    eng.close()


def test_shift_argument_checks_and_removal():
    N, F = 64, 1
    eng = xe.XEngine(N, F, 1024)
    bad = np.zeros(N, np.int32)
    bad[3] = xe.XENG_MAX_DELAY + 1
    assert xe.xeng_set_delays(eng.h, bad) == xe.XENG_ERR_RANGE
    bad[3] = -1
    assert xe.xeng_set_delays(eng.h, bad) == xe.XENG_ERR_RANGE
    d = np.zeros(N, np.int32)
    d[5] = 9
    eng.set_delays(d)
    blk = torch.from_numpy(np.random.default_rng(6).integers(0, 256, (256, F, N), dtype=np.uint8)).cuda()
    out = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    assert xe.xeng_correlate(eng.h, blk, 256, out) == xe.XENG_ERR_UNSUPPORTED
    assert xe.xeng_set_engine(eng.h, xe.XENG_ENGINE_DP4A) == xe.XENG_ERR_UNSUPPORTED
    # removing the delays (None, or all zero) brings back the plain path
    eng.set_delays(None)
    assert xe.xeng_correlate(eng.h, blk, 256, out) == xe.XENG_OK
    assert np.array_equal(out.cpu().numpy().astype(np.int64), oracle.correlate(blk.cpu().numpy()))
    eng.set_delays(np.zeros(N, np.int32))
    assert xe.xeng_correlate(eng.h, blk, 256, out) == xe.XENG_OK
    # the dp4a engine refuses delays
    eng.set_engine(xe.XENG_ENGINE_DP4A)
    assert xe.xeng_set_delays(eng.h, d) == xe.XENG_ERR_UNSUPPORTED
    eng.close()


# Delayed inputs in some 128-input blocks only (copied, the others read in place),
# whole 16-input chunks and single inputs, pushes longer and shorter than the
# delays and across the ring's end
@pytest.mark.parametrize("N,F,delays", [(512, 26, {0: 5, 130: 700, 131: 700}), (272, 2, {i: 40 for i in range(16, 32)}),
                                        (256, 3, {3: 1, 255: 999}), (1040, 1, {1039: 300, 500: 1}),
                                        (61, 4, {60: 17, 0: 1000})])
def test_shift_some_blocks(N, F, delays):
    d = np.zeros(N, np.int32)
    for i, v in delays.items():
        d[i] = v
    stream, got = run_stream(N, F, 2000, d, [900, 100, 700, 200, 1000], {1, 3, 4}, seed=N + F)
    check(stream, d, got)


# The same through the kernel over 256-input block pairs: substituted blocks in either
# CTA's half, both or neither, in the rows and the columns of diagonal pairs and others,
# in a last block of 16 inputs
@pytest.mark.parametrize("N,F,delays", [(1040, 3, {5: 700, 300: 1, 640: 41, 1039: 300}), (512, 2, {200: 33}),
                                        (528, 1, {0: 9, 128: 800, 256: 2, 384: 7, 520: 64}), (2048, 1, {1900: 500})])
def test_shift_some_blocks_by_pair_kernel(N, F, delays, monkeypatch):
    monkeypatch.setenv("XENG_FUSED_KERNEL", "pair")
    assert xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR, N, F, 900)[0] == xe.XENG_KERNEL_PAIR
    d = np.zeros(N, np.int32)
    for i, v in delays.items():
        d[i] = v
    stream, got = run_stream(N, F, 2000, d, [900, 100, 700, 200], {1, 3}, seed=N + F)
    check(stream, d, got)


# Substituted blocks across the cut of a launch whose last round goes to the one pass:
# 1280 x 17 channels, 15 by the pair kernel; a push that stores and one that adds
def test_shift_across_the_cut_of_a_launch():
    N, F, T, sms = 1280, 17, 6000, torch.cuda.get_device_properties(0).multi_processor_count
    kernel, cut = xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR, N, F, T, False, sms)
    assert kernel == xe.XENG_KERNEL_PAIR and 0 < cut < F
    assert xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR, N, F, T, True, sms) == (kernel, cut)
    d = np.zeros(N, np.int32)
    d[[5, 300, 700, 701, 1279]] = 7000, 1, 41, 5999, 300
    g = torch.Generator(device="cuda")
    g.manual_seed(9)
    stream = torch.randint(0, 256, (2 * T, F, N), dtype=torch.uint8, device="cuda", generator=g)
    eng = xe.XEngine(N, F, 2 * T)
    eng.set_delays(d)
    for k in range(2):
        eng.push(stream[k * T:(k + 1) * T])
        st = eng.stats(reset=True)
        assert st["correlate_launches"] == 1 and st["launches"] == 3  # rearranged, then two
    out = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    assert eng.dump(out) == 2 * T
    eng.close()
    keep = [0, cut - 1, cut, F - 1]
    want = oracle.correlate_shifted(np.ascontiguousarray(stream[:, keep].cpu().numpy()), d, 0, 2 * T)
    assert np.array_equal(out[keep].cpu().numpy().astype(np.int64), want)


# Many delayed inputs and a long integration: the history has no room for the pushes'
# own samples, which are read from the block; 65 channels of 1040 inputs
def test_shift_history_without_room_for_a_round():
    N, F, pushes = 1040, 65, [150, 64, 300]
    rng = np.random.default_rng(5)
    d = rng.integers(1, 120, N).astype(np.int32)
    d[-1] = 400
    stream = rng.integers(0, 256, size=(sum(pushes), F, N), dtype=np.uint8)
    eng = xe.XEngine(N, F, 32768)
    eng.set_delays(d)
    out = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    t = 0
    for k, n in enumerate(pushes):
        eng.push(torch.from_numpy(stream[t:t + n]).cuda(), n)
        t += n
        if k > 0:
            t_a = 0 if k == 1 else sum(pushes[:2])
            assert eng.dump(out) == t - t_a
            got = out[[0, F - 1]].cpu().numpy().astype(np.int64)
            assert np.array_equal(got, oracle.correlate_shifted(np.ascontiguousarray(stream[:, [0, F - 1]]), d, t_a, t))
    eng.close()


# A captured push and dump, replayed: every replay goes on from where the history's
# ring is, pushes of 300 samples shorter than the delays, an odd number of replays
def test_shift_captured_pushes():
    N, F, n = 272, 2, 300
    d = np.zeros(N, np.int32)
    d[[3, 130]] = 700, 41
    stream = np.random.default_rng(8).integers(0, 256, size=(6 * n, F, N), dtype=np.uint8)
    eng = xe.XEngine(N, F, 4096)
    eng.set_delays(d)
    block = torch.from_numpy(stream[:n]).cuda()
    out = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    eng.push(block, n, side.cuda_stream)
    assert eng.dump(out, side.cuda_stream) == n
    side.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        eng.push(block, n, side.cuda_stream)
        eng.dump(out, side.cuda_stream)
    for k in range(1, 6):
        block.copy_(torch.from_numpy(stream[k * n:(k + 1) * n]))
        torch.cuda.synchronize()
        graph.replay()
        torch.cuda.synchronize()
        want = oracle.correlate_shifted(stream[:(k + 1) * n], d, k * n, (k + 1) * n)
        assert np.array_equal(out.cpu().numpy().astype(np.int64), want), k
    eng.close()


# Pushes that are rearranged and pushes that decode to planes (8192 samples and more of
# few channels) in one stream: the history goes on from one to the other, pushes longer
# than it and shorter than the delays among them
@pytest.mark.parametrize("N,F,delays", [(272, 2, {3: 700, 130: 9500, 271: 1}), (512, 3, {200: 20000, 511: 40})])
def test_shift_pushes_rearranged_and_decoded(N, F, delays):
    d = np.zeros(N, np.int32)
    for i, v in delays.items():
        d[i] = v
    stream, got = run_stream(N, F, 30000, d, [900, 8192, 100, 300, 9000, 8191, 8500, 700], {1, 2, 4, 5, 7}, seed=N + F)
    check(stream, d, got)
