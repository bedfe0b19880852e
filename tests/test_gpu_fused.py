"""The fused decode + correlation.  Up to 256 inputs, single
CTAs over 128-input blocks: bit-exact against the oracle for tiny N (tiles
mostly padding), up to and above 128 inputs (diagonal items of two channels;
row items and diagonal items of the upper input halves), odd channel counts (a
diagonal item of one channel), ragged sample counts, one sample, several
launches adding into int32, pushes in pieces, host buffers, and many items per
CTA (both parities of the item sums, store and add).  Then both single passes
over block pairs, each forced for every case."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1503_06202_gb300 as xe  # noqa: E402


def correlate(blk, pieces=None, host=False, t_integ=None, engine=xe.XENG_ENGINE_TENSOR):
    T, F, N = blk.shape
    eng = xe.XEngine(N, F, t_integ or max(T, 1), engine)
    out = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    src = blk if host else torch.from_numpy(blk).cuda()
    if pieces:
        t = 0
        for p in pieces + [T - sum(pieces)]:
            eng.push(src[t:t + p], p)
            t += p
        eng.dump(out)
    else:
        eng.correlate(src, out, T)
    torch.cuda.synchronize()
    eng.close()
    return out.cpu().numpy().astype(np.int64)


@pytest.mark.parametrize("T,F,N", [(1, 1, 16), (127, 2, 16), (129, 3, 32), (1000, 2, 96), (300, 1, 128),
                                   (4097, 2, 144), (513, 2, 240), (1, 1, 256), (2049, 3, 256)])
def test_fused_shapes(T, F, N):
    rng = np.random.default_rng(T * 131 + F * 17 + N)
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    assert np.array_equal(correlate(blk), oracle.correlate(blk)), (T, F, N)


def test_fused_several_launches_and_pieces():
    # 140,000 samples = three launches of <= 65,536 adding into int32
    rng = np.random.default_rng(5)
    T, F, N = 140000, 2, 256
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    want = oracle.correlate(blk)
    assert np.array_equal(correlate(blk), want)
    assert np.array_equal(correlate(blk, pieces=[100, 65536, 3]), want)


def test_fused_int32_beyond_f32_range():
    # every sample -8-8i over 140,000 samples: Re = 17,920,000 > 2^24
    T, F, N = 140000, 1, 64
    out = correlate(np.zeros((T, F, N), np.uint8))
    assert (out[..., 0] == 128 * T).all() and (out[..., 1] == 0).all()


def test_fused_host_buffers_and_many_channels():
    # 300 channels, 450 items over the CTAs: several pieces per CTA, items cut between CTAs
    rng = np.random.default_rng(6)
    T, F, N = 640, 300, 256
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    want = oracle.correlate(blk)
    assert np.array_equal(correlate(blk), want)
    assert np.array_equal(correlate(blk, host=True), want)


@pytest.mark.parametrize("N", [64, 192, 256])
def test_fused_many_items_per_cta(N):
    # 1001 channels: N > 128 gives 1502 items (about ten per CTA), N <= 128 501;
    # pushed in two pieces, so the second launch adds into the first
    rng = np.random.default_rng(N)
    T, F = 96, 1001
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    want = oracle.correlate(blk)
    assert np.array_equal(correlate(blk), want)
    assert np.array_equal(correlate(blk, pieces=[33]), want)


@pytest.mark.parametrize("N", [64, 192])
def test_fused_items_split_over_many_ctas(N):
    # a few channels over a whole 32,768-sample launch: each item's stages are
    # split over many CTAs, whose partial blocks the item's first CTA adds up;
    # stored, then added by a second push
    rng = np.random.default_rng(N + 1)
    T, F = 32768, 5
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    want = oracle.correlate(blk)
    assert np.array_equal(correlate(blk), want)
    assert np.array_equal(correlate(blk, pieces=[20000]), want)


# How a launch's items (each of ceil(T / 128) stages) are cut over the CTAs:
# shared by several CTAs (as many as there are SMs for, stages uneven between
# them, at most 32, at least two stages each), whole, cut evenly, or -- 60 items
# of 256 stages -- even because two CTAs an item would leave SMs idle.
@pytest.mark.parametrize("T,F,N", [(2100, 1, 64), (2177, 1, 16), (4096, 8, 256), (4097, 12, 208), (5000, 25, 160),
                                   (9000, 1, 256), (2000, 256, 112), (3969, 52, 256), (5000, 110, 256),
                                   (32700, 40, 256)])
def test_small_items_shared_whole_or_cut(T, F, N):
    rng = np.random.default_rng(T + F + N)
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    if F > 16 and T > 1000:  # the oracle on the last channels and the first
        keep = [0, 1, F - 2, F - 1]
    else:
        keep = list(range(F))
    want = oracle.correlate(np.ascontiguousarray(blk[:, keep]))
    assert np.array_equal(correlate(blk)[keep], want)
    # the second push adds: its own cut of the rest
    assert np.array_equal(correlate(blk, pieces=[T // 3])[keep], want)


# Launches whose kernel is chosen by their shape: a few stages or rounds (one pass, N <=
# 256 too, where sharing or cutting the items would take longer).
@pytest.mark.parametrize("T,F,N", [(130, 40, 512), (1500, 26, 512), (700, 3, 1024), (200, 300, 128), (256, 90, 256),
                                   (8, 2, 16), (511, 7, 208), (1000, 3, 144), (2048, 8, 256), (4000, 150, 128),
                                   (4096, 48, 256)])
def test_kernel_by_launch_shape(T, F, N):
    rng = np.random.default_rng(T * 3 + F + N)
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    keep = sorted({0, 1, F // 2, F - 2, F - 1})
    want = oracle.correlate(np.ascontiguousarray(blk[:, keep]))
    assert np.array_equal(correlate(blk)[keep], want)
    # the later pushes add, the last of them a few samples
    assert np.array_equal(correlate(blk, pieces=[T // 2, T // 2 - 3])[keep], want)


# Above 256 inputs a last round of the pair kernel with few items goes to the one pass,
# as a second launch: 2048 x 7 channels (252 items on 76 clusters, six channels fill
# three rounds), 1280 x 17 (255, 15 channels).  A call and a push store, a second push
# adds; the channels on both sides of the cut against the oracle.
@pytest.mark.parametrize("N,F", [(2048, 7), (1280, 17)])
def test_last_round_of_the_pair_kernel_by_the_one_pass(N, F):
    T, sms = 6000, torch.cuda.get_device_properties(0).multi_processor_count
    kernel, cut = xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR, N, F, T, False, sms)
    assert kernel == xe.XENG_KERNEL_PAIR and 0 < cut < F
    assert xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR, N, F, T, True, sms) == (kernel, cut)
    g = torch.Generator(device="cuda")
    g.manual_seed(N)
    block = torch.randint(0, 256, (T, F, N), dtype=torch.uint8, device="cuda", generator=g)
    eng = xe.XEngine(N, F, 2 * T)
    out = torch.full((F, N * (N + 1) // 2, 2), 77, dtype=torch.int32, device="cuda")
    eng.correlate(block, out)
    st = eng.stats(reset=True)
    assert st["correlate_launches"] == 1 and st["launches"] == 2
    keep = sorted({0, cut - 1, cut, F - 1})
    want = torch.from_numpy(oracle.correlate(np.ascontiguousarray(block[:, keep].cpu().numpy())))
    assert torch.equal(out[keep].cpu().to(torch.int64), want)
    for _ in range(2):
        eng.push(block)
    assert eng.stats(reset=True)["launches"] == 4
    added = torch.full_like(out, 77)
    assert eng.dump(added) == 2 * T
    assert torch.equal(added, 2 * out)
    eng.close()


# Samples rearranged first (pack.cu): rows off 16 bytes, fewer inputs than a chunk,
# a block off a 16-byte boundary, several rounds (more than 32,768 samples)
@pytest.mark.parametrize("T,F,N,skip", [(1, 1, 1, 0), (300, 5, 7, 0), (1031, 3, 203, 0), (700, 26, 509, 0),
                                        (500, 2, 1025, 0), (33000, 1, 33, 0), (600, 3, 272, 1), (600, 3, 128, 8)])
def test_unaligned_rows_and_blocks(T, F, N, skip):
    rng = np.random.default_rng(T + 7 * F + N)
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    want = oracle.correlate(blk)
    flat = torch.zeros(blk.size + 64, dtype=torch.uint8, device="cuda")
    src = flat[skip:skip + blk.size].view(T, F, N)
    src.copy_(torch.from_numpy(blk))
    eng = xe.XEngine(N, F, T)
    out = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    eng.correlate(src, out, T)
    assert np.array_equal(out.cpu().numpy().astype(np.int64), want)
    eng.push(src, T // 3)
    eng.push(src[T // 3:], T - T // 3)
    eng.dump(out)
    assert np.array_equal(out.cpu().numpy().astype(np.int64), want)
    eng.close()
    assert np.array_equal(correlate(blk, host=True), want)


def test_fused_graph_replays_stay_exact():
    # one captured call replayed: the flags that publish split items' partial
    # blocks carry a count the device advances after every launch, so no replay
    # takes another's flags for its own
    rng = np.random.default_rng(77)
    T, F, N = 640, 300, 256  # 450 items over the CTAs, several cut between CTAs
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    want = oracle.correlate(blk)
    d = torch.from_numpy(blk).cuda()
    eng = xe.XEngine(N, F, T)
    out = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    eng.correlate(d, out, T)  # the kernel's scratch is allocated here, outside the capture
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        eng.correlate(d, out, T, s)
    for _ in range(4):
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy().astype(np.int64), want)
    eng.close()


# ---- the single passes over block pairs, for any N that is a multiple of 16: single
# ---- CTAs over pairs of 128-input blocks (onepass) and 2-CTA clusters over pairs of
# ---- 256-input blocks (pair).  Above 256 inputs the library picks one by N; the
# ---- environment variable XENG_FUSED_KERNEL forces either, so both run every case
# ---- (diagonal pairs, ragged last blocks, both CTAs' halves, inputs below 256)

FUSED = xe.XENG_ENGINE_TENSOR_FUSED


@pytest.fixture(params=["onepass", "pair"])
def fused_kernel(request, monkeypatch):
    monkeypatch.setenv("XENG_FUSED_KERNEL", request.param)
    return request.param


@pytest.mark.parametrize("T,F,N", [(1, 1, 16), (129, 3, 32), (513, 2, 240), (1, 1, 272), (127, 2, 288),
                                   (129, 2, 512), (1000, 3, 528), (300, 2, 784), (257, 1, 1024), (200, 2, 2048),
                                   (130, 1, 4096)])
def test_fused_raw_shapes(T, F, N, fused_kernel):
    rng = np.random.default_rng(T * 37 + F * 5 + N)
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    assert np.array_equal(correlate(blk, engine=FUSED), oracle.correlate(blk)), (T, F, N, fused_kernel)


@pytest.mark.parametrize("N,T", [(400, 70000), (1040, 36000)])
def test_fused_raw_several_launches_pieces_and_host_buffers(N, T, fused_kernel):
    # more than 32,768 samples = several launches adding into int32; pushes in pieces;
    # host buffers through the channel-group pipeline
    rng = np.random.default_rng(15 + N)
    F = 2
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    want = oracle.correlate(blk)
    assert np.array_equal(correlate(blk, engine=FUSED), want)
    assert np.array_equal(correlate(blk, pieces=[100, 32768, 3], engine=FUSED), want)
    T2, F2 = 3000, 40 if N < 512 else 6
    blk2 = rng.integers(0, 256, size=(T2, F2, N), dtype=np.uint8)
    assert np.array_equal(correlate(blk2, host=True, engine=FUSED), oracle.correlate(blk2))


def test_fused_raw_many_channels_per_cluster_and_plane_engine_agree(fused_kernel):
    # 90 channels x 3 block pairs over the 76 clusters (or 10 over the CTAs); the
    # two-pass engine gives the same bits
    rng = np.random.default_rng(16)
    T, F, N = 384, 90, 512
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    got = correlate(blk, engine=FUSED)
    d = torch.from_numpy(blk).cuda()
    eng = xe.XEngine(N, F, T, xe.XENG_ENGINE_TENSOR_PLANES)
    out = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    eng.correlate(d, out, T)
    torch.cuda.synchronize()
    eng.close()
    assert np.array_equal(got, out.cpu().numpy().astype(np.int64))
    assert np.array_equal(got[[0, 45, 89]], oracle.correlate(blk, f0=0, nf=F)[[0, 45, 89]])


@pytest.mark.parametrize("N", [384, 704, 1024])
def test_single_pass_many_items_per_cta_and_engines_agree(N, fused_kernel):
    # 300 channels of 6, 21 or 36 pairs of 128-input blocks (3, 6 or 10 of 256-input
    # blocks): several items per CTA or cluster, both accumulators and both sums
    # parities; the default engine (forced to the same kernel) and the planes engine
    # agree, and sampled channels match the oracle; stored, then added by a second push
    rng = np.random.default_rng(N)
    T, F = 160, 300
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    got = correlate(blk)
    assert np.array_equal(correlate(blk, pieces=[70]), got)
    d = torch.from_numpy(blk).cuda()
    eng = xe.XEngine(N, F, T, xe.XENG_ENGINE_TENSOR_PLANES)
    out = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    eng.correlate(d, out, T)
    torch.cuda.synchronize()
    eng.close()
    assert np.array_equal(got, out.cpu().numpy().astype(np.int64))
    pick = [0, 151, 299]
    assert np.array_equal(got[pick], oracle.correlate(np.ascontiguousarray(blk[:, pick])))


def test_fused_raw_int32_beyond_f32_range(fused_kernel):
    # every sample -8-8i over 70,000 samples (three launches): Re = 8,960,000 > 2^23
    T, F, N = 70000, 1, 272
    out = correlate(np.zeros((T, F, N), np.uint8), engine=FUSED)
    assert (out[..., 0] == 128 * T).all() and (out[..., 1] == 0).all()


@pytest.mark.parametrize("N,force", [(272, None), (512, None), (512, "pair")])
def test_single_pass_host_pipeline_channel_groups(N, force, monkeypatch):
    # host in, host out through the channel-group pipeline (at least two groups of
    # about 400 KB rows, each correlated and downloaded in four channel sub-ranges)
    # with the single-pass kernels (the one pass over 128-input block pairs, which such
    # short launches take, and 256-input block pairs): the same bits as device buffers,
    # sampled channels as the oracle
    if force:
        monkeypatch.setenv("XENG_FUSED_KERNEL", force)
    rng = np.random.default_rng(N + 5)
    T, F = 160, 2 * 409600 // N + 3
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    pinned = torch.from_numpy(blk).pin_memory()
    hout = torch.zeros((F, N * (N + 1) // 2, 2), dtype=torch.int32).pin_memory()
    eng = xe.XEngine(N, F, T)
    for _ in range(2):  # the second call reuses the staging buffers
        eng.correlate(pinned, hout)
    dout = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    eng.correlate(torch.from_numpy(blk).cuda(), dout)
    torch.cuda.synchronize()
    eng.close()
    got = hout.numpy().astype(np.int64)
    assert np.array_equal(got, dout.cpu().numpy().astype(np.int64))
    pick = [0, F // 2, F - 1]
    assert np.array_equal(got[pick], oracle.correlate(np.ascontiguousarray(blk[:, pick])))


@pytest.mark.parametrize("N", [3584, 3600])
def test_default_engine_at_its_single_pass_bound(N):
    # the default engine takes the single pass up to 3584 inputs (here, two stages, the
    # one pass) and decodes to planes above: both exact against the oracle on a
    # few sampled channels, and the same bits as the single-pass engine at 3600
    assert xe.xeng_kernel_choice(xe.XENG_ENGINE_TENSOR, N, 2, 160)[0] == (
        xe.XENG_KERNEL_ONEPASS if N == 3584 else xe.XENG_KERNEL_PLANES)
    rng = np.random.default_rng(N + 7)
    T, F = 160, 2
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    got = correlate(blk)
    assert np.array_equal(got, oracle.correlate(blk))
    if N > 3584:
        assert np.array_equal(correlate(blk, engine=FUSED), got)


# A short first launch takes the one pass, but has the N <= 256 kernel's scratch made:
# a long one may be captured next
def test_long_launch_captured_after_a_short_one():
    T, F, N = 6000, 2, 256
    blk = np.random.default_rng(3).integers(0, 256, size=(T, F, N), dtype=np.uint8)
    block = torch.from_numpy(blk).cuda()
    out = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    eng = xe.XEngine(N, F, T)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    eng.correlate(block, out, 128, s.cuda_stream)
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        eng.correlate(block, out, T, s.cuda_stream)
    for _ in range(2):
        g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().astype(np.int64), oracle.correlate(blk))
    eng.close()


# Long calls of few channels, above 256 inputs, decode to planes where samples would be
# rearranged (from 8192 samples, up to 1536 channels x inputs in 128-input blocks): both
# sides of both lines, one call, pushes of both kinds, and one captured after a short call
@pytest.mark.parametrize("N,F", [(283, 4), (283, 5), (1025, 1), (257, 1)])
def test_long_unaligned_calls_of_few_channels(N, F):
    T = 8192 + 8191
    blk = np.random.default_rng(N + F).integers(0, 256, size=(T, F, N), dtype=np.uint8)
    want = oracle.correlate(blk)
    assert np.array_equal(correlate(blk[:8191]), oracle.correlate(blk[:8191]))
    assert np.array_equal(correlate(blk), want)
    for pieces in ([8191], [8192], [100, 9000]):
        assert np.array_equal(correlate(blk, pieces=pieces), want)
    block = torch.from_numpy(blk).cuda()
    out = torch.empty((F, N * (N + 1) // 2, 2), dtype=torch.int32, device="cuda")
    eng = xe.XEngine(N, F, T)
    s = torch.cuda.Stream()
    torch.cuda.synchronize()
    eng.correlate(block, out, 128, s.cuda_stream)
    s.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        eng.correlate(block, out, T, s.cuda_stream)
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy().astype(np.int64), want)
    eng.close()


# The single-pass engine with rows that TMA cannot address: rearranged up to 3584 inputs,
# decoded to planes above, gates and delays too
@pytest.mark.parametrize("N", [3583, 3601, 4001])
def test_single_pass_engine_unaligned(N):
    blk = np.random.default_rng(N).integers(0, 256, size=(140, 1, N), dtype=np.uint8)
    want = oracle.correlate(blk)
    assert np.array_equal(correlate(blk, engine=FUSED), want)
    assert np.array_equal(correlate(blk, pieces=[70], engine=FUSED), want)
