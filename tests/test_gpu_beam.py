"""Beamforming (Sec. IV-C-3) through the C ABI, bit-exact against the oracle:
ragged sample counts and input counts (vs the 128 tiles), every padded beam
width, the full int8 weight range including -128, the largest magnitudes,
host and device weights, per-channel weights, sampled outputs of the full
Pathfinder-size workload, and the argument checks."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
import paper_1503_06202_gb300 as xe  # noqa: E402


def run_beams(blk, w_re, w_im, host_weights=False):
    T, F, N = blk.shape
    B = w_re.shape[1]
    bf = xe.XBeam(N, F, B)
    if host_weights:
        bf.set_weights(np.ascontiguousarray(w_re, np.int8), np.ascontiguousarray(w_im, np.int8))
    else:
        bf.set_weights(torch.from_numpy(np.ascontiguousarray(w_re, np.int8)).cuda(),
                       torch.from_numpy(np.ascontiguousarray(w_im, np.int8)).cuda())
    out = torch.empty((T, F, B, 2), dtype=torch.int32, device="cuda")
    bf.run(torch.from_numpy(blk).cuda(), out)
    torch.cuda.synchronize()
    bf.close()
    return out.cpu().numpy().astype(np.int64)


def random_case(seed, T, F, N, B):
    rng = np.random.default_rng(seed)
    blk = rng.integers(0, 256, size=(T, F, N), dtype=np.uint8)
    w_re = rng.integers(-128, 128, size=(F, B, N), dtype=np.int64)
    w_im = rng.integers(-128, 128, size=(F, B, N), dtype=np.int64)
    return blk, w_re, w_im


@pytest.mark.parametrize("B", [1, 4, 5, 8, 13, 16, 17, 32, 33, 64])
def test_beams_every_width_ragged(B):
    blk, w_re, w_im = random_case(100 + B, 300, 3, 208, B)   # 300 = 2 tiles + 44; 208 = 128 + 80
    assert np.array_equal(run_beams(blk, w_re, w_im), oracle.beamform(blk, w_re, w_im))


def test_beams_small_inputs_host_weights():
    blk, w_re, w_im = random_case(7, 129, 2, 16, 3)
    assert np.array_equal(run_beams(blk, w_re, w_im, host_weights=True), oracle.beamform(blk, w_re, w_im))


def test_beams_extreme_magnitudes_max_inputs():
    # every byte 0x00 (x = -8 - 8i) with weights -128 - 128i at N = 4096:
    # y = N * 2048i, the largest imaginary part; and (-128 + 127i) for a mixed sign
    T, F, N = 130, 1, xe.XENG_MAX_INPUTS
    blk = np.zeros((T, F, N), np.uint8)
    w_re = np.full((F, 2, N), -128, np.int64)
    w_im = np.full((F, 2, N), -128, np.int64)
    w_im[:, 1] = 127
    got = run_beams(blk, w_re, w_im)
    assert np.array_equal(got, oracle.beamform(blk, w_re, w_im))
    assert (got[:, :, 0, 1] == N * 2048).all()


def test_beams_weights_change_and_channels_independent():
    blk, w_re, w_im = random_case(8, 256, 4, 128, 4)
    bf = xe.XBeam(128, 4, 4)
    out = torch.empty((256, 4, 4, 2), dtype=torch.int32, device="cuda")
    dblk = torch.from_numpy(blk).cuda()
    for k in range(2):
        # second set: i * w (clipped to int8: -(-128) does not fit)
        wr, wi = (w_re, w_im) if k == 0 else (np.clip(-w_im, -128, 127), w_re)
        bf.set_weights(np.ascontiguousarray(wr, np.int8), np.ascontiguousarray(wi, np.int8))
        bf.run(dblk, out)
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy().astype(np.int64), oracle.beamform(blk, wr, wi)), k
    # zero weights for channel 2 only: its beams vanish, the others are unchanged
    w2 = w_re.copy()
    w2[2] = 0
    wi2 = w_im.copy()
    wi2[2] = 0
    bf.set_weights(np.ascontiguousarray(w2, np.int8), np.ascontiguousarray(wi2, np.int8))
    bf.run(dblk, out)
    got = out.cpu().numpy().astype(np.int64)
    assert (got[:, 2] == 0).all()
    assert np.array_equal(got, oracle.beamform(blk, w2, wi2))
    bf.close()


def test_beams_full_pathfinder_sampled():
    # the Pathfinder-size block (256 inputs, 1024 channels, 32768 samples) with
    # 16 beams; the oracle checks sampled (sample, channel) rows of the output
    import synth
    rec = synth.PATHFINDER_FULL
    T, F, N, B = rec.T, rec.F, rec.N, 16
    blk = rec.device()
    rng = np.random.default_rng(9)
    w_re = rng.integers(-128, 128, size=(F, B, N), dtype=np.int64)
    w_im = rng.integers(-128, 128, size=(F, B, N), dtype=np.int64)
    bf = xe.XBeam(N, F, B)
    bf.set_weights(np.ascontiguousarray(w_re, np.int8), np.ascontiguousarray(w_im, np.int8))
    out = torch.empty((T, F, B, 2), dtype=torch.int32, device="cuda")
    bf.run(blk, out)
    torch.cuda.synchronize()
    ts = np.unique(np.concatenate([rng.integers(0, T, 40), [0, T - 1]]))
    fs = np.unique(np.concatenate([rng.integers(0, F, 12), [0, F - 1]]))
    sub = blk[torch.from_numpy(ts).cuda()][:, torch.from_numpy(fs).cuda()].cpu().numpy()
    want = oracle.beamform(np.ascontiguousarray(sub), w_re[fs], w_im[fs])
    got = out[torch.from_numpy(ts).cuda()][:, torch.from_numpy(fs).cuda()].cpu().numpy().astype(np.int64)
    assert np.array_equal(got, want)
    bf.close()


def test_beams_argument_checks():
    bf = xe.XBeam(64, 2, 3)
    blk = torch.zeros((100, 2, 64), dtype=torch.uint8, device="cuda")
    out = torch.empty((100, 2, 3, 2), dtype=torch.int32, device="cuda")
    assert xe.xbeam_run(bf.h, blk, 0, out) == xe.XENG_OK              # nothing to do
    assert xe.xbeam_run(bf.h, blk, -1, out) == xe.XENG_ERR_ARG
    assert xe.xbeam_run(bf.h, blk.cpu(), 100, out) == xe.XENG_ERR_ARG  # host block
    flat = torch.empty(100 * 2 * 3 * 2 + 1, dtype=torch.int32, device="cuda")
    assert xe.xbeam_run(bf.h, blk, 100, flat[1:]) == xe.XENG_ERR_ARG   # out not 8-byte aligned
    # weights all zero before the first xbeam_set_weights: every beam is 0
    bf.run(blk, out)
    torch.cuda.synchronize()
    assert (out == 0).all()
    bf.close()


def test_beams_repeat_the_same_bits():
    # short items of 32 beams, where the raw ring runs fastest: every pass over the
    # same block gives the bits of the oracle (channel by channel on sampled rows)
    T, F, N, B = 16384, 128, 256, 32
    g = torch.Generator(device="cuda")
    g.manual_seed(3)
    blk = torch.randint(0, 256, (T, F, N), dtype=torch.uint8, device="cuda", generator=g)
    rng = np.random.default_rng(4)
    w_re = rng.integers(-128, 128, size=(F, B, N), dtype=np.int64)
    w_im = rng.integers(-128, 128, size=(F, B, N), dtype=np.int64)
    bf = xe.XBeam(N, F, B)
    bf.set_weights(np.ascontiguousarray(w_re, np.int8), np.ascontiguousarray(w_im, np.int8))
    first, out = (torch.empty((T, F, B, 2), dtype=torch.int32, device="cuda") for _ in range(2))
    bf.run(blk, first)
    for _ in range(60):
        bf.run(blk, out)
        assert torch.equal(out, first)
    ts = np.unique(rng.integers(0, T, 60))
    want = oracle.beamform(np.ascontiguousarray(blk[torch.from_numpy(ts).cuda()].cpu().numpy()), w_re, w_im)
    assert np.array_equal(first[torch.from_numpy(ts).cuda()].cpu().numpy().astype(np.int64), want)
    bf.close()


def beams_64bit(blk, w_re, w_im):
    """The beams of a device block as 64-bit products give them, int32 [T][F][B][2]."""
    T, F, N = blk.shape
    out = torch.empty((T, F, w_re.shape[1], 2), dtype=torch.int32, device="cuda")
    for f in range(F):
        re, im = (blk[:, f] >> 4).double() - 8, (blk[:, f] & 15).double() - 8
        wr, wi = w_re[f].double().T, w_im[f].double().T
        out[:, f, :, 0] = (re @ wr - im @ wi).to(torch.int32)  # integers below 2^53: exact
        out[:, f, :, 1] = (re @ wi + im @ wr).to(torch.int32)
    return out


def test_beams_every_value_of_passes_among_others():
    # passes over two handles' blocks with nothing waiting in between, as a loop runs
    # them, copies on another stream taking memory time from some: every value of every
    # beam is what 64 bits give
    T, F, N, B = 16384, 128, 256, 32
    g = torch.Generator(device="cuda")
    g.manual_seed(5)
    cases = []
    for _ in range(2):
        blk = torch.randint(0, 256, (T, F, N), dtype=torch.uint8, device="cuda", generator=g)
        w = torch.randint(-128, 128, (2, F, B, N), dtype=torch.int8, device="cuda", generator=g)
        bf = xe.XBeam(N, F, B)
        bf.set_weights(w[0], w[1])
        cases.append((bf, blk, torch.empty((T, F, B, 2), dtype=torch.int32, device="cuda"), beams_64bit(blk, *w)))
    side, a = torch.cuda.Stream(), torch.zeros(1 << 28, dtype=torch.uint8, device="cuda")
    b = torch.empty_like(a)
    torch.cuda.synchronize()
    for k in range(200):
        with torch.cuda.stream(side):
            for _ in range(k % 4):
                b.copy_(a)
        for c in (0, 1, 0):
            bf, blk, out, _ = cases[c]
            bf.run(blk, out)
        for _, _, out, want in cases:
            assert torch.equal(out, want), k
    torch.cuda.synchronize()
    for bf, *_ in cases:
        bf.close()


# Beams staged and stored by TMA, staged and stored by threads (odd B, or out on an
# 8-byte but not a 16-byte boundary) or stored straight from registers, four, two or one
# at a time: both sides of every line of the choice, ragged samples
@pytest.mark.parametrize("N,B,off", [(16, 1, 0), (16, 2, 8), (16, 3, 0), (144, 3, 8), (144, 4, 16), (16, 4, 0),
                                     (16, 8, 8), (256, 16, 8), (256, 32, 8), (256, 64, 8), (512, 28, 0), (640, 28, 0),
                                     (640, 32, 0), (656, 32, 0), (768, 18, 0), (784, 18, 0), (768, 32, 16), (2304, 30, 0),
                                     (1408, 17, 0), (1536, 17, 0), (3328, 32, 8), (3328, 31, 0), (2048, 20, 8)])
def test_beams_staged_and_direct_stores(N, B, off):
    T, F = 300, 2
    blk, w_re, w_im = random_case(N + B + off, T, F, N, B)
    flat = torch.full((T * F * B * 2 + 64,), 77, dtype=torch.int32, device="cuda")
    lo, n = 8 + off // 4, T * F * B * 2
    bf = xe.XBeam(N, F, B)
    bf.set_weights(np.ascontiguousarray(w_re, np.int8), np.ascontiguousarray(w_im, np.int8))
    bf.run(torch.from_numpy(blk).cuda(), flat[lo:lo + n].view(T, F, B, 2))
    got = flat.cpu().numpy().astype(np.int64)
    bf.close()
    assert np.array_equal(got[lo:lo + n].reshape(T, F, B, 2), oracle.beamform(blk, w_re, w_im))
    assert (got[:lo] == 77).all() and (got[lo + n:] == 77).all()
