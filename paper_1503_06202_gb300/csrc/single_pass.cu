// single_pass.cu -- which of the single-pass kernels (the nibble split of paper
// Sec. II-A fused into the correlation of Sec. IV-C-1) takes a block of N
// inputs, and their common launch, for handles and batches alike.
#include <cstdlib>
#include <cstring>

#include "tc_ptx.cuh"
#include "xeng_internal.h"

// Up to 256 inputs: single CTAs over the upper-triangle 128-input blocks
// (correlate_small.cu).  0 disables it (such blocks decode to planes).
#ifndef XENG_FUSED_SMALL
#define XENG_FUSED_SMALL 1
#endif
// Above 256 inputs the single pass runs either the 2-CTA pair kernel over
// 256-input block pairs (correlate_pair.cu) or single CTAs over 128-input block
// pairs (correlate_onepass.cu), whichever costs less by the measured time of
// one block pair (GB300, 1024 channels x 8192 samples: 1.09-1.20 ms per 256 x
// 256 pair, 0.35-0.44 ms per 128 x 128 pair, in units of 10 us).  The pair
// kernel does a quarter of the MMAs per block in a quarter of the items, but
// pads N to 256: it wins unless ceil(N / 128) is odd, and the one pass's cost
// per pair grows above about 1900 inputs (one pass / pair, ms: N = 384 2.35 /
// 3.22; 512 3.66 / 3.26; 640 5.26 / 6.75; 768 7.50 / 6.75; 896 9.79 / 11.05;
// 1024 13.06 / 11.09; 1152 15.98 / 16.96; 1408 23.15 / 23.90; 1664 32.13 /
// 33.70; 1920 51.88 / 42.12; 2176 67.87 / 53.46: the ratio of the two costs
// must lie between 3.25 and 3.33).  A cost of 0 forces that kernel, for every
// launch shape too (launch_rule.h).
#ifndef XENG_PAIR_COST
#define XENG_PAIR_COST 118
#endif
#ifndef XENG_ONEPASS_COST
#define XENG_ONEPASS_COST 36
#endif
// Above this many inputs the default engine and batches decode to planes first
// (two passes) instead of the single pass: the decode pass grows with N, the
// correlation with N^2, and the plane GEMM does a block pair about 15% faster
// than the pair kernel's converters feed it (GB300, 8192 samples, ms single /
// two passes: N = 2048 x 1024 channels 43.5 / 45.1, N = 3072 x 512 46.8 / 47.7,
// N = 4096 x 256 40.8 / 40.0; a fit of both puts the crossover near 3600).
#ifndef XENG_FUSED_MAX_N
#define XENG_FUSED_MAX_N 3584
#endif
#include "launch_rule.h"

namespace xeng {

cudaError_t status_alloc(int **d_err, int **h_err)
{
    *d_err = *h_err = nullptr;
    StatusBlock sb = {0, 0, nullptr};
    cudaError_t e = cudaMallocHost(h_err, sizeof(int));
    if (e == cudaSuccess) {
        **h_err = 0;
        void *m = nullptr;
        e = cudaHostGetDevicePointer(&m, *h_err, 0);
        sb.mirror = static_cast<int *>(m);
    }
    if (e == cudaSuccess) e = cudaMalloc(d_err, sizeof sb);
    if (e == cudaSuccess) e = cudaMemcpy(*d_err, &sb, sizeof sb, cudaMemcpyHostToDevice);
    if (e != cudaSuccess) {
        cudaGetLastError();
        status_free(*d_err, *h_err);
        *d_err = *h_err = nullptr;
    }
    return e;
}

void status_free(int *d_err, int *h_err)
{
    cudaFree(d_err);
    if (h_err) cudaFreeHost(h_err);
}

int single_pass_force_from_env()
{
    const char *env = getenv("XENG_FUSED_KERNEL");
    if (!env) return 0;
    if (!strcmp(env, "pair")) return kSinglePair;
    if (!strcmp(env, "onepass")) return kSingleOnepass;
    if (!strcmp(env, "none")) return kSingleNone;
    return 0;
}

int single_pass_kernel(const uint8_t *block, int32_t N, int force, bool bounded, int32_t pitch)
{
    if (force == kSingleNone || (bounded && N > XENG_FUSED_MAX_N)) return 0;
    const int k = force ? force : N <= 256 ? kSingleSmall : use_pair_kernel(N) ? kSinglePair : kSingleOnepass;
    switch (k) {
    case kSingleSmall: return XENG_FUSED_SMALL && small_ok(block, N, pitch) ? k : 0;
    case kSinglePair: return pair_ok(block, N, pitch) ? k : 0;
    default: return onepass_ok(block, N, pitch) ? k : 0;
    }
}

cudaError_t small_scratch_alloc(SmallScratch *sc, int num_sms, cudaStream_t s)
{
    if (sc->ws) return cudaSuccess;
    cudaError_t e = cudaMalloc(&sc->ws, small_ws_bytes(num_sms));
    if (e == cudaSuccess) e = cudaMalloc(&sc->flags, small_flags_bytes(num_sms));
    if (e == cudaSuccess) e = cudaMemsetAsync(sc->flags, 0, small_flags_bytes(num_sms), s);
    if (e != cudaSuccess) {
        cudaGetLastError();
        small_scratch_free(sc);
    }
    return e;
}

void small_scratch_free(SmallScratch *sc)
{
    cudaFree(sc->ws);
    cudaFree(sc->flags);
    sc->ws = nullptr;
    sc->flags = nullptr;
}

cudaError_t launch_single_pass(int kernel, const uint8_t *block, int64_t T_block, int64_t t0, int64_t nt, int32_t F,
                               int32_t N, int32_t f0, int32_t nf, int32_t *acc, int accumulate, SmallScratch *sc,
                               int *err, int num_sms, cudaStream_t s, const CUtensorMap *maps, int32_t spb,
                               int32_t pitch, const SubBlocks *sub, int max_ctas)
{
    if (kernel == kSingleSmall) {
        cudaError_t e = small_scratch_alloc(sc, num_sms, s);
        if (e != cudaSuccess) return e;
        return launch_correlate_small(block, T_block, t0, nt, F, N, f0, nf, acc, accumulate, sc->ws, sc->flags, err,
                                      num_sms, s, maps, spb, pitch, sub, max_ctas);
    }
    if (kernel == kSinglePair)
        return launch_correlate_pair(block, T_block, t0, nt, F, N, f0, nf, acc, accumulate, err, num_sms, s, maps,
                                     spb, pitch, sub);
    if (kernel == kSingleOnepass)
        return launch_correlate_onepass(block, T_block, t0, nt, F, N, f0, nf, acc, accumulate, err, num_sms, s, maps,
                                        spb, pitch, sub);
    return cudaErrorInvalidValue;
}

cudaError_t launch_single_pass_shaped(int kernel, const uint8_t *block, int64_t T_block, int64_t t0, int64_t nt,
                                      int32_t F, int32_t N, int32_t f0, int32_t nf, int32_t *acc, int accumulate,
                                      SmallScratch *sc, int *err, int num_sms, cudaStream_t s, int32_t pitch,
                                      const SubBlocks *sub, int64_t *launches)
{
    if (kernel == kSingleSmall) {
        // with the first launch, whichever kernel that takes: a later one may be captured
        const cudaError_t e0 = small_scratch_alloc(sc, num_sms, s);
        if (e0 != cudaSuccess) return e0;
    }
    const int k = single_pass_by_shape(kernel, N, nf, nt, accumulate, num_sms);
    const int32_t cut = single_pass_cut(k, N, nf, nt, accumulate, num_sms);
    const int32_t first = cut ? cut : nf;
    cudaError_t e = launch_single_pass(k, block, T_block, t0, nt, F, N, f0, first, acc, accumulate, sc, err, num_sms, s,
                                       nullptr, 0, pitch, sub);
    if (e != cudaSuccess || !cut) return e;
    if (launches) ++*launches;
    SubBlocks rest;
    if (sub) {
        rest = *sub;
        rest.f0 += cut;
    }
    return launch_single_pass(kSingleOnepass, block, T_block, t0, nt, F, N, f0 + cut, nf - cut,
                              acc + (int64_t)cut * N * (N + 1), accumulate, sc, err, num_sms, s, nullptr, 0, pitch,
                              sub ? &rest : nullptr);
}

cudaError_t encode_raw_map(CUtensorMap *map, const uint8_t *block, int64_t T_block, int32_t F, int32_t N,
                           int32_t pitch, int stage, bool wide)
{
    EncodeTiledFn enc = encode_tiled();
    if (!enc) return cudaErrorNotSupported;
    // a 128-byte swizzle gives the MN-major operand layout; inputs past N and
    // samples past the block read as zero bytes, nibbles 0 that add nothing (the
    // converters zero the samples past the launch; rows and columns past N are never
    // written)
    const cuuint64_t p = (cuuint64_t)(pitch ? pitch : N);
    cuuint64_t dims[3] = {(cuuint64_t)N, (cuuint64_t)F, (cuuint64_t)T_block};
    cuuint64_t strides[2] = {p, p * F};
    cuuint32_t box[3] = {128, 1, (cuuint32_t)stage}, estr[3] = {1, 1, 1};
    if (enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, (void *)block, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            wide ? CU_TENSOR_MAP_L2_PROMOTION_L2_256B : CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    return cudaSuccess;
}

int single_pass_stage(int kernel)
{
    if (kernel == kSingleSmall) return small_stage_samples();
    if (kernel == kSinglePair) return pair_stage_samples();
    if (kernel == kSingleOnepass) return onepass_stage_samples();
    return 0;
}

}  // namespace xeng
