// pack.cu -- raw samples rearranged for the single-pass kernels: rows of whole
// 16-byte chunks, which TMA can address, holding the samples that a launch
// integrates.  One pass serves
//   blocks whose rows TMA cannot address (N not a multiple of 16, a block off a
//   16-byte boundary): a copy at a pitch of 16-byte chunks;
//   gates and flags (paper Sec. IV-C-4, Sec. IV-A): the rows of one gate, in
//   order, a flagged sample replaced by the byte 0x88 (value 0 + 0i) and the
//   usable samples per (channel, input) counted;
//   time shifts (Sec. IV-C-5): inputs read d samples late, from the block or,
//   before it, from the history of the delayed inputs.
// Decoding such blocks to planes instead moves a byte in and two out, and the
// correlation reads those two (three times over, at 256 inputs); here it is a
// byte in, a byte out, and a byte read by the kernel that splits nibbles in
// shared memory.  Bound by HBM: each thread owns one 16-byte chunk of the row
// and walks down the samples, four rows of loads in flight.
#include "xeng_internal.h"

namespace xeng {
namespace {

constexpr int kPackThreads = 256;
constexpr int kPackRows = 4;       // rows loaded before any is stored
constexpr int kPackSpan = 256;     // rows per thread at most (byte-lane counts are widened every 240)

// The 16 bytes at p, any alignment, of which the first n are wanted (the rest
// may come out as anything): only 16-byte words that hold a wanted byte are read.
__device__ __forceinline__ uint4 load16(const uint8_t *p, int n)
{
    const int a = (int)(reinterpret_cast<uintptr_t>(p) & 15);
    const uint4 *q = reinterpret_cast<const uint4 *>(p - a);
    const uint4 lo = __ldg(q);
    if (a == 0) return lo;
    const uint4 hi = a + n > 16 ? __ldg(q + 1) : lo;
    uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    if (a & 8) {
        #pragma unroll
        for (int k = 0; k < 6; k++) w[k] = w[k + 2];
    }
    if (a & 4) {
        #pragma unroll
        for (int k = 0; k < 5; k++) w[k] = w[k + 1];
    }
    const int s = 8 * (a & 3);
    return make_uint4(__funnelshift_r(w[0], w[1], s), __funnelshift_r(w[1], w[2], s),
                      __funnelshift_r(w[2], w[3], s), __funnelshift_r(w[3], w[4], s));
}

// kAligned: every source chunk is 16-byte aligned.  Thread = (row of the block's
// rows, chunk): chunk `col` of the [nf][pitch / 16] chunks of a sample.
template <bool kAligned, bool kValid>
__global__ void __launch_bounds__(kPackThreads)
pack_kernel(const PackArgs a, int cols_per_block, int rows_per_block, int span)
{
    const int cpr = a.pitch / 16;
    const int64_t col = (int64_t)blockIdx.x * cols_per_block + threadIdx.x % cols_per_block;
    const int rsub = threadIdx.x / cols_per_block;
    if (col >= (int64_t)a.nf * cpr || rsub >= rows_per_block) return;
    const int c = (int)(col / cpr), ic = (int)(col % cpr) * 16;
    const int n = min(16, a.N - ic);
    const int64_t row_bytes = (int64_t)a.F * a.N;
    const int64_t off = (int64_t)(a.f0 + c) * a.N + ic;
    const int64_t out_row = (int64_t)a.nf * a.pitch;
    const int64_t first = (int64_t)blockIdx.y * span * rows_per_block + rsub;
    const int64_t last = min(a.nt, ((int64_t)blockIdx.y + 1) * span * rows_per_block);
    uint8_t *out = a.out + col * 16;
    uint32_t acc[4] = {0, 0, 0, 0};                       // usable samples, a byte per input
    uint32_t acc16[8] = {0, 0, 0, 0, 0, 0, 0, 0};         // the same, 16-bit lanes
    int rows = 0, pending = 0;
    auto widen = [&]() {
        #pragma unroll
        for (int k = 0; k < 4; k++) {
            acc16[2 * k] += acc[k] & 0x00FF00FFu;
            acc16[2 * k + 1] += (acc[k] >> 8) & 0x00FF00FFu;
            acc[k] = 0;
        }
        pending = 0;
    };
    for (int64_t t = first; t < last; t += (int64_t)kPackRows * rows_per_block) {
        uint4 x[kPackRows], v[kPackRows];
        #pragma unroll
        for (int k = 0; k < kPackRows; k++) {
            const int64_t tk = t + (int64_t)k * rows_per_block;
            if (tk >= last) break;
            const int64_t src = (a.idx ? (int64_t)__ldg(a.idx + tk) : a.t0 + tk) * row_bytes + off;
            x[k] = kAligned ? __ldg(reinterpret_cast<const uint4 *>(a.block + src)) : load16(a.block + src, n);
            if (kValid)
                v[k] = kAligned ? __ldg(reinterpret_cast<const uint4 *>(a.valid + src)) : load16(a.valid + src, n);
        }
        #pragma unroll
        for (int k = 0; k < kPackRows; k++) {
            const int64_t tk = t + (int64_t)k * rows_per_block;
            if (tk >= last) break;
            uint32_t w[4] = {x[k].x, x[k].y, x[k].z, x[k].w};
            if (kValid) {
                const uint32_t vw[4] = {v[k].x, v[k].y, v[k].z, v[k].w};
                #pragma unroll
                for (int j = 0; j < 4; j++) {
                    const uint32_t z = __vcmpeq4(vw[j], 0u);  // 0xFF in each flagged byte
                    w[j] = (w[j] & ~z) | (0x88888888u & z);
                    acc[j] += ~z & 0x01010101u;
                }
            }
            ++rows;
            *reinterpret_cast<uint4 *>(out + tk * out_row) = make_uint4(w[0], w[1], w[2], w[3]);
        }
        if (kValid && (pending += kPackRows) > 240 - kPackRows) widen();
    }
    if (!a.counts) return;
    if (kValid) widen();
    int32_t *cnt = a.counts + (int64_t)c * a.N + ic;
    #pragma unroll
    for (int m = 0; m < 16; m++) {
        const int usable = kValid ? (int)((acc16[2 * (m >> 2) + (m & 1)] >> (16 * ((m >> 1) & 1))) & 0xFFFFu) : rows;
        if (m < n && usable) atomicAdd(cnt + m, usable);
    }
}

// Shifted rows: chunk j of a row is the block's 16-input chunk a.chunks[j] (or j
// where a.chunks is null).  A chunk without delayed inputs is copied, one whose
// inputs share a delay is copied from that many samples earlier, others byte by
// byte where an input is delayed.
__global__ void __launch_bounds__(kPackThreads)
pack_shifted_kernel(const PackArgs a, const ShiftArgs sa, int cols_per_block, int rows_per_block, int span)
{
    const int cpr = a.pitch / 16;
    const int64_t col = (int64_t)blockIdx.x * cols_per_block + threadIdx.x % cols_per_block;
    const int rsub = threadIdx.x / cols_per_block;
    if (col >= (int64_t)a.nf * cpr || rsub >= rows_per_block) return;
    const int c = (int)(col / cpr), j = (int)(col % cpr);
    const int ic = (a.chunks ? a.chunks[j] : j) * 16;
    if (ic >= a.N) return;  // past the inputs: never read
    const int n = min(16, a.N - ic);
    const int64_t f = a.f0 + c;
    const int64_t out_row = (int64_t)a.nf * a.pitch;
    const int64_t first = (int64_t)blockIdx.y * span * rows_per_block + rsub;
    const int64_t last = min(a.nt, ((int64_t)blockIdx.y + 1) * span * rows_per_block);
    const int cd = n == 16 ? sa.chunk_delay[ic >> 4] : -1;
    uint32_t delayed = 0;  // inputs of a mixed chunk that are
    if (cd < 0)
        for (int m = 0; m < n; m++) delayed |= (sa.delay[ic + m] > 0 ? 1u : 0u) << m;
    uint8_t *out = a.out + col * 16;
    for (int64_t t = first; t < last; t += rows_per_block) {
        const int64_t tt = a.t0 + t;  // sample of the block before the shift
        uint32_t todo = cd > tt ? (1u << n) - 1u : delayed;  // a shared delay reaching before the block: byte by byte
        const int64_t from = cd > 0 && cd <= tt ? tt - cd : tt;
        const uint4 x = load16(a.block + (from * a.F + f) * a.N + ic, n);
        uint32_t w[4] = {x.x, x.y, x.z, x.w};
        while (todo) {
            const int m = __ffs(todo) - 1;
            todo &= todo - 1;
            const int i = ic + m;
            const int64_t src = tt - sa.delay[i];
            const uint32_t byte = src >= 0 ? a.block[(src * a.F + f) * a.N + i]
                                           : sa.hist[((sa.H + src) * a.F + f) * sa.S + sa.slot[i]];
            #pragma unroll
            for (int k = 0; k < 4; k++)
                if (k == m >> 2) w[k] = (w[k] & ~(0xFFu << (8 * (m & 3)))) | (byte << (8 * (m & 3)));
        }
        *reinterpret_cast<uint4 *>(out + t * out_row) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// Blocks of 256 threads over the chunks of a row (all of them, or 256) and, where
// a row is shorter, several rows; each thread walks at most kPackSpan rows, fewer
// where that would leave SMs without a few blocks each.
struct PackGrid {
    dim3 grid;
    int cols, rows, span;
};

PackGrid pack_grid(const PackArgs &a, int num_sms)
{
    PackGrid g;
    const int64_t cols = (int64_t)a.nf * (a.pitch / 16);
    g.cols = (int)(cols < kPackThreads ? cols : kPackThreads);
    g.rows = kPackThreads / g.cols;
    const int64_t bx = (cols + g.cols - 1) / g.cols;
    g.span = kPackSpan;
    while (g.span > 2 * kPackRows && bx * ((a.nt + (int64_t)g.span * g.rows - 1) / ((int64_t)g.span * g.rows)) < 16 * num_sms)
        g.span /= 2;
    g.grid = dim3((unsigned)bx, (unsigned)((a.nt + (int64_t)g.span * g.rows - 1) / ((int64_t)g.span * g.rows)));
    return g;
}

bool pack_args_ok(const PackArgs &a)
{
    return a.block && a.out && a.pitch > 0 && a.pitch % 16 == 0 && a.nt <= kMaxChunkSamples &&
           (reinterpret_cast<uintptr_t>(a.out) & 15) == 0;
}

}  // namespace

cudaError_t launch_pack(const PackArgs &a, int num_sms, cudaStream_t s)
{
    if (a.nf <= 0 || a.nt <= 0) return cudaSuccess;
    if (!pack_args_ok(a) || a.pitch < a.N || a.chunks) return cudaErrorInvalidValue;
    const PackGrid g = pack_grid(a, num_sms);
    const bool aligned = a.N % 16 == 0 && (reinterpret_cast<uintptr_t>(a.block) & 15) == 0 &&
                         (reinterpret_cast<uintptr_t>(a.valid) & 15) == 0;
    auto kernel = a.valid ? (aligned ? pack_kernel<true, true> : pack_kernel<false, true>)
                          : (aligned ? pack_kernel<true, false> : pack_kernel<false, false>);
    kernel<<<g.grid, kPackThreads, 0, s>>>(a, g.cols, g.rows, g.span);
    return cudaGetLastError();
}

cudaError_t launch_pack_shifted(const PackArgs &a, const ShiftArgs &sa, int num_sms, cudaStream_t s)
{
    if (a.nf <= 0 || a.nt <= 0) return cudaSuccess;
    if (!pack_args_ok(a) || (!a.chunks && a.pitch < a.N)) return cudaErrorInvalidValue;
    const PackGrid g = pack_grid(a, num_sms);
    pack_shifted_kernel<<<g.grid, kPackThreads, 0, s>>>(a, sa, g.cols, g.rows, g.span);
    return cudaGetLastError();
}

}  // namespace xeng
