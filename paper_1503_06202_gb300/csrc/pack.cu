// pack.cu -- raw samples rearranged for the single-pass kernels: rows of whole
// 16-byte chunks, which TMA can address, holding the samples that a launch
// integrates.  One pass serves
//   blocks whose rows TMA cannot address (N not a multiple of 16, a block off a
//   16-byte boundary): a copy at a pitch of 16-byte chunks;
//   gates and flags (paper Sec. IV-C-4, Sec. IV-A): the rows of one gate, in
//   order, a flagged sample replaced by the byte 0x88 (value 0 + 0i) and the
//   usable samples per (channel, input) counted;
//   time shifts (Sec. IV-C-5): the delayed inputs read d samples late from their
//   history.
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
constexpr int kPackCountSpan = 32; // rows per thread, where a block adds its counts to memory, unless SMs idle

// Blocks of 256 threads over the `all` columns of a row (all of them, or 256) and,
// where a row is shorter, several rows; each thread walks at most kPackSpan rows, fewer
// where that would leave SMs without a few blocks each.
struct PackGrid {
    int64_t all = 0;
    int cols = 1, rows = 1, span = 1, nx = 0, ny = 0;  // nx * ny blocks a set
};

PackGrid pack_grid(const PackArgs &a, int64_t all, int num_sms)
{
    PackGrid g;
    if (all <= 0) return g;
    g.all = all;
    g.cols = (int)(all < kPackThreads ? all : kPackThreads);
    g.rows = kPackThreads / g.cols;
    const int64_t nx = (all + g.cols - 1) / g.cols, sets = a.sets > 0 ? a.sets : 1;
    auto ny = [&]() { return (a.nt + (int64_t)g.span * g.rows - 1) / ((int64_t)g.span * g.rows); };
    g.span = kPackSpan;
    auto few = [&]() {
        return sets * nx * ny() < (a.valid && a.counts && g.span <= kPackCountSpan ? 2 : 16) * (int64_t)num_sms;
    };
    while (g.span > 2 * kPackRows && few()) g.span /= 2;
    g.nx = (int)nx;
    g.ny = (int)ny();
    return g;
}

// The 16 bytes at p, any alignment, of which the first n are wanted (the rest
// may come out as anything): only 16-byte words that hold a wanted byte are read.
// Without branches, so that several rows' loads are in flight at once.
struct Loaded16 {
    uint4 lo, hi;
    int a;
};
__device__ __forceinline__ Loaded16 load16(const uint8_t *p, int n)
{
    Loaded16 l;
    l.a = (int)(reinterpret_cast<uintptr_t>(p) & 15);
    const uint4 *q = reinterpret_cast<const uint4 *>(p - l.a);
    l.lo = __ldg(q);
    l.hi = __ldg(q + (l.a + n > 16 ? 1 : 0));
    return l;
}

__device__ __forceinline__ uint4 value16(const Loaded16 &l)
{
    uint32_t w[8] = {l.lo.x, l.lo.y, l.lo.z, l.lo.w, l.hi.x, l.hi.y, l.hi.z, l.hi.w};
    #pragma unroll
    for (int k = 0; k < 6; k++) w[k] = l.a & 8 ? w[k + 2] : w[k];
    #pragma unroll
    for (int k = 0; k < 5; k++) w[k] = l.a & 4 ? w[k + 1] : w[k];
    const int s = 8 * (l.a & 3);
    return make_uint4(__funnelshift_r(w[0], w[1], s), __funnelshift_r(w[1], w[2], s),
                      __funnelshift_r(w[2], w[3], s), __funnelshift_r(w[3], w[4], s));
}

// Column `col` of a row's chunks: channel c, 16-byte chunk j of the packed row,
// inputs ic .. of the block.
__device__ __forceinline__ void pack_column(const PackArgs &a, int64_t col, int &c, int &j, int &ic)
{
    const int per = a.chunks ? a.n_chunks : a.pitch / 16;
    c = (int)(col / per);
    const int k = (int)(col - (int64_t)c * per);
    j = a.chunks ? a.chunks[k].x : k;
    ic = 16 * (a.chunks ? a.chunks[k].y : k);
}

// Where a block keeps the usable samples of input m of its column `lc`, so that the
// lanes of a warp, each with its own column, meet two to a bank.
__device__ __forceinline__ int count_slot(int lc, int m) { return lc * 16 + ((m + lc) & 15); }

// kAligned: every source chunk is 16-byte aligned.  Thread = (row of the block's
// rows, chunk of a sample); block (bx, by) of set `set`.  kValid: the usable samples
// per input are added up in `count` (shared memory, 16 a column, zeroed by the caller).
template <bool kAligned, bool kValid>
__device__ __forceinline__ void pack_rows(const PackArgs &a, const PackGrid &g, int bx, int by, int set, int *count)
{
    const int64_t cols = g.all;
    const int cols_per_block = g.cols, rows_per_block = g.rows, span = g.span;
    constexpr int kRows = !kAligned && kValid ? kPackRows / 2 : kPackRows;  // registers
    const int lc = threadIdx.x % cols_per_block;
    const int64_t col = (int64_t)bx * cols_per_block + lc;
    const int rsub = threadIdx.x / cols_per_block;
    if (col >= cols || rsub >= rows_per_block) return;
    int c, j, ic;
    pack_column(a, col, c, j, ic);
    const int n = min(16, a.N - ic);
    const int64_t row_bytes = (int64_t)a.F * a.N;
    const int64_t off = (int64_t)(a.f0 + c) * a.N + ic;
    const int32_t *idx = a.sets ? a.idx + a.set_first[set] : a.idx;
    const int64_t have = a.sets ? a.set_first[set + 1] - a.set_first[set] : a.nt;
    const int64_t out_row = (int64_t)a.nf * a.pitch * max(a.sets, 1);
    const int64_t first = (int64_t)by * span * rows_per_block + rsub;
    const int64_t end = min(a.nt, ((int64_t)by + 1) * span * rows_per_block);
    const int64_t last = min(have, end);
    uint8_t *out = a.out + ((int64_t)set * a.nf + c) * a.pitch + j * 16;
    uint32_t acc[4] = {0, 0, 0, 0};                       // usable samples, a byte per input
    uint32_t acc16[8] = {0, 0, 0, 0, 0, 0, 0, 0};         // the same, 16-bit lanes
    int pending = 0;
    auto widen = [&]() {
        #pragma unroll
        for (int k = 0; k < 4; k++) {
            acc16[2 * k] += acc[k] & 0x00FF00FFu;
            acc16[2 * k + 1] += (acc[k] >> 8) & 0x00FF00FFu;
            acc[k] = 0;
        }
        pending = 0;
    };
    for (int64_t t = first; t < last; t += (int64_t)kRows * rows_per_block) {
        Loaded16 x[kRows], v[kRows];
        #pragma unroll
        for (int k = 0; k < kRows; k++) {
            const int64_t tk = t + (int64_t)k * rows_per_block;
            if (tk >= last) break;
            const int64_t src = (idx ? (int64_t)__ldg(idx + tk) : a.t0 + tk) * row_bytes + off;
            if (kAligned) x[k].lo = __ldg(reinterpret_cast<const uint4 *>(a.block + src));
            else x[k] = load16(a.block + src, n);
            if (kValid && kAligned) v[k].lo = __ldg(reinterpret_cast<const uint4 *>(a.valid + src));
            else if (kValid) v[k] = load16(a.valid + src, n);
        }
        #pragma unroll
        for (int k = 0; k < kRows; k++) {
            const int64_t tk = t + (int64_t)k * rows_per_block;
            if (tk >= last) break;
            const uint4 xv = kAligned ? x[k].lo : value16(x[k]);
            uint32_t w[4] = {xv.x, xv.y, xv.z, xv.w};
            if (kValid) {
                const uint4 vv = kAligned ? v[k].lo : value16(v[k]);
                const uint32_t vw[4] = {vv.x, vv.y, vv.z, vv.w};
                #pragma unroll
                for (int j = 0; j < 4; j++) {
                    const uint32_t z = __vcmpeq4(vw[j], 0u);  // 0xFF in each flagged byte
                    w[j] = (w[j] & ~z) | (0x88888888u & z);
                    acc[j] += ~z & 0x01010101u;
                }
            }
            *reinterpret_cast<uint4 *>(out + tk * out_row) = make_uint4(w[0], w[1], w[2], w[3]);
        }
        if (kValid && (pending += kRows) > 240 - kRows) widen();
    }
    if (have < end) {  // value 0 + 0i past the set's samples
        int64_t t = first;
        if (t < have) t += (have - t + rows_per_block - 1) / rows_per_block * rows_per_block;
        for (; t < end; t += rows_per_block)
            *reinterpret_cast<uint4 *>(out + t * out_row) = make_uint4(0x88888888u, 0x88888888u, 0x88888888u, 0x88888888u);
    }
    if (!a.counts) return;
    if (kValid) {
        widen();
        #pragma unroll
        for (int m = 0; m < 16; m++)
            atomicAdd(count + count_slot(lc, m), (int)((acc16[2 * (m >> 2) + (m & 1)] >> (16 * ((m >> 1) & 1))) & 0xFFFFu));
    } else if (by == 0 && rsub == 0) {  // every sample usable: the first block adds the set's
        int32_t *cnt = a.counts + ((int64_t)set * a.nf + c) * a.N + ic;
        for (int m = 0; m < n; m++) atomicAdd(cnt + m, (int)have);
    }
}

// The chunks that hold a delayed input: copied, with the delayed inputs' samples
// from the history's ring, which holds the launch's too -- their rows are dense
// there, so that reading them d samples back stays in L2, where the block's rows
// do not.  In blocks of their own: among plain ones they kept whole warps waiting
// (N = 496 x 188 channels x 30,415 samples, 7 inputs delayed, 1.9 ms with the two
// mixed, 1.58 as two launches, 1.52 as the blocks of one).  !kAhead, where a ring of that size would not be
// worth its memory: the launch's own samples from the block.
template <bool kAhead>
__device__ __forceinline__ void pack_shifted_rows(const PackArgs &a, const ShiftArgs &sa, const PackGrid &g, int bx, int by)
{
    const int64_t cols = g.all;
    const int cols_per_block = g.cols, rows_per_block = g.rows, span = g.span;
    const int64_t col = (int64_t)bx * cols_per_block + threadIdx.x % cols_per_block;
    const int rsub = threadIdx.x / cols_per_block;
    if (col >= cols || rsub >= rows_per_block) return;
    int c, j, ic;
    pack_column(a, col, c, j, ic);
    const int n = min(16, a.N - ic);
    const int64_t f = a.f0 + c;
    const int64_t row_bytes = (int64_t)a.F * a.N, ring_bytes = (int64_t)a.F * sa.S;
    const uint8_t *blk = a.block + a.t0 * row_bytes + f * a.N + ic;
    const int64_t out_row = (int64_t)a.nf * a.pitch;
    const int64_t first = (int64_t)by * span * rows_per_block + rsub;
    const int64_t last = min(a.nt, ((int64_t)by + 1) * span * rows_per_block);
    int slot0 = -1;        // ring column of the chunk's first delayed input
    uint32_t delayed = 0;  // its delayed inputs
    for (int m = 0; m < n; m++)
        if (sa.delay[ic + m] > 0) {
            if (slot0 < 0) slot0 = sa.slot[ic + m];
            delayed |= 1u << m;
        }
    const uint8_t *ring = sa.hist + f * sa.S + slot0;
    const int64_t head = sa.head();
    uint8_t *out = a.out + (int64_t)c * a.pitch + j * 16;
    for (int64_t t = first; t < last; t += (int64_t)kPackRows * rows_per_block) {
        Loaded16 x[kPackRows];
        uint32_t w[kPackRows][4];
        #pragma unroll
        for (int k = 0; k < kPackRows; k++)
            x[k] = load16(blk + min(t + (int64_t)k * rows_per_block, last - 1) * row_bytes, n);
        #pragma unroll
        for (int k = 0; k < kPackRows; k++) {
            const uint4 xv = value16(x[k]);
            w[k][0] = xv.x;
            w[k][1] = xv.y;
            w[k][2] = xv.z;
            w[k][3] = xv.w;
        }
        int s = 0;
        for (uint32_t todo = delayed; todo; todo &= todo - 1, ++s) {
            const int m = __ffs(todo) - 1;
            const int64_t d = sa.delay[ic + m];
            const uint32_t byte = 0xFFu << (8 * (m & 3));
            uint32_t b[kPackRows];
            #pragma unroll
            for (int k = 0; k < kPackRows; k++) {
                const int64_t src = min(t + (int64_t)k * rows_per_block, last - 1) - d;
                const uint8_t *from = !kAhead && src >= 0 ? blk + src * row_bytes + m : ring + sa.row(head, src) * ring_bytes + s;
                b[k] = 0x01010101u * __ldg(from);
            }
            #pragma unroll
            for (int k = 0; k < kPackRows; k++) {
                #pragma unroll
                for (int q = 0; q < 4; q++) {
                    const uint32_t here = q == m >> 2 ? byte : 0u;
                    w[k][q] = (w[k][q] & ~here) | (b[k] & here);
                }
            }
        }
        #pragma unroll
        for (int k = 0; k < kPackRows; k++) {
            const int64_t tk = t + (int64_t)k * rows_per_block;
            if (tk >= last) break;
            *reinterpret_cast<uint4 *>(out + tk * out_row) = make_uint4(w[k][0], w[k][1], w[k][2], w[k][3]);
        }
    }
}

// A block's counts go to memory from shared memory, consecutive inputs by consecutive
// threads: added by each thread, 16 inputs apart, they took longer than the samples where
// a row is short and its blocks many (GB300, one gate with flags, N = 560 x 5 channels x
// 26,713 samples 278 us and so 46; without flags, N = 256 x 64 x 8192, 277 and 43 with
// the samples counted once).  Blocks an SM: unaligned rows, without flags, 42 us with
// four and 47 with three (N = 203 x 64 x 10,007).
template <bool kAligned, bool kValid>
__global__ void __launch_bounds__(kPackThreads, kValid ? 3 : kAligned ? 0 : 4)
pack_kernel(const __grid_constant__ PackArgs a, const PackGrid g)
{
    if constexpr (!kValid) {
        pack_rows<kAligned, false>(a, g, (int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z, nullptr);
    } else {
        __shared__ int count[16 * kPackThreads];
        for (int k = threadIdx.x; k < 16 * g.cols; k += kPackThreads) count[k] = 0;
        __syncthreads();
        pack_rows<kAligned, true>(a, g, (int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z, count);
        __syncthreads();
        if (!a.counts) return;
        // the block's columns from its first on: channel c0, chunk k0
        const int per = a.pitch / 16, m = threadIdx.x & 15;
        const int64_t col0 = (int64_t)blockIdx.x * g.cols, c0 = col0 / per;
        const int k0 = (int)(col0 - c0 * per), cols = (int)min((int64_t)g.cols, g.all - col0);
        for (int lc = threadIdx.x >> 4; lc < cols; lc += kPackThreads / 16) {
            const int c = (k0 + lc) / per, ic = 16 * (k0 + lc - c * per), usable = count[count_slot(lc, m)];
            if (ic + m < a.N && usable) atomicAdd(a.counts + ((int64_t)blockIdx.z * a.nf + c0 + c) * a.N + ic + m, usable);
        }
    }
}

// The chunks of `a` and, after their blocks, those of `b`, which hold delayed inputs.
template <bool kAligned, bool kAhead>
__global__ void __launch_bounds__(kPackThreads)
pack_shifted_kernel(const __grid_constant__ PackArgs a, const __grid_constant__ PackArgs b,
                    const __grid_constant__ ShiftArgs sa, const PackGrid ga, const PackGrid gb)
{
    const int na = ga.nx * ga.ny, x = (int)blockIdx.x;
    if (x < na) pack_rows<kAligned, false>(a, ga, x % ga.nx, x / ga.nx, 0, nullptr);
    else pack_shifted_rows<kAhead>(b, sa, gb, (x - na) % gb.nx, (x - na) / gb.nx);
}

bool pack_args_ok(const PackArgs &a)
{
    return a.block && a.out && a.pitch > 0 && a.pitch % 16 == 0 && a.nt <= kMaxChunkSamples &&
           (reinterpret_cast<uintptr_t>(a.out) & 15) == 0;
}

bool rows_aligned(const PackArgs &a)
{
    return a.N % 16 == 0 && (reinterpret_cast<uintptr_t>(a.block) & 15) == 0 &&
           (reinterpret_cast<uintptr_t>(a.valid) & 15) == 0;
}

}  // namespace

cudaError_t launch_pack(const PackArgs &a, int num_sms, cudaStream_t s)
{
    const int64_t cols = (int64_t)a.nf * (a.pitch / 16);
    if (cols <= 0 || a.nt <= 0) return cudaSuccess;
    if (!pack_args_ok(a) || a.chunks || a.pitch < a.N || a.sets > kMaxGates || (a.sets > 0 && !a.idx))
        return cudaErrorInvalidValue;
    const PackGrid g = pack_grid(a, cols, num_sms);
    const bool aligned = rows_aligned(a);
    auto kernel = a.valid ? (aligned ? pack_kernel<true, true> : pack_kernel<false, true>)
                          : (aligned ? pack_kernel<true, false> : pack_kernel<false, false>);
    kernel<<<dim3((unsigned)g.nx, (unsigned)g.ny, a.sets > 0 ? a.sets : 1), kPackThreads, 0, s>>>(a, g);
    return cudaGetLastError();
}

cudaError_t launch_pack_shifted(const PackArgs &a, int32_t n_shifted, const ShiftArgs &sa, int num_sms, cudaStream_t s)
{
    if (a.nf <= 0 || a.nt <= 0 || a.n_chunks + n_shifted <= 0) return cudaSuccess;
    if (!pack_args_ok(a) || !a.chunks || a.n_chunks < 0 || n_shifted < 0 || a.valid || a.idx || a.sets)
        return cudaErrorInvalidValue;
    PackArgs b = a;
    b.chunks = a.chunks + a.n_chunks;
    b.n_chunks = n_shifted;
    const PackGrid ga = pack_grid(a, (int64_t)a.nf * a.n_chunks, num_sms);
    const PackGrid gb = pack_grid(b, (int64_t)b.nf * b.n_chunks, num_sms);
    const int64_t blocks = (int64_t)ga.nx * ga.ny + (int64_t)gb.nx * gb.ny;
    if (blocks > 2147483647LL) return cudaErrorInvalidValue;
    const bool aligned = rows_aligned(a);
    auto kernel = sa.ahead ? (aligned ? pack_shifted_kernel<true, true> : pack_shifted_kernel<false, true>)
                           : (aligned ? pack_shifted_kernel<true, false> : pack_shifted_kernel<false, false>);
    kernel<<<(unsigned)blocks, kPackThreads, 0, s>>>(a, b, sa, ga, gb);
    return cudaGetLastError();
}

}  // namespace xeng
