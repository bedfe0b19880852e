// raw_offset.cuh -- from raw-nibble accumulators to visibilities, in the f32
// pipe.  With p, q the raw nibbles of a sample, P, Q their sums over the n <=
// 32,768 samples of a launch, S = P + Q and D = P - Q (paper Sec. II-A: a
// nibble holds its value + 8),
//     Re V_ij = 2^18 acc_re - 8 (S_i + S_j) + 128 n,
//     Im V_ij = 2^18 acc_im + 8 (D_i - D_j).
// With M = 1.5 x 2^23 added, every step is exact in f32 and the sum's bit
// pattern is the integer's plus a constant: M, 128 n, 8 S and 8 D are multiples
// of 8 below 2^27, so their sums are exact; the fused multiply-add rounds V + M
// once, and -112 n <= Re V <= 128 n <= 2^22, |Im V| <= 120 n put it in
// [2^23, 2^24], where the spacing is 1 (2^24 itself follows the binade's last
// pattern).  An add and a multiply-add for the value and one integer add stand
// for a multiply, a conversion (a quarter-rate instruction) and three to five
// integer operations.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace xeng {
namespace {

constexpr float kRawScale = 262144.0f;         // accumulators hold integer sums / 2^18
constexpr float kFloatToInt = 12582912.0f;     // M = 1.5 x 2^23
constexpr uint32_t kFloatToIntBits = 0x4B400000u;

// Where the sums of input k (and the terms in their place) of an item lie in
// shared memory: two entries more after every 16 inputs, so that the eight lanes
// of a converter warp that add the sums of inputs 16 l + m (l their lane's chunk)
// hit eight banks and not one.
__host__ __device__ constexpr int sum_slot(int k) { return k + 2 * (k >> 4); }

// An input's terms (-8 S, 8 D) of its nibble sums (P, Q).
__device__ __forceinline__ float2 offset_terms(int2 pq)
{
    return make_float2(-8.0f * (float)(pq.x + pq.y), 8.0f * (float)(pq.x - pq.y));
}

// The visibility part of accumulator word `acc`; `terms` is M plus its offset terms.
__device__ __forceinline__ uint32_t raw_to_int(uint32_t acc, float scale, float terms)
{
    return __float_as_uint(__fmaf_rn(scale, __uint_as_float(acc), terms)) - kFloatToIntBits;
}

}  // namespace
}  // namespace xeng
