// triangle_add.cuh -- what the single-pass epilogues share when a launch adds
// to the triangle instead of storing it (a later piece of an integration).
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace xeng {
namespace {

// Ask L2 for the values that a warp adds columns i_lo .. i_hi - 1 to, inputs
// j_warp .. j_warp + 31, of one channel's triangle `out`: one column per lane
// at a time, each a run of at most 256 bytes (three 128-byte lines).  The
// epilogue reads these one 8-column chunk ahead of their use, a microsecond from
// HBM; issued an item ahead, this takes the reads to L2's latency.  GB300, pushes
// of 256 samples, 256 channels x 512 inputs: 172 us without it.
__device__ __forceinline__ void prefetch_triangle(const int2 *out, int N, int j_warp, int i_lo, int i_hi, int i_step,
                                                  int lane)
{
    // lanes 8k .. 8k + 7 take the eight columns of every fourth chunk
    for (int i0 = i_lo + (lane >> 3) * i_step; i0 < i_hi; i0 += 4 * i_step) {
        const int i = i0 + (lane & 7);
        const int j0 = max(i, j_warp), j1 = min(j_warp + 31, N - 1);
        if (j0 > j1) continue;
        const int base = i * N - i * (i - 1) / 2 - i;
        const uintptr_t first = reinterpret_cast<uintptr_t>(out + base + j0);
        const uintptr_t last = reinterpret_cast<uintptr_t>(out + base + j1);
        for (uintptr_t p = first & ~(uintptr_t)127; p <= last; p += 128)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(p < first ? first : p));
    }
}

}  // namespace
}  // namespace xeng
