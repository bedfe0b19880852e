// launch_rule.h -- which single-pass kernel takes a launch, and how it is cut, from
// sizes alone: host code without CUDA calls, part of single_pass.cu, which defines the
// build parameters XENG_PAIR_COST and XENG_ONEPASS_COST.
#pragma once
#include <algorithm>
#include <cstdint>

#include "xeng_internal.h"

namespace xeng {

// Evenly cut items of the N <= 256 kernel: stages per CTA at least.  Shared items:
// stages per CTA at least, CTAs per item at most (build parameters).
constexpr int kSMinPiece = 32;
#ifndef XENG_SMALL_MIN_SHARED
#define XENG_SMALL_MIN_SHARED 2
#endif
#ifndef XENG_SMALL_MAX_SHARED
#define XENG_SMALL_MAX_SHARED 32
#endif
constexpr int kSMinShared = XENG_SMALL_MIN_SHARED, kSMaxShared = XENG_SMALL_MAX_SHARED;

// ns of a 128-sample stage of an item above 256 inputs, from the two build parameters,
// and whether one of them, as 0, forces its kernel.
constexpr int64_t kPairStageNs = 1200 * (int64_t)XENG_PAIR_COST / 118;
constexpr int64_t kOnepassStageNs = 770 * (int64_t)XENG_ONEPASS_COST / 36;
constexpr bool kCostForces = XENG_PAIR_COST == 0 || XENG_ONEPASS_COST == 0;

static bool use_pair_kernel(int32_t N)
{
    const int64_t b2 = (N + 255) / 256, b1 = (N + 127) / 128;
    return (int64_t)XENG_PAIR_COST * (b2 * (b2 + 1) / 2) < (int64_t)XENG_ONEPASS_COST * (b1 * (b1 + 1) / 2);
}

int small_split(int64_t n_items, int n_k, int num_sms, int32_t *split)
{
    // Few items: as many CTAs per item as there are SMs for, each with at least
    // kSMinShared stages -- unless an even cut would leave a CTA over 16 stages
    // less to do (GB300, N = 256 x 40 channels x 32,768 samples, 60 items: 162 us
    // with two CTAs per item on 120 SMs, 159 cut evenly over 152).
    const int64_t total = n_items * n_k;
    int64_t s = num_sms / n_items;
    if (s > n_k / kSMinShared) s = n_k / kSMinShared;
    if (s > kSMaxShared) s = kSMaxShared;
    if (s >= 2 && n_k / s <= total / num_sms + 16) {
        *split = (int32_t)s;
        return (int)(n_items * s);
    }
    // Short items: whole ones, since a partial block costs as much as the stages
    // that an even cut saves (GB300, N = 256 x 128 channels x 256 samples: 25 us;
    // cut evenly into pieces of kSMinPiece stages, 209).
    if (n_k < kSMinPiece) {
        *split = kSmallWhole;
        return (int)(n_items < num_sms ? n_items : num_sms);
    }
    *split = kSmallEven;
    const int64_t grid = total / kSMinPiece;
    return (int)(grid < num_sms ? grid : num_sms);
}

// Channels whose block pairs fill whole rounds of the pair kernel, where the rest
// takes less than another round in the one pass (5 us for the second launch); 0:
// one launch for all.  GB300, N = 1024 x 64 channels x 8192 samples, 640 items on
// 76 clusters: 717 us in nine rounds, 690 as eight and a launch of four channels.
int32_t single_pass_cut(int kernel, int32_t N, int64_t nf, int64_t nt, int accumulate, int num_sms)
{
    if (kernel != kSinglePair || kCostForces) return 0;
    const int64_t n_k = (nt + 127) / 128, units = num_sms / 2;
    const int64_t b2 = (N + 255) / 256, per = b2 * (b2 + 1) / 2, b1 = (N + 127) / 128, per1 = b1 * (b1 + 1) / 2;
    const int64_t full = nf * per / units, cut = full * units / per;
    if (cut <= 0 || cut >= nf) return 0;
    const int64_t ones = ((nf - cut) * per1 + num_sms - 1) / num_sms;
    const int64_t t_round = kPairStageNs * n_k + (accumulate ? 12300 : 7400);
    return ones * (kOnepassStageNs * n_k + (accumulate ? 3200 : 1600)) + 5000 < t_round ? (int32_t)cut : 0;
}

int64_t single_pass_ns(int kernel, int32_t N, int64_t nf, int64_t nt, int accumulate, int num_sms, int *best)
{
    // Rounds of the grid times an item's time in ns, fitted to launches of 2 .. 256
    // stages of 128 samples (GB300; us per item at 2 / 8 / 64 / 256 stages, storing:
    // pair kernel 8.4 / 16.8 / 83.5 / 314, one pass 3.0 / 7.8 / 52 / 204, N <= 256
    // kernel 7.9 / 14.9 / --; adding: 14.7 / -- / 87 / --, 5.3 / 9.3 / 55 / --,
    // 14.9 / 24.8 / --).  At 64 stages and many rounds the first two are in the ratio
    // of XENG_PAIR_COST and XENG_ONEPASS_COST.  A few rounds, and short launches,
    // favour the one pass, whose items are the smallest and whose epilogue overlaps
    // the next item (us a call, the N-only choice / the one pass: N = 1024 x 4
    // channels x 32,768 samples 322 / 207; 512 x 256 x 256 100 / 65; 256 x 256 x 256
    // 32 / 25); above about 1900 inputs and many channels its items take a quarter
    // longer.
    const int64_t n_k = (nt + 127) / 128;
    auto rounds = [](int64_t items, int64_t units) { return (items + units - 1) / units; };
    const int64_t b2 = (N + 255) / 256, b1 = (N + 127) / 128;
    const int64_t ones = rounds(nf * (b1 * (b1 + 1) / 2), num_sms);
    int64_t t_one = ones * (kOnepassStageNs * n_k + (accumulate ? 3200 : 1600));
    if (N > 1900 && ones > 8 && n_k > 32) t_one += t_one / 4;
    if (kernel == kSingleSmall) {
        // By how it cuts its items: between CTAs (an exchange of partial blocks, then
        // the stages of one CTA) or whole.  The exchange costs more than the stages it
        // takes off the CTAs of a short launch (us a call, the N <= 256 kernel / the
        // one pass: N = 256 x 8 channels x 1024 samples 22.3 / 14.3, x 2048 22.5 / 19.2,
        // x 4096 26.1 / 30.6; 256 x 48 x 4096 37.9 / 31.3, x 8192 56.0 / 54.4; 160 x 2
        // x 256 15.0 / 9.0; 128 x 152 x 4096 39.5 / 27.7, x 32,768 168 / 191).
        const int64_t items = N > 128 ? nf + (nf + 1) / 2 : (nf + 1) / 2;
        const int64_t n_one = accumulate ? 3200 : 1600;
        int32_t split;
        const int grid = small_split(items, (int)n_k, num_sms, &split);
        int64_t t_small;
        if (split == kSmallWhole)
            t_small = 2000 + rounds(items, num_sms) * (1100 * n_k + (accumulate ? 13500 : 5000));
        else if (split == kSmallEven)  // one item a CTA is as good as whole
            t_small = (grid == items ? 6000 : 18000) + 1200 * (items * n_k / grid) + (accumulate ? 11000 * items / grid : 0);
        else
            t_small = 9000 + 25 * N + 1100 * n_k / split + (accumulate ? 5500 : 0);
        const int64_t t = ones * ((N > 128 ? 770 : 680) * n_k + n_one);
        *best = t_small <= t ? kernel : kSingleOnepass;
        return std::min(t_small, t);
    }
    const int64_t t_pair = rounds(nf * (b2 * (b2 + 1) / 2), num_sms / 2) * (kPairStageNs * n_k + (accumulate ? 12300 : 7400));
    *best = kCostForces ? kernel : t_pair < t_one ? kSinglePair : kSingleOnepass;
    return *best == kSinglePair ? t_pair : t_one;
}

int single_pass_by_shape(int kernel, int32_t N, int64_t nf, int64_t nt, int accumulate, int num_sms)
{
    if (kernel != kSingleSmall && kernel != kSinglePair && kernel != kSingleOnepass) return kernel;
    int best = 0;
    single_pass_ns(kernel, N, nf, nt, accumulate, num_sms, &best);
    return best;
}

}  // namespace xeng
