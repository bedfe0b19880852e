// xeng_internal.h -- declarations shared by the library's translation units.
#pragma once
#include <cstdint>
#include <vector>
#include <cuda.h>
#include <cuda_runtime.h>

namespace xeng {

constexpr int kTile = 128;          // inputs per tensor-engine tile, samples per K chunk
constexpr int kMaxChunkSamples = 65536;  // f32 sums stay <= 128 * 65536 = 2^23 (exact)
// Raw-nibble launches (the fused kernel, the tensor path's raw planes): their
// integer sums stay <= 450 * 32768 = 14,745,600 < 2^24, the range in which the
// GPU tests (test_raw_nibble_sums_up_to_2_24, test_raw_nibble_unit_terms_above_2_23)
// show the tensor core's f32 accumulation exact with unit increments.
constexpr int kFusedMaxSamples = 32768;

// Device-side status codes written to the handle's error word.
enum DevStatus : int {
    kDevOk = 0,
    kDevTimeoutProducer = 1,
    kDevTimeoutMma = 2,
    kDevTimeoutEpilogue = 3,
};

// What the kernels' `err` points at, in device memory: their status word and
// the device address of its mirror in pinned host memory (may be null).
struct StatusBlock {
    int status;
    int pad_;
    int *mirror;
};
// A zeroed status block and its zeroed mirror (both null on failure).
cudaError_t status_alloc(int **d_err, int **h_err);
void status_free(int *d_err, int *h_err);

inline int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }
inline int64_t n_baselines(int64_t n) { return n * (n + 1) / 2; }

// Standalone decode: block [T][F][N] bytes -> planes [nf][2][n_pad][t_pad] E4M3 codes.
cudaError_t launch_decode(const uint8_t *block, int64_t T, int32_t F, int32_t N,
                          int32_t f0, int32_t nf, uint8_t *planes, int64_t t_pad,
                          int64_t n_pad, cudaStream_t s);

// The same decode as a persistent TMA pipeline (one CTA per SM): needs N a
// multiple of 16 and a 16-byte aligned block (decode_tma_ok), t_pad and n_pad
// multiples of 128.  A stalled pipeline sets *err and returns.
bool decode_tma_ok(const uint8_t *block, int32_t N);
// partials non-null: raw-nibble planes (E4M3 codes of u / 512) and per-tile
// per-input nibble sums [nf][t_pad / 128][n_pad] of (P, Q); null: decoded planes.
cudaError_t launch_decode_tma(const uint8_t *block, int64_t T, int32_t F, int32_t N, int32_t f0, int32_t nf,
                              uint8_t *planes, int64_t t_pad, int64_t n_pad, int *err, int num_sms, cudaStream_t s,
                              int2 *partials = nullptr);
// sums[fl][i] = (S, D) = (P + Q, P - Q) over all sample tiles of the partials
cudaError_t launch_plane_sums(const int2 *partials, int32_t nf, int32_t n_tb, int32_t n_pad, int2 *sums, int num_sms,
                              cudaStream_t s);

// Gated / flagged decode of channels [f0, f0 + nf): tile rows are block rows
// idx[0 .. Tg) (one gate's samples); samples whose valid byte is 0 decode to
// zero; usable samples per (channel, input) are added to counts[fl][N] (may be null).
cudaError_t launch_decode_gather(const uint8_t *block, int32_t F, int32_t N, int32_t f0, int32_t nf, const int32_t *idx,
                                 int64_t Tg, const uint8_t *valid, uint8_t *planes, int64_t t_pad, int64_t n_pad,
                                 int32_t *counts, cudaStream_t s);

// Gate accumulator sets of a handle (Sec. IV-C-4) and their usable-sample
// counts: counts[g][k] = (dirty ? counts[g][k] : 0) + base[g] for k < per_gate
// (base: samples of the set pushed without a validity mask).
constexpr int kMaxGates = 64;
struct GateBase {
    int64_t v[kMaxGates];
};
cudaError_t launch_counts_finish(int32_t *counts, int dirty, const GateBase &base, int32_t G, int64_t per_gate,
                                 cudaStream_t s);

// Batched decode: one launch over the tiles of several blocks.
struct DecodeJob {
    const uint8_t *block;  // [T][F][N]
    uint8_t *planes;       // [F][2][n_pad][pitch]: this job fills columns [0, t_pad) of every row
    int64_t T, t_pad, n_pad;
    int64_t pitch;         // bytes between plane rows (>= t_pad)
    int64_t cta0;          // first CTA of this job in the launch
    int32_t F, N;
    int32_t vec_ok;        // 16-byte loads allowed (see decode_vec_ok)
    int32_t pad_;
};
int decode_vec_ok(const uint8_t *block, int32_t N);
// CTAs one job takes in a batched decode launch.
inline int64_t decode_ctas(int64_t t_pad, int64_t n_pad, int64_t F) { return (t_pad / 128) * (n_pad / 128) * F; }
// Time shifting (Sec. IV-C-5): input i of the pushed block is read d_i
// samples late; the samples before the block come from the history.
struct ShiftArgs {
    const int32_t *delay = nullptr;        // [N] delay of input i, samples
    const int32_t *slot = nullptr;         // [N] history column of input i (-1: not delayed), in the inputs' order
    const int32_t *chunk_delay = nullptr;  // [ceil(N/16)] delay shared by inputs 16c..16c+15, or -1
    // [cap][F][S] samples of the delayed inputs, a ring of rows: sample 0 of the
    // block (or of the launch, see launch_pack_shifted) belongs at row head(), and
    // every sample from max(delay) before it on is there
    const uint8_t *hist = nullptr;
    // where: {row of the last append's first sample, its rows, a ticket}, in device
    // memory, so that captured pushes go on from where the ring is when they run
    const int64_t *state = nullptr;
    int64_t cap = 0;
    int32_t S = 0;
    int32_t ahead = 0;  // != 0: the launch's own samples are there too, appended last
    __device__ int64_t head() const
    {
        const int64_t r = state[0] + (ahead ? 0 : state[1]);
        return r >= cap ? r - cap : r;
    }
    // the row of sample src, |src| <= cap
    __device__ int64_t row(int64_t head, int64_t src) const
    {
        const int64_t r = head + src;
        return r < 0 ? r + cap : r >= cap ? r - cap : r;
    }
};
// Decode samples t0 .. t0 + nt - 1 of the block (T_block samples) with the
// shift applied, channels f0 .. f0 + nf - 1, into planes as launch_decode.
cudaError_t launch_decode_shifted(const uint8_t *block, int64_t t0, int64_t nt, int32_t F, int32_t N, int32_t f0,
                                  int32_t nf, const ShiftArgs &sa, uint8_t *planes, int64_t t_pad, int64_t n_pad,
                                  cudaStream_t s);
// Batched TMA decode: job j's block [T][F][N] into its planes [F][2][n_pad][t_pad]
// through the maps encode_decode_tma_maps writes (device array: raw map 2j,
// plane map 2j + 1); tiles tile0[j] .. tile0[j] + n_ib * F * n_tb - 1 are job
// j's.  prepare_decode_tma_batch sets the kernel's shared-memory limit (call
// it before capturing a launch in a graph).
struct DecTmaJob {
    int64_t tile0;
    int64_t T;
    int32_t n_ib, n_tb, F, N, n_pad;
    int32_t x0;          // first plane column of the job in its plane map (a multiple of 128)
    int2 *partials;      // non-null: raw-nibble planes, the tiles' (P, Q) sums to
                         // partials[fl][x0 / 128 + tb][n_pad] ...
    int32_t part_n_tb;   // ... whose rows per channel are part_n_tb
    int32_t pad_;
};
// Totals of raw-nibble partial sums for several jobs in one launch: job j's
// sums[fl][i] = (S, D) over tile rows 0 .. n_tb - 1 of partials[fl][.][i]
// (rows per channel part_n_tb); its entries are k = first .. first + F * n_pad - 1.
struct SumJob {
    const int2 *partials;
    int2 *sums;
    int64_t first;
    int32_t n_tb, part_n_tb, n_pad, pad_;
};
cudaError_t launch_plane_sums_batch(const SumJob *jobs, int32_t n_jobs, int64_t total, int num_sms, cudaStream_t s);
bool encode_decode_tma_maps(const uint8_t *block, int64_t T, int32_t F, int32_t N, uint8_t *planes, int64_t t_pad,
                            int64_t n_pad, CUtensorMap *raw_map, CUtensorMap *plane_map);
cudaError_t prepare_decode_tma_batch();
cudaError_t launch_decode_tma_batch(const CUtensorMap *maps, const DecTmaJob *jobs, int n_jobs, int64_t n_tiles,
                                    int *err, int num_sms, cudaStream_t s);

// After a plain decode of samples t0 .. t0 + nt - 1 into planes: rewrite the
// rows of the S delayed inputs (inputs[s] has history column s) with their
// shifted samples, as launch_decode_shifted computes them.
cudaError_t launch_shift_fixup(const uint8_t *block, int64_t t0, int64_t nt, int32_t F, int32_t N, int32_t f0,
                               int32_t nf, const ShiftArgs &sa, const int32_t *inputs, uint8_t *planes, int64_t t_pad,
                               int64_t n_pad, cudaStream_t s);
// Appends samples t0 .. t0 + m - 1 of the block's S delayed inputs, listed in
// `inputs`, to the ring (m <= cap) and updates its state (ShiftArgs).
cudaError_t launch_shift_history(uint8_t *hist, const uint8_t *block, int64_t t0, int64_t m, int32_t F, int32_t N,
                                 const int32_t *inputs, int32_t S, int64_t cap, int64_t *state, cudaStream_t s);

// Raw samples rearranged into rows of `pitch` bytes (a multiple of 16) per
// channel, out[nt][nf][pitch], for a single-pass launch: row t is the block's
// sample t0 + t, or idx[t] where idx (device memory) is given; channels
// f0 .. f0 + nf - 1.  launch_pack (pitch >= N) also replaces samples whose
// `valid` byte is 0 by 0x88 and adds the usable samples to counts[nf][N]; both
// may be null.  launch_pack_shifted takes two lists of 16-byte chunks, `chunks`
// (device memory; position in the packed row, 16-input chunk of the block): n_chunks
// that are copied and then n_shifted that hold delayed inputs, to which it applies the
// delays of `sa` (head(): row of sample t0), whose ring has to hold the launch's
// samples already where sa.ahead; the others of the row are left as they are.  nt <=
// kMaxChunkSamples.  launch_pack with
// sets > 0: that many lists of samples side by side, out[nt][sets][nf][pitch] and
// counts[sets][nf][N], set k's samples idx[set_first[k]] .. idx[set_first[k + 1] - 1],
// its rows past them 0x88.
struct PackArgs {
    const uint8_t *block = nullptr;
    int64_t t0 = 0, nt = 0;
    int32_t F = 0, N = 0, f0 = 0, nf = 0;
    const int32_t *idx = nullptr;
    const uint8_t *valid = nullptr;
    int32_t *counts = nullptr;
    const int2 *chunks = nullptr;
    int32_t n_chunks = 0;
    int32_t pitch = 0;
    uint8_t *out = nullptr;
    int32_t sets = 0;
    int32_t set_first[kMaxGates + 1];
};
cudaError_t launch_pack(const PackArgs &a, int num_sms, cudaStream_t s);
cudaError_t launch_pack_shifted(const PackArgs &a, int32_t n_shifted, const ShiftArgs &sa, int num_sms, cudaStream_t s);

// What the three single-pass launches below share.  A block's rows are `pitch`
// bytes per channel (0: N), a multiple of 16; N itself need not be one.  With
// `sub`, the 128-input blocks b with slot[b] >= 0 are read from packed
// [nt][F][128 n] (16-byte aligned) instead, at inputs 128 slot[b] ..: the
// launch's samples, rearranged (launch_pack_shifted), the launch's channels from
// its channel f0 on.
constexpr int kMaxBlocks = 32;  // 128-input blocks of 4096 inputs
struct SubBlocks {
    const uint8_t *packed;
    int32_t n, F, f0;
    int8_t slot[kMaxBlocks];
};
// The raw block's tensor map of their stages (3D: input, channel, sample; boxes of
// 128 inputs x 1 channel x `stage` samples, 128-byte swizzle).  `wide`: L2 fetches
// 256 bytes for a miss, for launches that read the next 128 inputs too.
cudaError_t encode_raw_map(CUtensorMap *map, const uint8_t *block, int64_t T_block, int32_t F, int32_t N,
                           int32_t pitch, int stage, bool wide = true);

// Decode fused into the correlation for N <= 256 (small_ok: pitch % 16 == 0, block
// 16-byte aligned): samples t0 .. t0 + nt - 1 (nt <= kFusedMaxSamples) of the
// block (T_block samples), channels f0 .. f0 + nf - 1, stored (accumulate = 0)
// or added into acc [nf][N(N+1)/2][2] (8-byte aligned); no decoded planes.
// Single CTAs over upper-triangle 128 x 128 blocks only (three per channel of
// 129..256 inputs).  The launch's work is split evenly over the CTAs; an item
// cut between CTAs is completed through ws (scratch of small_ws_bytes(num_sms))
// and flags (small_flags_bytes(num_sms), zeroed once: a flag per CTA, the
// count of launches on them and an arrival counter, with which the last CTA of
// each launch advances the count, so replays of a captured launch stay apart).
// max_ctas (0: num_sms): CTAs at most, where others are to run beside them.
bool small_ok(const uint8_t *block, int32_t N, int32_t pitch = 0);
size_t small_ws_bytes(int num_sms);
size_t small_flags_bytes(int num_sms);
cudaError_t launch_correlate_small(const uint8_t *block, int64_t T_block, int64_t t0, int64_t nt, int32_t F, int32_t N,
                                   int32_t f0, int32_t nf, int32_t *acc, int accumulate, int2 *ws, int *flags,
                                   int *err, int num_sms, cudaStream_t s,
                                   const CUtensorMap *maps = nullptr, int32_t spb = 0,
                                   int32_t pitch = 0, const SubBlocks *sub = nullptr, int max_ctas = 0);
int small_stage_samples();  // its stage

// One pass over the raw bytes for N up to 4096 (rows of 16-byte multiples, block
// 16-byte aligned; used above 256 inputs): single CTAs over every channel's
// upper-triangle pairs of 128-input blocks, the nibble split and each pair's
// nibble sums in shared memory; nt <= kFusedMaxSamples, acc 8-byte aligned.
bool onepass_ok(const uint8_t *block, int32_t N, int32_t pitch = 0);
cudaError_t launch_correlate_onepass(const uint8_t *block, int64_t T_block, int64_t t0, int64_t nt, int32_t F,
                                     int32_t N, int32_t f0, int32_t nf, int32_t *acc, int accumulate, int *err,
                                     int num_sms, cudaStream_t s,
                                     const CUtensorMap *maps = nullptr, int32_t spb = 0,
                                     int32_t pitch = 0, const SubBlocks *sub = nullptr);
int onepass_stage_samples();  // its stage

// Decode fused into the correlation for N <= 4096 (rows of 16-byte multiples, block
// 16-byte aligned), as launch_correlate_small: 2-CTA clusters over every
// channel's upper-triangle pairs of 256-input blocks, nibble sums in shared
// memory; nt <= kFusedMaxSamples, acc 8-byte aligned.
bool pair_ok(const uint8_t *block, int32_t N, int32_t pitch = 0);
cudaError_t launch_correlate_pair(const uint8_t *block, int64_t T_block, int64_t t0, int64_t nt, int32_t F, int32_t N,
                                  int32_t f0, int32_t nf, int32_t *acc, int accumulate, int *err, int num_sms,
                                  cudaStream_t s,
                                  const CUtensorMap *maps = nullptr, int32_t spb = 0,
                                  int32_t pitch = 0, const SubBlocks *sub = nullptr);
// One job of a listed launch of the pair kernel (a batch's jobs in one
// persistent launch): its raw block's tensor map (encode_raw_map, in device
// memory, 64-byte aligned), its output [F][N(N+1)/2][2] (stored) and sizes: nt
// <= kFusedMaxSamples samples in n_k stages, nt2 256-input blocks and
// pairs_per_ch upper-triangle block pairs per channel, its items item0 ..
// item0 + F * pairs_per_ch - 1 of the launch (jobs in increasing item0).
struct PairJob {
    const CUtensorMap *map;
    int32_t *acc;
    int32_t N, nt, n_k, nt2, pairs_per_ch, item0;
};
cudaError_t launch_correlate_pair_listed(const PairJob *jobs, int32_t n_jobs, int64_t n_items, int *err, int num_sms,
                                         cudaStream_t s);
int pair_stage_samples();  // its stage

// The single-pass kernel (single_pass.cu) that takes a block of N inputs:
// kSingleSmall (N <= 256), kSingleOnepass or kSinglePair (above, by the
// measured cost of their block pairs), or 0 where none applies (N not a
// multiple of 16 (where `pitch` is not given), block not 16-byte aligned, a kernel
// switched off, or
// `bounded` and N above the build's XENG_FUSED_MAX_N, where two passes are
// faster).  `force`: 0, a kernel to take for every N it covers, or kSingleNone.
enum SinglePass { kSingleNone = -1, kSingleSmall = 1, kSingleOnepass = 2, kSinglePair = 3 };
// The environment variable XENG_FUSED_KERNEL: "pair", "onepass" (force that
// kernel), "none" (no single pass for the default engine and batches), else 0.
int single_pass_force_from_env();
int single_pass_kernel(const uint8_t *block, int32_t N, int force, bool bounded, int32_t pitch = 0);
// For one launch of nf channels x nt samples, storing or adding, whose kernel is
// not forced: the kernel whose rounds of the grid take less time -- of the two over
// block pairs, or (kernel = kSingleSmall) of that one and the one pass.  All three
// read the same stages.
int single_pass_by_shape(int kernel, int32_t N, int64_t nf, int64_t nt, int accumulate, int num_sms);
// The time that this choice, *best, takes by the same rule, in ns.
int64_t single_pass_ns(int kernel, int32_t N, int64_t nf, int64_t nt, int accumulate, int num_sms, int *best);
// Channels that a launch of the pair kernel (by shape) takes before the one pass takes
// the others; 0: all.
int32_t single_pass_cut(int kernel, int32_t N, int64_t nf, int64_t nt, int accumulate, int num_sms);
// How a launch of the N <= 256 kernel cuts its items (n_k stages each) over the
// CTAs, at most one per SM: *split CTAs share each item (2 or more), or all stages
// are cut evenly (kSmallEven), or the items stay whole (kSmallWhole); returns the grid.
constexpr int kSmallEven = 0, kSmallWhole = 1;
int small_split(int64_t n_items, int n_k, int num_sms, int32_t *split);
// Scratch of the N <= 256 kernel, allocated at its first launch (flags zeroed
// on the stream) and owned by the caller.
struct SmallScratch {
    int2 *ws = nullptr;
    int *flags = nullptr;
};
cudaError_t small_scratch_alloc(SmallScratch *sc, int num_sms, cudaStream_t s);
void small_scratch_free(SmallScratch *sc);
// One launch of single-pass kernel `kernel` over samples t0 .. t0 + nt - 1
// (nt <= kFusedMaxSamples) and channels f0 .. f0 + nf - 1 of the block.  With
// `maps` (device memory, 64-byte aligned), the samples come instead from
// consecutive blocks of spb stages each, block k through maps[k] (made by
// encode_raw_map); block is then unused and t0 must be 0.  max_ctas: of the N <= 256
// kernel.
cudaError_t launch_single_pass(int kernel, const uint8_t *block, int64_t T_block, int64_t t0, int64_t nt, int32_t F,
                               int32_t N, int32_t f0, int32_t nf, int32_t *acc, int accumulate, SmallScratch *sc,
                               int *err, int num_sms, cudaStream_t s, const CUtensorMap *maps = nullptr,
                               int32_t spb = 0, int32_t pitch = 0, const SubBlocks *sub = nullptr, int max_ctas = 0);
// The same launch with the kernel chosen by its shape (single_pass_by_shape); what
// would be a last round of the pair kernel with few items may go to the one pass,
// as a second launch (counted in *launches).
cudaError_t launch_single_pass_shaped(int kernel, const uint8_t *block, int64_t T_block, int64_t t0, int64_t nt,
                                      int32_t F, int32_t N, int32_t f0, int32_t nf, int32_t *acc, int accumulate,
                                      SmallScratch *sc, int *err, int num_sms, cudaStream_t s, int32_t pitch = 0,
                                      const SubBlocks *sub = nullptr, int64_t *launches = nullptr);
// A kernel's stage in samples.
int single_pass_stage(int kernel);

// Beamforming (Sec. IV-C-3).  The host fills T, F, N, B, out and err; the
// launcher fills the rest.
struct BfArgs {
    int64_t T = 0;
    int32_t F = 0, N = 0, B = 0;
    int32_t n_kc = 0;       // 128-input K chunks
    int32_t n_tt = 0;       // 128-sample tiles
    int64_t n_items = 0;    // F * n_tt
    int32_t f_fastest = 0;  // item order: channel fastest, else sample tile fastest
    int32_t tma_out = 0;    // B even, out 16-byte aligned: staged beams are stored by TMA
    int32_t vec = 1;        // beams per direct store: 4 (B % 4 == 0, out 32-byte aligned), 2 (as tma_out) or 1
    const uint8_t *block = nullptr;  // [T][F][N]
    int32_t *out = nullptr; // [T][F][B][2]
    const int32_t *corr = nullptr;  // [F][Bp][2] offset terms (8 sum(w_re - w_im), 8 sum(w_re + w_im))
    int *err = nullptr;
};
int beam_padded(int32_t n_beams);  // 4, 8, 16, 32 or 64
cudaError_t launch_beam_weights(const int8_t *w_re, const int8_t *w_im, int32_t F, int32_t B, int32_t N,
                                uint8_t *wdev, int32_t *corr, cudaStream_t s);
cudaError_t launch_beamform(const uint8_t *block, const uint8_t *wdev, const int32_t *corr, BfArgs a, int num_sms,
                            cudaStream_t s);

cudaError_t launch_decode_batch(const DecodeJob *jobs, int n_jobs, int64_t total_ctas, cudaStream_t s);

// Tensor-core correlation of decoded planes (tcgen05, FP8 E4M3, f32 in TMEM).
// acc: int32 [nf][N(N+1)/2][2] of the channel group; accumulate = add to it.
struct TcArgs {
    const uint8_t *planes;
    int64_t t_pad;
    int32_t n_pad;
    int32_t N;
    int32_t nf;
    int32_t *acc;
    int32_t accumulate;
    int32_t *err;
    // raw-nibble planes: per channel of the launch, (S, D) of every input row
    // [nf][n_pad], and the samples integrated (<= kFusedMaxSamples); null: decoded planes
    const int2 *sums = nullptr;
    int64_t n_samples = 0;
};
cudaError_t launch_correlate_tc(const TcArgs &a, int num_sms, cudaStream_t s);
// The same correlation with cta_group::2: clusters of two CTAs compute
// 256 x 256 tiles (a.n_pad must be a multiple of 256).
cudaError_t launch_correlate_tc2(const TcArgs &a, int num_sms, cudaStream_t s);

// Batched (listed) launches: a job table, per-job tensor maps and a work list
// partitioned by CTA, all in device memory.
struct JobDesc {
    int32_t *out;      // [F][N(N+1)/2][2] int32 of the job
    int32_t n_pad;     // inputs rounded up to 128
    int32_t N;
    int32_t mode;      // epilogue: 0 store, 1 add (read-modify-write), 2 atomic add (items share tiles)
    int32_t n_samples; // raw-nibble planes: samples integrated (the offset terms' n)
    const int2 *sums;  // raw-nibble planes: (S, D) per [F][n_pad]; null: decoded planes
};
struct WorkItem {
    int32_t job, fl;   // job index, channel within the job
    int16_t I, J;      // 128-input tile pair, I <= J
    int32_t kc0, kc1;  // 128-sample chunks [kc0, kc1), at most kMaxChunkSamples / 128 of them
};
struct ListArgs {
    const CUtensorMap *maps;   // [n_jobs], 64-byte aligned
    const JobDesc *jobs;       // [n_jobs]
    const WorkItem *items;     // [n_items]
    const int32_t *cta_begin;  // [grid + 1]: CTA b runs items [cta_begin[b], cta_begin[b + 1]);
                               // nullptr: CTA b runs items b, b + grid, b + 2 grid, ... < n_items
    int32_t *err;              // device status word
    int64_t n_items;
};
cudaError_t encode_planes_map(CUtensorMap *map, const uint8_t *planes, int64_t t_pad, int64_t rows);
cudaError_t prepare_correlate_tc_listed();
// Bounded-wait self-test (no fault, no hang): *status = device status word
// after one thread's wait ran out, *left = threads that gave up (all of them).
cudaError_t selftest_wait_timeout(int64_t limit_ns, int *status, int *left);  // kernel attributes; call before any stream capture
cudaError_t launch_correlate_tc_listed(const ListArgs &L, int grid, cudaStream_t s);

// Plain CUDA-core correlation straight from the bytes (dp4a, int32).
cudaError_t launch_correlate_dp4a(const uint8_t *block, int64_t T, int32_t F, int32_t N,
                                  int32_t *acc, int32_t accumulate, cudaStream_t s);

}  // namespace xeng
