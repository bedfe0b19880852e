// correlate_small.cu -- the whole X-engine step for up to 256 inputs in one
// kernel: the nibble split (paper Sec. II-A) fused into the Hermitian
// correlation (Sec. IV-C-1, Eq. 1), with no decoded planes in HBM, and only
// the upper-triangle 128 x 128 blocks of each channel computed.
//
// A channel of 129..256 inputs has three upper-triangle blocks of 128 inputs:
// (0,0), (0,1) and (1,1).  A pair of CTAs computing the full 256 x 256 product
// does a fourth, (1,0), that the triangle never stores: the two CTAs of a
// cta_group::2 MMA share its B operand, so neither can leave its lower block
// out.  Here each CTA works alone (cta_group::1, M = 128) on items of equal
// cost, each two 128 x 128 complex blocks, 512 TMEM columns:
//   column item of channel c:     A = inputs 128..255, B = inputs 0..255 (one
//                                 N = 256 MMA per product): blocks (0,1), (1,1)
//   diagonal item of channels c, c':  block (0,0) of each (one N = 256 and
//                                 two N = 128 MMAs per product pair)
// Up to 128 inputs a channel is one diagonal block, and every item is a
// diagonal item over two channels.  Per stage an item reads two raw tiles of
// 128 inputs x 128 samples ("X" and "Y": the channel's two input halves, or the
// two channels' lower halves).  The A operand holds inputs j and B inputs i, so
// TMEM lanes are inputs j and a warp's store of column i is one 256-byte run of
// the triangle's row i.
//
// The launch's work -- its items in order, each of n_k stages of 128 samples --
// is cut over the CTAs in one of three ways (small_split).  Few items are
// shared by several CTAs each, at one piece a CTA: all write their corrected
// partial blocks to a workspace, raise a flag stamped with the launch's epoch,
// wait (bounded) for the item's other flags, and each adds up and stores its
// share of the item's 8-column chunks.  Many short items stay whole.  Otherwise
// the sequence is cut evenly, so every CTA does the same number of MMAs whether
// or not the items divide evenly: an item cut between CTAs is finished by its
// owner, the CTA holding its first stages (which reaches them last), which adds
// the others' partial blocks to its own.  A cooperative launch keeps every CTA
// resident, so the waits end.  Bound by latency where calls are small: N = 256
// x 8 channels x 4096 samples (12 items of 32 stages) takes 23-24 us on 144 CTAs,
// 54-61 us on the 12 that pieces of 32 stages at least allowed.  Where the exchange
// of partial blocks (about 10 us) would cost more than it saves, the one pass over
// 128-input block pairs runs instead (single_pass_by_shape).
//
// The TMA writes raw tiles with a 128-byte swizzle: rows are samples, each 128
// input bytes -- the canonical MN-major layout of an 8-bit tcgen05 operand
// (inputs along M or N, samples along K).  The converter warps split each byte
// at its own offset into the Re plane (high nibble) and the Im plane (low
// nibble) of a plane stage; the raw slots form their own ring, so the TMA runs
// ahead of the conversion.  The MMAs of a column item's stage
// (both operands MN-major; B spans the X and Y tiles, the leading byte offset
// stepping from one to the other):
//     Re += A_re B_re^T + A_im B_im^T,   Im += A_re B_im^T + (-A_im) B_re^T;
// a diagonal item's tile against itself: [B_im | B_re] as one N = 256 operand.
//
// The planes hold raw nibbles: a byte whose low four bits are u (0..15) and
// whose high four bits are clear is the FP8 E4M3 code of u / 512 (the
// subnormal binade and the first normal one share the spacing 2^-9).  With p,
// q the Re and Im nibbles and x = (p - 8) + i (q - 8), over a launch of n
// samples
//     Re V_ij = sum(p_i p_j + q_i q_j) - 8 (S_i + S_j) + 128 n,
//     Im V_ij = sum(q_i p_j - p_i q_j) + 8 (D_i - D_j),
// with S = P + Q, D = P - Q and P, Q the sums of an input's nibbles, which the
// converters form as they split (byte lanes, widened to 16-bit lanes every
// four stages, totalled per piece in shared memory); a piece of an item is
// corrected with its own n and sums, and the pieces' results add up to the
// item's.  The MMA sums are integers / 2^18 of at most 450 n; launches of at
// most 32,768 samples keep them below 2^24, exact in f32.
//
// Roles (576 threads):
//   warp 0       TMA producer: raw tiles into the raw ring
//   warp 1       TMEM allocation; MMA issuer
//   warps 2..9   converters: raw slot -> Re and Im planes of a plane stage, nibble sums
//   warps 10..17 epilogue: TMEM -> packed int32 triangle, one warp per TMEM lane
//                quadrant and block of the item (items shared by up to 14 CTAs: the
//                converters too, their one piece done)
#include <cstring>

#include "tc_ptx.cuh"
#include "triangle_add.cuh"
#include "raw_offset.cuh"
#include "xeng_internal.h"

namespace xeng {
namespace {

// Samples per stage (a build parameter, 64 or 128): every stage carries a fixed
// cost in the pipeline (barrier round trips, a commit, the converters' fence),
// so fewer, larger stages run faster although the rings then hold two plane
// stages instead of four (measured on GB300, full Pathfinder rate: 64 samples
// 3.17 ms, 128 samples 2.99 ms).  The rings hold 208 KB (64) or 192 KB (128).
#ifndef XENG_SMALL_KC
#define XENG_SMALL_KC 128
#endif
constexpr int kSKc = XENG_SMALL_KC;         // samples per stage
static_assert(kSKc == 64 || kSKc == 128, "64 or 128 samples per stage");
constexpr int kSBox = kSKc * 128;           // one raw tile or plane tile: kSKc samples x 128 inputs
constexpr int kSRawBytes = 2 * kSBox;       // raw slot: tiles X and Y
constexpr int kSPlaneBytes = 4 * kSBox;     // plane stage: Im_X, Im_Y, Re_X, Re_Y
// Ring depths (build parameters; 4 x 32 KB + 5 x 16 KB fill the shared memory).
#ifndef XENG_SMALL_PLANE_STAGES
#define XENG_SMALL_PLANE_STAGES (4 * 64 / XENG_SMALL_KC)
#endif
#ifndef XENG_SMALL_RAW_SLOTS
#define XENG_SMALL_RAW_SLOTS (XENG_SMALL_KC == 128 ? 2 : 5)
#endif
constexpr int kSPlanes = XENG_SMALL_PLANE_STAGES, kSRaws = XENG_SMALL_RAW_SLOTS;

constexpr int kSConvWarp0 = 2, kSConvWarps = 8;
constexpr int kSEpiWarp0 = kSConvWarp0 + kSConvWarps, kSEpiWarps = 8;
constexpr int kSThreads = 32 * (kSEpiWarp0 + kSEpiWarps);
constexpr uint32_t kSTmemCols = 512;
constexpr int kSSumPar = sum_slot(256);  // entries per item parity
constexpr int kSSums = 2 * kSSumPar * 8;  // per item parity: (P, Q) of the item's 256 inputs (X tile, then Y tile; sum_slot)
// barriers: raw full and empty per slot, plane full and empty per stage; acc full,
// acc empty, drain; sums full and empty per parity
constexpr int kSBars = 2 * kSRaws + 2 * kSPlanes + 3 + 4;
constexpr size_t kSSmem =
    1024 + (size_t)kSPlanes * kSPlaneBytes + (size_t)kSRaws * kSRawBytes + kSSums + kSBars * 8 + 16;
static_assert(kSSmem <= 232448, "shared memory over the per-CTA limit");
constexpr int kSJoin = 14;  // CTAs an item at most for the converters to join its epilogue
constexpr int kSChunks = 2 * kSBox / 16 / (32 * kSConvWarps);  // 16-byte chunks per converter thread and stage
static_assert(kSChunks * 32 * kSConvWarps * 16 == 2 * kSBox, "the converter threads cover both tiles");
constexpr int kSWiden = 16 / kSChunks;  // stages between widenings of the byte-lane sums (<= 240)

// Instruction descriptor, kind::f8f6f4: D f32, A and B E4M3, both MN-major
// (bits 15, 16), N = n, M = 128; bit 13 negates A.
__host__ __device__ constexpr uint32_t small_idesc(int n, bool neg_a)
{
    return (1u << 4) | (neg_a ? (1u << 13) : 0u) | (1u << 15) | (1u << 16) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(128 >> 4) << 24);
}

// MN-major operand with a 128-byte swizzle: rows of 128 elements along M/N,
// 8-row groups along K 1 KB apart (stride byte offset), version 1.  The
// leading byte offset `lbo` is the step between 128-element atoms along M/N,
// where an N = 256 operand continues (one-atom operands ignore it).
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

struct SmallArgs {
    int64_t t0, nt;        // samples t0 .. t0 + nt - 1 of the block, nt <= kFusedMaxSamples
    int32_t F, N, f0, nf;  // channels f0 .. f0 + nf - 1
    int32_t n_items, n_k;  // items; stages (of kSKc samples) per item
    int32_t split;         // CTAs per item (>= 2: shared items), else kSmallEven or kSmallWhole
    int32_t quot, rest;    // the sequence's n_items * n_k stages (kSmallEven) or its items (kSmallWhole) over
                           // the grid: CTA b takes quot of them, one more if b < rest
    int32_t *acc;          // [nf][N(N+1)/2][2], channel f0 + fl at fl
    int accumulate;        // 0: store, 1: add
    int2 *ws;              // [grid][2][16][4][128][2] partial blocks: (block, 8-column chunk, column pair, row)
    int *flags;            // [grid]: this launch's epoch once the CTA's partial is in ws
    int *epoch;            // [0]: launches so far on these flags (this launch's epoch is [0] + 1);
                           // [1]: CTAs of this launch finished
    int *err;
    const CUtensorMap *maps;  // null: raw_map over one block; else a map per block of spb stages,
    int32_t spb;              // the launch's samples running through the blocks in order
    int32_t sub;              // != 0: the 128-input blocks b with slot[b] >= 0 come from sub_map,
    int32_t sub_f0;           // channel fl of the launch at its channel sub_f0 + fl
    int8_t slot[kMaxBlocks];
};

// A CTA's work: the stages [lo, hi) of the launch's sequence (item-major), as
// pieces (item, stages k0 .. k1 - 1).  How the sequence is cut (small_split):
//   kSmallEven  evenly.  A piece with k0 > 0 (only ever a CTA's first) adds its
//               partial block through ws; the CTA whose piece starts the item
//               (its owner) adds them into its own and stores.
//   kSmallWhole between items only: no partial blocks.
//   2 or more   `split` CTAs share each item, one piece each: all of them write
//               their partials of the chunks the others finish, and each adds up
//               and stores its share of the item's 8-column chunks.
struct Piece {
    int it, k0, k1;
};

__device__ __forceinline__ int range_lo(const SmallArgs &a, int b)
{
    if (a.split > kSmallWhole) return (b / a.split) * a.n_k + (b % a.split) * a.n_k / a.split;
    return (b * a.quot + min(b, a.rest)) * (a.split == kSmallWhole ? a.n_k : 1);
}

// kSmallEven: the CTA whose range holds stage x of the sequence.
__device__ __forceinline__ int stage_cta(const SmallArgs &a, int x)
{
    const int more = a.rest * (a.quot + 1);  // stages of the CTAs that take one more
    return x < more ? x / (a.quot + 1) : a.rest + (x - more) / a.quot;
}

__device__ __forceinline__ bool next_piece(const SmallArgs &a, int &x, int hi, Piece &p)
{
    if (x >= hi) return false;
    p.it = x / a.n_k;
    const int first = p.it * a.n_k;
    p.k0 = x - first;
    p.k1 = min(hi - first, a.n_k);
    x = first + p.k1;
    return true;
}

// Item `it`.  N > 128: per channel pair (2m, 2m + 1) the column item of 2m, the
// diagonal item of both, the column item of 2m + 1 (an odd last channel: its
// column item and a diagonal item of it alone).  N <= 128: diagonal items of channel
// pairs.  fy < 0: no second channel (its tile repeats the first; nothing stored).
struct SmallItem {
    bool col;
    int fx, fy;  // channels (local) of the X and Y tiles: inputs 0..127, but a column item's Y 128..255
};

__device__ __forceinline__ SmallItem small_item(const SmallArgs &a, int it)
{
    SmallItem w;
    if (a.N > 128) {
        const int m = it / 3, r = it - 3 * m;
        w.col = r != 1;
        if (w.col) {
            w.fx = w.fy = 2 * m + (r >> 1);
        } else {
            w.fx = 2 * m;
            w.fy = 2 * m + 1 < a.nf ? 2 * m + 1 : -1;
        }
    } else {
        w.col = false;
        w.fx = 2 * it;
        w.fy = 2 * it + 1 < a.nf ? 2 * it + 1 : -1;
    }
    return w;
}

// kAdd: add into acc (a.accumulate != 0) instead of storing; kShared: several
// CTAs per item (a.split >= 2); kJoin: there the converter warps take half of the
// epilogue (a.split <= kSJoin).  Templates so that each launch carries only its
// own epilogue (the adding one needs more registers).
template <bool kAdd, bool kShared, bool kJoin>
__global__ void __launch_bounds__(kSThreads, 1)
correlate_small_kernel(const __grid_constant__ CUtensorMap raw_map, const __grid_constant__ CUtensorMap diag_map,
                       const __grid_constant__ CUtensorMap sub_map, const __grid_constant__ SmallArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t sbase = (raw + 1023u) & ~1023u;
    uint8_t *sgen = smem_raw + (sbase - raw);
    // plane stages first, then the raw slots, the item sums and the barriers
    const uint32_t raw0 = sbase + kSPlanes * kSPlaneBytes;
    const uint32_t sums_u = raw0 + kSRaws * kSRawBytes;
    const uint32_t bars = sums_u + kSSums;
    int2 *sums = reinterpret_cast<int2 *>(sgen + (sums_u - sbase));  // [parity][sum_slot] (P, Q)
    float2 *terms = reinterpret_cast<float2 *>(sums);                // in their place: the epilogue's offset terms
    auto plane = [&](int s) { return sbase + (uint32_t)(s * kSPlaneBytes); };
    auto slot = [&](int s) { return raw0 + (uint32_t)(s * kSRawBytes); };
    auto rawf = [&](int s) { return bars + 8u * s; };
    auto rawe = [&](int s) { return bars + 8u * (kSRaws + s); };
    auto full = [&](int s) { return bars + 8u * (2 * kSRaws + s); };
    auto empty = [&](int s) { return bars + 8u * (2 * kSRaws + kSPlanes + s); };
    const uint32_t accf = bars + 8u * (2 * kSRaws + 2 * kSPlanes);
    const uint32_t acce = accf + 8u;
    const uint32_t drain = accf + 16u;
    auto sums_full = [&](int par) { return accf + 24u + 8u * par; };
    auto sums_empty = [&](int par) { return accf + 40u + 8u * par; };
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(smem_raw + (bars + 8u * kSBars - raw));
    // this launch's flag value, read once at the start: the last CTA of the launch
    // to finish advances the count (at the end), after every CTA has read it here
    int *s_epoch = reinterpret_cast<int *>(tmem_slot + 1);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int *err = a.err;
    const int lo = range_lo(a, (int)blockIdx.x), hi = range_lo(a, (int)blockIdx.x + 1);

    if (threadIdx.x == 0) {
        for (int s = 0; s < kSRaws; s++) {
            mbar_init(rawf(s), 1);
            mbar_init(rawe(s), kSConvWarps);  // one arrival per converter warp
        }
        for (int s = 0; s < kSPlanes; s++) {
            mbar_init(full(s), kSConvWarps);
            mbar_init(empty(s), 1);
        }
        mbar_init(accf, 1);
        mbar_init(acce, kSEpiWarps);
        mbar_init(drain, 1);
        for (int par = 0; par < 2; par++) {
            mbar_init(sums_full(par), kSConvWarps);
            mbar_init(sums_empty(par), kSEpiWarps);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(&raw_map) : "memory");
        *s_epoch = *(volatile int *)a.epoch + 1;
    }
    for (int k = threadIdx.x; k < 2 * kSSumPar; k += kSThreads) sums[k] = make_int2(0, 0);
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(kSTmemCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;

    bool conv_ok = true;  // a converter's
    auto epilogue = [&]() {
        constexpr int warp0 = kJoin ? kSConvWarp0 : kSEpiWarp0;
        constexpr int tail = 32 * (kSEpiWarp0 + kSEpiWarps - warp0);  // its threads
        const int q = warp & 3;                     // TMEM lane quadrant this warp may access
        const int et = (int)threadIdx.x - 32 * warp0;
        const int h = kJoin ? et >> 7 & 1 : et >> 7;  // the item's block: columns 128h.. of Re and Im
        constexpr int halves = kJoin ? 2 : 1;       // warps a quadrant and block
        const int half = kJoin ? et >> 8 : 0;
        const int row = q * 32 + lane;              // TMEM lane: input j within its 128-input block
        const int N = a.N;                          // <= 256
        const int nt = (int)a.nt;
        const int64_t nb = (int64_t)N * (N + 1) / 2;
        const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16);
        // partial blocks in ws: [CTA][block h][chunk c / 8][column pair][row], 16 bytes each,
        // so that a warp's 32 rows are one 512-byte run
        constexpr int kWs = 2 * 16 * 4 * 128;    // 16-byte words per CTA
        const int wsi = h * 16 * 4 * 128 + row;  // + (c / 8) * 512 + 128 per column pair
        int4 *const ws = reinterpret_cast<int4 *>(a.ws);
        uint32_t uses = 0;
        int local = 0;
        int x = lo;
        Piece pc;
        while (next_piece(a, x, hi, pc)) {
            const SmallItem w = small_item(a, pc.it);
            const int par = local & 1;
            // the piece's samples inside the launch: 64 n from each of the two products
            const float n128 = (float)(128 * ((pc.k1 * kSKc < nt ? pc.k1 * kSKc : nt) - pc.k0 * kSKc));
            const bool owner = pc.k0 == 0;
            // an owner whose item runs on: the CTAs after it that hold the rest
            // (shared items: the item's other CTAs, which this one meets later)
            const int c_lo = kShared ? pc.it * a.split : (int)blockIdx.x + 1;
            const int c_hi = kShared ? c_lo + a.split - 1
                                    : owner && pc.k1 < a.n_k ? stage_cta(a, (pc.it + 1) * a.n_k - 1) : 0;
            // Block h: column items' inputs j = 128.. against i = 128h..; diagonal items'
            // channel fx or fy, both 0..127.  Sums: X tile at 0, Y tile at 128.
            const int fl = w.col ? w.fx : (h ? w.fy : w.fx);
            const int j_warp = (w.col ? 128 : 0) + q * 32;
            const int j = j_warp + lane;
            const int i_base = w.col ? 128 * h : 0;
            const bool lane_ok = j < N;
            const bool warp_ok = fl >= 0 && j_warp < N;
            int2 *out = reinterpret_cast<int2 *>(a.acc) + (int64_t)fl * nb;
            // warp-uniform: columns inside the channel and up to some lane's diagonal
            auto chunk_ok = [&](const int c) { return c < 128 && i_base + c < N && i_base + c <= j_warp + 31; };
            // the triangle's values of columns c .. c + 7 (adding launches): pair (i, j) sits
            // at i*N - i*(i-1)/2 + (j - i) in the channel's triangle and row i + 1 starts
            // N - i - 1 pairs after row i, so per column the warp's 32 consecutive inputs j
            // are one 256-byte run
            auto load_old = [&](const int c, int2 (&o)[8]) {
                const int i0 = i_base + c;
                const int last = lane_ok ? min(j - i0, N - 1 - i0) : -1;
                int off = i0 * N - i0 * (i0 - 1) / 2 - i0 + j;
                #pragma unroll
                for (int e = 0; e < 8; e++) {
                    if (e <= last) o[e] = __ldcg(out + off);
                    off += N - (i0 + e) - 1;
                }
            };
            int2 old[8];
            if (kAdd && !kShared) {
                int nx = x;
                Piece np;
                if (next_piece(a, nx, hi, np)) {  // the next item's values, to L2
                    const SmallItem nw = small_item(a, np.it);
                    const int nfl = nw.col ? nw.fx : (h ? nw.fy : nw.fx);
                    if (nfl >= 0 && np.k0 == 0)
                        prefetch_triangle(reinterpret_cast<const int2 *>(a.acc) + (int64_t)nfl * nb, N,
                                          (nw.col ? 128 : 0) + q * 32, nw.col ? 128 * h : 0,
                                          min(N, nw.col ? 128 * h + 128 : 128), 8, lane);
                }
                if (owner && warp_ok && chunk_ok(0)) load_old(0, old);  // under the wait for the accumulator
            }
            bool ok = (!kJoin || conv_ok) && mbar_wait_backoff(accf, uses & 1u, err, kDevTimeoutEpilogue, 128);
            ok = ok && mbar_wait_backoff(sums_full(par), (uint32_t)((local >> 1) & 1), err, kDevTimeoutEpilogue, 128);
            if (et == 0 && !kShared)
                for (int b = c_lo; ok && b <= c_hi; b++) ok = flag_wait(a.flags + b, *s_epoch, err, kDevTimeoutEpilogue);
            // the barrier ORs the warps' failures, so they leave together
            if (bar_any(2, tail, !ok)) break;
            ++uses;
            fence_after();
            // every input's offset terms in place of its sums (read by all the warps)
            if (!kJoin || et < 256) {
                const int m = par * kSSumPar + sum_slot(et);
                terms[m] = offset_terms(sums[m]);
            }
            named_bar_sync(2, tail);
            const float2 *ci = terms + par * kSSumPar + sum_slot(128 * h);  // inputs i of the columns
            const float2 tj = terms[par * kSSumPar + sum_slot((w.col ? 128 : 128 * h) + row)];
            const float re_j = kFloatToInt + n128 + tj.x, im_j = kFloatToInt - tj.y;
            // TMEM columns of the block: column items Re at 128h.., Im at 256 + 128h..;
            // diagonal items Re at 256h.., Im (negated) at 256h + 128..
            const uint32_t tre = taddr + (w.col ? 128u * h : 256u * h);
            const uint32_t tim = tre + (w.col ? 256u : 128u);
            const float im_scale = w.col ? kRawScale : -kRawScale;
            // the piece's visibilities in place of the accumulator words of columns c .. c + 7
            auto correct = [&](const int c, uint32_t (&vre)[8], uint32_t (&vim)[8]) {
                #pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    const float4 t2 = *reinterpret_cast<const float4 *>(ci + sum_slot(c) + e);  // the same for every lane: a broadcast
                    vre[e] = raw_to_int(vre[e], kRawScale, re_j + t2.x);
                    vim[e] = raw_to_int(vim[e], im_scale, im_j + t2.y);
                    vre[e + 1] = raw_to_int(vre[e + 1], kRawScale, re_j + t2.z);
                    vim[e + 1] = raw_to_int(vim[e + 1], im_scale, im_j + t2.w);
                }
            };
            auto put_partial = [&](const int c, const uint32_t (&vre)[8], const uint32_t (&vim)[8]) {
                int4 *d = ws + (int64_t)blockIdx.x * kWs + wsi + (c >> 3) * 512;
                #pragma unroll
                for (int e = 0; e < 8; e += 2)
                    __stcg(d + e * 64, make_int4((int)vre[e], (int)vim[e], (int)vre[e + 1], (int)vim[e + 1]));
            };
            auto add_partial = [&](const int b, const int c, uint32_t (&vre)[8], uint32_t (&vim)[8]) {
                const int4 *src = ws + (int64_t)b * kWs + wsi + (c >> 3) * 512;
                #pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    const int4 v = __ldcg(src + e * 64);
                    vre[e] += (uint32_t)v.x;
                    vim[e] += (uint32_t)v.y;
                    vre[e + 1] += (uint32_t)v.z;
                    vim[e + 1] += (uint32_t)v.w;
                }
            };
            // Stores columns c .. c + 7, or adds them to the values in `old`.
            auto put_chunk = [&](const int c, const uint32_t (&vre)[8], const uint32_t (&vim)[8]) {
                const int i0 = i_base + c;
                const int last = lane_ok ? min(j - i0, N - 1 - i0) : -1;  // elements e <= last are pairs of the triangle
                int off = i0 * N - i0 * (i0 - 1) / 2 - i0 + j;
                #pragma unroll
                for (int e = 0; e < 8; e++) {
                    if (e <= last)
                        __stcs(out + off, kAdd ? make_int2(old[e].x + (int)vre[e], old[e].y + (int)vim[e])
                                               : make_int2((int)vre[e], (int)vim[e]));
                    off += N - (i0 + e) - 1;
                }
            };
            // Calls fn(c, re, im) with the corrected values of the chunks c = c0, c0 + step, ...
            // Where registers allow, in two sets: the next chunk's TMEM loads run under this
            // chunk's stores.
            auto for_chunks = [&](const int c0, const int step, auto &&fn) {
                if (kAdd || kShared) {
                    // adding: the next chunk's old values are loaded under this chunk's TMEM
                    // loads and stores
                    for (int c = c0; warp_ok && chunk_ok(c); c += step) {
                        uint32_t vre[8], vim[8];
                        int2 next[8];
                        tmem_ld8(tre + c, vre);
                        tmem_ld8(tim + c, vim);
                        if (kAdd && !kShared && owner && chunk_ok(c + step)) load_old(c + step, next);
                        tmem_ld_wait();
                        correct(c, vre, vim);
                        fn(c, vre, vim);
                        if (kAdd && !kShared) {
                            #pragma unroll
                            for (int e = 0; e < 8; e++) old[e] = next[e];
                        }
                    }
                    return;
                }
                uint32_t ra[8], ia[8], rb[8], ib[8];
                int c = c0;
                if (!warp_ok || !chunk_ok(c)) return;
                tmem_ld8(tre + c, ra);
                tmem_ld8(tim + c, ia);
                tmem_ld_wait();
                for (;;) {
                    const int c1 = c + step;
                    const bool ok1 = chunk_ok(c1);
                    if (ok1) {
                        tmem_ld8(tre + c1, rb);
                        tmem_ld8(tim + c1, ib);
                    }
                    correct(c, ra, ia);
                    fn(c, ra, ia);
                    if (!ok1) break;
                    tmem_ld_wait();
                    c = c1 + step;
                    const bool ok2 = chunk_ok(c);
                    if (ok2) {
                        tmem_ld8(tre + c, ra);
                        tmem_ld8(tim + c, ia);
                    }
                    correct(c1, rb, ib);
                    fn(c1, rb, ib);
                    if (!ok2) break;
                    tmem_ld_wait();
                }
            };
            if (kShared) {
                // chunk c of block h is finished by the item's CTA (16 h + c / 8) % split, its
                // chunks of a block by the halves in turn
                const int part = (int)blockIdx.x - c_lo;
                for_chunks(8 * half, 8 * halves, [&](const int c, const uint32_t (&vre)[8], const uint32_t (&vim)[8]) {
                    if (lane_ok && (16 * h + (c >> 3)) % a.split != part) put_partial(c, vre, vim);
                });
                __threadfence();  // the partials are visible at GPU scope before the flag below
                named_bar_sync(2, tail);
                if (et == 0) st_release_gpu(a.flags + blockIdx.x, *s_epoch);
                ok = et >= a.split || flag_wait(a.flags + c_lo + et, *s_epoch, err, kDevTimeoutEpilogue);
                if (bar_any(2, tail, !ok)) break;
                const int first = (part + a.split - 16 * h % a.split) % a.split;  // 16 h + first = part (mod split)
                for_chunks(8 * (first + half * a.split), 8 * halves * a.split, [&](const int c, uint32_t (&vre)[8], uint32_t (&vim)[8]) {
                    if (!lane_ok) return;
                    if (kAdd) load_old(c, old);
                    #pragma unroll 4
                    for (int p = 1; p < a.split; p++)
                        add_partial(c_lo + (part + p < a.split ? part + p : part + p - a.split), c, vre, vim);
                    put_chunk(c, vre, vim);
                });
            } else {
                for_chunks(0, 8, [&](const int c, uint32_t (&vre)[8], uint32_t (&vim)[8]) {
                    if (!owner) {  // a later piece of the item: the partial goes to this CTA's slot
                        if (lane_ok) put_partial(c, vre, vim);
                        return;
                    }
                    // the item's later pieces (none for a whole item)
                    for (int b = c_lo; lane_ok && b <= c_hi; b++) add_partial(b, c, vre, vim);
                    put_chunk(c, vre, vim);
                });
            }
            if (!owner && !kShared) __threadfence();  // the partial is visible at GPU scope before the flag below
            // every epilogue thread is done with this parity's sums: clear them for
            // the piece after next, then hand TMEM and the buffer back
            named_bar_sync(2, tail);
            if (!owner && !kShared && et == 0) st_release_gpu(a.flags + blockIdx.x, *s_epoch);
            for (int k = et; k < kSSumPar; k += tail) sums[par * kSSumPar + k] = make_int2(0, 0);
            fence_before();
            __syncwarp();
            if (lane == 0 && warp >= kSEpiWarp0) {
                mbar_arrive(acce);
                mbar_arrive(sums_empty(par));
            }
            ++local;
        }
    };
    if (warp == 0) {
        {
            // ---------------- TMA producer (the whole warp, one elected lane issuing) ----------------
            int s = 0, issued = 0;
            uint32_t ph = 0;
            bool ok = true;
            int x = lo;
            Piece pc;
            while (ok && next_piece(a, x, hi, pc)) {
                const SmallItem w = small_item(a, pc.it);
                const int fX = a.f0 + w.fx, fY = a.f0 + (w.fy >= 0 ? w.fy : w.fx);
                // where each tile's block is: map, input, channel, sample (block 0 of channel fx,
                // and block 0 or 1 of fy; a substituted block's in sub_map, whose
                // samples are the launch's)
                const int sX = a.sub ? a.slot[0] : -1, sY = a.sub ? a.slot[w.col ? 1 : 0] : -1;
                const CUtensorMap *own = w.col ? &raw_map : &diag_map;
                const CUtensorMap *mX = sX >= 0 ? &sub_map : own, *mY = sY >= 0 ? &sub_map : own;
                const int xX = sX >= 0 ? 128 * sX : 0, xY = sY >= 0 ? 128 * sY : w.col ? 128 : 0;
                const int cX = sX >= 0 ? a.sub_f0 + fX - a.f0 : fX, cY = sY >= 0 ? a.sub_f0 + fY - a.f0 : fY;
                int zX = (sX >= 0 ? 0 : (int)a.t0) + pc.k0 * kSKc, zY = (sY >= 0 ? 0 : (int)a.t0) + pc.k0 * kSKc;
                for (int kc = pc.k0; kc < pc.k1; kc++) {
                    ok = __all_sync(0xffffffffu, mbar_try_wait(rawe(s), ph ^ 1u) ||
                                                     mbar_wait(rawe(s), ph ^ 1u, err, kDevTimeoutProducer));
                    if (!ok) break;
                    if (a.maps) {  // blocks of spb stages, each with its own map
                        mX = mY = a.maps + kc / a.spb;
                        zX = zY = (kc % a.spb) * kSKc;
                    }
                    if (elect_one()) {
                        mbar_expect_tx(rawf(s), kSRawBytes);
                        tma_load_3d(slot(s), mX, xX, cX, zX, rawf(s));
                        tma_load_3d(slot(s) + kSBox, mY, xY, cY, zY, rawf(s));
                    }
                    zX += kSKc;
                    zY += kSKc;
                    ++issued;
                    if (++s == kSRaws) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
            }
            if (!ok) {
                // Let the copies already issued land before the CTA can exit.
                for (int k = 1; k <= kSRaws && k <= issued; k++) {
                    int sk = s - k, p = (int)ph;
                    if (sk < 0) { sk += kSRaws; p ^= 1; }
                    (void)mbar_wait(rawf(sk), (uint32_t)p, err, kDevTimeoutProducer);
                }
            }
        }
    } else if (warp == 1) {
        {
            // ---------------- MMA issuer (the whole warp, one elected lane issuing) ----------------
            int s = 0;
            uint32_t ph = 0, uses = 0;
            bool ok = true;
            int x = lo;
            Piece pc;
            while (ok && next_piece(a, x, hi, pc)) {
                const SmallItem w = small_item(a, pc.it);
                if (!__all_sync(0xffffffffu, mbar_wait(acce, (uses & 1u) ^ 1u, err, kDevTimeoutMma))) break;
                ++uses;
                fence_after();
                for (int kc = pc.k0; kc < pc.k1; kc++) {
                    ok = __all_sync(0xffffffffu, mbar_try_wait(full(s), ph) ||
                                                     mbar_wait(full(s), ph, err, kDevTimeoutMma));
                    if (!ok) break;
                    fence_after();
                    const uint32_t st = plane(s);
                    if (elect_one()) {
                        if (w.col) {
                            // A = Y rows (TMEM lanes: inputs j), B = X and Y columns (inputs i; the
                            // Y plane kSBox after the X plane): Re in columns 0..255, Im in 256..511
                            const uint64_t dre = sdesc(st + 2 * kSBox, kSBox), dim = sdesc(st, kSBox);
                            const uint64_t are = sdesc(st + 3 * kSBox, kSBox), aim = sdesc(st + kSBox, kSBox);
                            #pragma unroll
                            for (int kk = 0; kk < kSKc / 32; kk++) {  // +32 samples = +4 KB = +256 in the address field
                                const uint32_t acc = (kc != pc.k0 || kk != 0) ? 1u : 0u;
                                const uint64_t k4 = 256u * kk;
                                mma_f8(tmem, are + k4, dre + k4, small_idesc(256, false), acc);
                                mma_f8(tmem, aim + k4, dim + k4, small_idesc(256, false), 1u);
                                mma_f8(tmem + 256u, are + k4, dim + k4, small_idesc(256, false), acc);
                                mma_f8(tmem + 256u, aim + k4, dre + k4, small_idesc(256, true), 1u);
                            }
                        } else {
                            // each tile against itself, in columns 256h..: one N = 256 MMA of
                            // A_im against [B_im | B_re] (Re_h 16 KB after Im_h) gives
                            // [Im Im^T | Im Re^T]; A_re B_re^T completes Re, and (-A_re) B_im^T
                            // makes the second half Im Re^T - Re Im^T, minus Im of x_i conj(x_j) with
                            // A = x_j.  (Four N = 128 MMAs per tile instead ran at about 72% of the
                            // tensor rate.)
                            #pragma unroll
                            for (int h = 0; h < 2; h++) {
                                const uint64_t dim = sdesc(st + h * kSBox, 2 * kSBox), dre = sdesc(st + (2 + h) * kSBox, 2 * kSBox);
                                const uint32_t d = tmem + 256u * h;
                                #pragma unroll
                                for (int kk = 0; kk < kSKc / 32; kk++) {
                                    const uint32_t acc = (kc != pc.k0 || kk != 0) ? 1u : 0u;
                                    const uint64_t k4 = 256u * kk;
                                    mma_f8(d, dim + k4, dim + k4, small_idesc(256, false), acc);
                                    mma_f8(d, dre + k4, dre + k4, small_idesc(128, false), 1u);
                                    mma_f8(d + 128u, dre + k4, dim + k4, small_idesc(128, true), 1u);
                                }
                            }
                        }
                        mma_commit(empty(s));
                    }
                    if (++s == kSPlanes) {
                        s = 0;
                        ph ^= 1u;
                    }
                }
                if (!ok) break;
                if (elect_one()) mma_commit(accf);
            }
            // Drain: every MMA issued above has finished once this completes.
            if (elect_one()) mma_commit(drain);
            (void)mbar_wait(drain, 0u, err, kDevTimeoutMma);
        }
    } else if (warp < kSEpiWarp0) {
        // ---------------- converters ----------------
        // Thread u (0..255) takes tile g = u / 128 and, in it, the 16-byte chunks
        // v + 128 k (v = u % 128, k < kSChunks): sample rows v / 8 + 16 k,
        // physical chunk v % 8 -- a quarter-warp covers one whole 128-byte row, so
        // the accesses are bank-conflict-free.  The rows' swizzle (chunk ^ row % 8)
        // is the same for all of them, so the thread always holds the same 16
        // inputs: logical chunk lc = (v % 8) ^ (v / 8 % 8).
        const int u = (warp - kSConvWarp0) * 32 + lane;
        const int g = u >> 7, v = u & 127;
        const int r0 = v >> 3, lc = (v & 7) ^ (r0 & 7);
        const uint32_t off0 = (uint32_t)(g * kSBox + v * 16);  // chunk k at off0 + 2048 k within a slot / plane pair
        const int nt = (int)a.nt;                               // <= kFusedMaxSamples
        int rs = 0, ps = 0, local = 0;
        uint32_t rph = 0, pph = 0;
        bool &ok = conv_ok;
        int x = lo;
        Piece pc;
        for (; ok && next_piece(a, x, hi, pc); ++local) {
            // nibble sums of the thread's 16 inputs: byte lanes over up to 16
            // samples (<= 240), then 16-bit lanes (<= 15 x 2048 samples)
            uint32_t pb[4] = {0, 0, 0, 0}, qb[4] = {0, 0, 0, 0};
            uint32_t P16[8] = {0, 0, 0, 0, 0, 0, 0, 0}, Q16[8] = {0, 0, 0, 0, 0, 0, 0, 0};
            auto widen = [&]() {
                #pragma unroll
                for (int w = 0; w < 4; w++) {
                    P16[2 * w] += pb[w] & 0x00FF00FFu;
                    P16[2 * w + 1] += (pb[w] >> 8) & 0x00FF00FFu;
                    Q16[2 * w] += qb[w] & 0x00FF00FFu;
                    Q16[2 * w + 1] += (qb[w] >> 8) & 0x00FF00FFu;
                    pb[w] = qb[w] = 0;
                }
            };
            for (int kc = pc.k0; kc < pc.k1; kc++) {
                ok = mbar_wait_backoff(rawf(rs), rph, err, kDevTimeoutProducer, XENG_CONV_SLEEP_NS);
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                const int rows_left = nt - kc * kSKc;  // samples of this stage inside the launch (may exceed kSKc)
                const uint8_t *src = sgen + (slot(rs) - sbase) + off0;
                uint4 x[kSChunks];
                #pragma unroll
                for (int k = 0; k < kSChunks; k++) {
                    x[k] = *reinterpret_cast<const uint4 *>(src + 2048 * k);
                    if (r0 + 16 * k >= rows_left) x[k] = make_uint4(0, 0, 0, 0);  // past the launch: adds nothing
                }
                // The raw slot goes back to the producer with the plane stage below, once
                // the plane stores (which consume the loaded words) are done.  An arrival
                // right after the loads, with nothing waiting for their data, let the TMA
                // refill the slot under loads still in flight (measured on GB300: whole
                // items wrong in about one launch in two when the MMAs stalled behind a
                // long epilogue); one whose address depended on the loaded words was
                // exact but 1% slower than this.
                const int rcur = rs;
                if (++rs == kSRaws) {
                    rs = 0;
                    rph ^= 1u;
                }
                ok = mbar_wait_backoff(empty(ps), pph ^ 1u, err, kDevTimeoutProducer, XENG_CONV_SLEEP_NS);
                if (!__all_sync(0xffffffffu, ok)) {
                    ok = false;
                    break;
                }
                uint8_t *dim = sgen + (plane(ps) - sbase) + off0;  // Im_X / Im_Y
                uint8_t *dre = dim + 2 * kSBox;                    // Re_X / Re_Y
                #pragma unroll
                for (int k = 0; k < kSChunks; k++) {
                    uint4 re, im;
                    re.x = (x[k].x >> 4) & 0x0F0F0F0Fu;
                    re.y = (x[k].y >> 4) & 0x0F0F0F0Fu;
                    re.z = (x[k].z >> 4) & 0x0F0F0F0Fu;
                    re.w = (x[k].w >> 4) & 0x0F0F0F0Fu;
                    im.x = x[k].x & 0x0F0F0F0Fu;
                    im.y = x[k].y & 0x0F0F0F0Fu;
                    im.z = x[k].z & 0x0F0F0F0Fu;
                    im.w = x[k].w & 0x0F0F0F0Fu;
                    *reinterpret_cast<uint4 *>(dre + 2048 * k) = re;
                    *reinterpret_cast<uint4 *>(dim + 2048 * k) = im;
                    pb[0] += re.x; pb[1] += re.y; pb[2] += re.z; pb[3] += re.w;
                    qb[0] += im.x; qb[1] += im.y; qb[2] += im.z; qb[3] += im.w;
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // planes visible to the MMAs
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(full(ps));
                    mbar_arrive(rawe(rcur));
                }
                if (++ps == kSPlanes) {
                    ps = 0;
                    pph ^= 1u;
                }
                if ((kc - pc.k0 + 1) % kSWiden == 0) widen();
            }
            if (!ok) break;
            widen();
            // the four lanes of a warp holding the same inputs (rows differing in
            // their two low bits: lanes ^ 9, ^ 18) add up -- two in 16-bit lanes
            // (<= 2 x 15 x 2048), the other two in 32 bits -- then one of them adds
            // the warp's totals into the item's sums; input 4w + b is byte b of word w
            uint32_t P32[16], Q32[16];
            #pragma unroll
            for (int k = 0; k < 8; k++) {
                P16[k] += __shfl_xor_sync(0xffffffffu, P16[k], 9);
                Q16[k] += __shfl_xor_sync(0xffffffffu, Q16[k], 9);
            }
            #pragma unroll
            for (int m = 0; m < 16; m++) {
                const int w = m >> 2, b = m & 3;
                P32[m] = (P16[2 * w + (b & 1)] >> (16 * (b >> 1))) & 0xFFFFu;
                Q32[m] = (Q16[2 * w + (b & 1)] >> (16 * (b >> 1))) & 0xFFFFu;
                P32[m] += __shfl_xor_sync(0xffffffffu, P32[m], 18);
                Q32[m] += __shfl_xor_sync(0xffffffffu, Q32[m], 18);
            }
            const int par = local & 1;
            // the buffer was last read (and cleared) by the epilogue two items ago
            ok = mbar_wait_backoff(sums_empty(par), (uint32_t)((local >> 1) & 1) ^ 1u, err, kDevTimeoutProducer,
                                   XENG_CONV_SLEEP_NS);
            if (!__all_sync(0xffffffffu, ok)) {
                ok = false;
                break;
            }
            if ((r0 & 3) == 0) {
                int *sp = reinterpret_cast<int *>(sums + par * kSSumPar + sum_slot(g * 128 + lc * 16));
                #pragma unroll
                for (int m = 0; m < 16; m++) {
                    atomicAdd(sp + 2 * m, (int)P32[m]);
                    atomicAdd(sp + 2 * m + 1, (int)Q32[m]);
                }
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(sums_full(par));
        }
    } else if (!kJoin) {
        epilogue();
    }
    if (kJoin && warp >= kSConvWarp0) epilogue();

    __syncwarp();
    fence_before();
    __syncthreads();
    fence_after();
    if (warp == 1) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kSTmemCols));
    }
    // One launch more on these flags: the last CTA to get here (every CTA read the
    // epoch when it started, before getting here) advances the count and resets
    // the arrivals, so the next launch -- or the next replay of a captured one --
    // takes a fresh epoch.  Epochs run 1 .. 2^31 - 1, never 0 (an unset flag).
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(a.epoch + 1, 1) == (int)gridDim.x - 1) {
            const int e = *(volatile int *)a.epoch;
            a.epoch[1] = 0;
            a.epoch[0] = e >= 0x7FFFFFFE ? 0 : e + 1;
            __threadfence();
        }
    }
}

}  // namespace

bool small_ok(const uint8_t *block, int32_t N, int32_t pitch)
{
    return N >= 1 && N <= 256 && (pitch ? pitch : N) % 16 == 0 && (reinterpret_cast<uintptr_t>(block) & 15) == 0;
}

size_t small_ws_bytes(int num_sms) { return (size_t)num_sms * 2 * 16 * 128 * 8 * sizeof(int2); }
size_t small_flags_bytes(int num_sms) { return (size_t)(num_sms + 2) * sizeof(int); }

int small_stage_samples() { return kSKc; }

cudaError_t launch_correlate_small(const uint8_t *block, int64_t T_block, int64_t t0, int64_t nt, int32_t F, int32_t N,
                                   int32_t f0, int32_t nf, int32_t *acc, int accumulate, int2 *ws, int *flags,
                                   int *err, int num_sms, cudaStream_t s,
                                   const CUtensorMap *maps, int32_t spb,
                                   int32_t pitch, const SubBlocks *sub, int max_ctas)
{
    if (nf <= 0 || nt <= 0) return cudaSuccess;
    if (!small_ok(maps ? nullptr : block, N, pitch) || (sub && maps) || (maps && (spb < 1 || t0 != 0)) || nt > kFusedMaxSamples ||
        t0 < 0 || t0 + nt > T_block || T_block > 2147483647LL ||
        f0 < 0 || f0 + nf > F || num_sms < 1 || (reinterpret_cast<uintptr_t>(acc) & 7) != 0 || !ws || !flags)
        return cudaErrorInvalidValue;
    const int64_t n_items = N > 128 ? (int64_t)nf + (nf + 1) / 2 : (int64_t)(nf + 1) / 2;
    const int n_k = (int)((nt + kSKc - 1) / kSKc);
    if (n_items * n_k > 2147483647LL && sub) return cudaErrorInvalidValue;
    if (n_items * n_k > 2147483647LL) {  // stages are counted in 32 bits
        const int32_t half = nf / 4 * 2;
        const cudaError_t e = launch_correlate_small(block, T_block, t0, nt, F, N, f0, half, acc, accumulate, ws, flags,
                                                     err, num_sms, s, maps, spb, pitch, nullptr, max_ctas);
        if (e != cudaSuccess) return e;
        return launch_correlate_small(block, T_block, t0, nt, F, N, f0 + half, nf - half,
                                      acc + (int64_t)half * N * (N + 1), accumulate, ws, flags, err, num_sms, s, maps,
                                      spb, pitch, nullptr, max_ctas);
    }
    CUtensorMap map, diag_map, sub_map;
    memset(&map, 0, sizeof map);  // not read with `maps`: the stages take the blocks' maps
    memset(&diag_map, 0, sizeof diag_map);
    memset(&sub_map, 0, sizeof sub_map);
    if (!maps) {
        cudaError_t e0 = encode_raw_map(&map, block, T_block, F, N, pitch, kSKc);
        // Above 128 inputs a diagonal item reads a channel's first 128 only: fetching
        // 256 bytes there brings in the rest for nothing (GB300, full Pathfinder band,
        // whose time the board's power sets: 3.25 ms, 3.15 without).
        if (e0 == cudaSuccess) e0 = encode_raw_map(&diag_map, block, T_block, F, N, pitch, kSKc, N <= 128);
        if (e0 != cudaSuccess) return e0;
    }
    if (sub) {
        cudaError_t e0 = encode_raw_map(&sub_map, sub->packed, nt, sub->F, 128 * sub->n, 0, kSKc);
        if (e0 != cudaSuccess) return e0;
    }
    int32_t split = 0;
    const int grid = small_split(n_items, n_k, max_ctas > 0 && max_ctas < num_sms ? max_ctas : num_sms, &split);
    // Shared items: up to 14 CTAs an item the converters join the epilogue, their one piece
    // done: 4 and 12 an item gain, 16 and 32 lose (us, without / with: N = 256 x 8 channels x 4096
    // samples, 12 CTAs an item, 25.1 / 23.6, adding 30.3 / 26.3; 160 x 24 x 4096, 4 an item,
    // 29.2 / 26.0; 256 x 6 x 8192, 16 an item, 25.4 / 25.8; 64 x 1 x 32,768, 32, 27.2 / 28.5).
    auto kern = accumulate ? correlate_small_kernel<true, false, false> : correlate_small_kernel<false, false, false>;
    if (split > kSJoin)
        kern = accumulate ? correlate_small_kernel<true, true, false> : correlate_small_kernel<false, true, false>;
    else if (split >= 2)
        kern = accumulate ? correlate_small_kernel<true, true, true> : correlate_small_kernel<false, true, true>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSSmem);
    if (e != cudaSuccess) return e;
    SmallArgs a;
    a.t0 = t0;
    a.nt = nt;
    a.F = F;
    a.N = N;
    a.f0 = f0;
    a.nf = nf;
    a.n_items = (int32_t)n_items;
    a.n_k = n_k;
    a.acc = acc;
    a.accumulate = accumulate;
    a.ws = ws;
    a.flags = flags;
    a.epoch = flags + num_sms;
    a.err = err;
    a.maps = maps;
    a.spb = spb;
    a.sub = sub ? 1 : 0;
    a.sub_f0 = sub ? sub->f0 : 0;
    if (sub) memcpy(a.slot, sub->slot, sizeof a.slot);
    a.split = split;
    a.quot = (int32_t)((split == kSmallWhole ? n_items : n_items * n_k) / grid);
    a.rest = (int32_t)((split == kSmallWhole ? n_items : n_items * n_k) % grid);
    // the CTAs of a split item wait for each other's partials: a cooperative
    // launch has every CTA resident at once (or fails)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid, 1, 1);
    cfg.blockDim = dim3(kSThreads, 1, 1);
    cfg.dynamicSmemBytes = kSSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, map, diag_map, sub_map, a);
}

}  // namespace xeng
