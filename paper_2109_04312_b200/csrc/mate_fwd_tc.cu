// Tensor-core forward of multi-view attention (head formula and pattern of Section 3) for bf16,
// d = 64, on sm_100a.  One persistent, warp-specialised CTA per SM takes units (see FwdUnit), longest first, from
// a shared counter: 256 query rows of one (example, head) in the head's view
// order (Section 3.1: per-head traversal order) against the key tiles those rows may attend.
//
//   warps 0-3   softmax of half 0 (query rows 0..127 of the unit), one thread per row
//   warps 4-7   softmax of half 1 (rows 128..255)
//   warps 8, 9  issue the tcgen05.mma of half 0 / half 1 (one elected lane each)
//   warps 10,11 padding rows
//   warps 12-15 loaders: Q, K, V rows by view-order index (the gather of Section 3.1 fused into the loads) into 128-byte
//               swizzled shared memory, 16 bytes per lane and copy, 32 rows of every load per warp; K/V tiles whose rows lie
//               in place in the tensors by one bulk tensor copy each.  Either kind completes on the tile's barrier by
//               itself, so no warp waits for its copies in order to signal them.
//
// Per key tile and half:   S = Q K^T  (tcgen05.mma, M = 128, N <= 128, K = 64, accumulator in TMEM)
//                          P = exp2(S c - m), row sum
//                          O += P V   (tcgen05.mma, M = 128, N = 64, P read from TMEM; O stays there)
//
// The base m of a row.  The largest score of a row's first tile serves for the whole unit: powers of two
// cost no precision (P is bf16 with fp32's exponent range, O and the row sum are fp32), so a later score may
// exceed it by up to 2^60.  That is read off the row sum when the unit is done: a row whose sum has
// left [2^-100, 2^60] sends the unit through once more, with the running max of online softmax (`exact`).
// The common case therefore has no max, no rescaling and no wait between the scores and the exponentials.
//
// What bounds it: the exponentials (16 per clock and SM: 1024 clk per 128 x 128 half tile, against 512 clk
// of tensor pipe), as far as everything else hides behind them.
//   - A thread takes its whole row of S (128 columns) into registers in one go (setmaxnreg) and gives S
//     back at once, so the Q K^T of the half's next tile runs under all of this tile's arithmetic.
//   - On a scheduler one warp of each half shares the exponential unit.  Holding one half back, so that its loads
//     fall under the other's exponentials, is not worth its instructions: 37 heads of 8192 dense positions 840 us
//     with it against 845 without, table batches of 4 x 2048 to 2 x 4096 tokens 0.3 us slower with it.
//   - Two threads per row (four warps per scheduler) hide the latencies as well, but the control flow of twice
//     the warps takes more issue slots than that gains.
//   - The instruction cache is about 32 KB for all roles of the CTA; straight-line code that misses it issues
//     at a third of the rate, from L2 at a sixth.  Rarely taken paths are rolled, and
//     the padding rows' loop is not unrolled (it was 8 KB).  Exact units have the path of full tiles all the same: on large
//     scores 4 x 2048 tokens take 60.0 us with it and 72.6 without, 1 x 8192 99.7 and 121.8, others the same.
// Key tiles of range B are visited by a half only where they meet the segments of its rows, and inside
// a tile a warp evaluates only the 32-column chunks that meet the segments of its 32 rows.  The scatter
// back to the original token order is fused into the epilogue.
//
// The unit's record and what the softmax threads need of its rows (original position, key range) travel
// through shared memory with the unit's Q, so no role waits for global memory between two units.
#include <cuda.h>
#include <cuda_bf16.h>

#include "load_ring.h"
#include "mate_internal.h"
#include "sm100_ptx.cuh"
#include "tc_tiles.cuh"

namespace mate {

#ifdef MATE_TRACE
__device__ long long g_trace[kTraceCtas * 32];
#endif

namespace {

using namespace ptx;

constexpr int kSoftmaxWarps = 8;
constexpr int kMmaWarp = kSoftmaxWarps;   // one MMA-issuing warp per half
constexpr int kMmaWarps = 2;
constexpr int kPadWarp0 = kMmaWarp + kMmaWarps;
constexpr int kPadWarps = 2;
constexpr int kLoadWarp0 = kPadWarp0 + kPadWarps;
constexpr int kLoadWarps = 4;
static_assert(kTile == 32 * kLoadWarps, "a row of a tile per loader thread");
constexpr int kThreads = 32 * (kLoadWarp0 + kLoadWarps);
constexpr int kStages = 4;                   // K/V ring
using QRing = LoadRing<2>;
using KVRing = LoadRing<kStages>;
// registers per thread after the roles have split: 256 x 176 + 256 x 80 = 65,536 = the 512 x 128 the CTA is
// launched with
constexpr int kRegsSoftmax = 176, kRegsOther = 80;

constexpr int kSchedDepth = 4;
constexpr uint32_t kOffQ = 0;                                // [2 buffers][2 halves] x 16 KB
constexpr uint32_t kOffKV = 4 * kTileBytes;                  // [kStages] x (K 16 KB, V 16 KB)
constexpr uint32_t kOffMeta = kOffKV + kStages * 2 * kTileBytes;    // [2 buffers] x (perm, seg_lo, seg_hi) of 256 rows
constexpr uint32_t kOffStage = kOffMeta + 2 * 3 * kUnitRows * 4;    // [softmax warps] x 32 rows x 64 bytes
constexpr uint32_t kOffUnit = kOffStage + kSoftmaxWarps * 2048;     // [kSchedDepth] unit records
constexpr uint32_t kOffBar = kOffUnit + kSchedDepth * sizeof(FwdUnit);
constexpr uint32_t kSmemBytes = kOffBar + 512 + 1024;        // + slack for the 1024-byte alignment
static_assert(kSmemBytes <= 232448, "shared memory per CTA");
// tensor memory: S of half h at column 128 h; O at 256 + 64 h; P (bf16 pairs) at 384 + 64 h
constexpr uint32_t kTmemCols = 512;
constexpr uint32_t kTmemO = 256;
constexpr uint32_t kTmemP = 384;
constexpr float kRescale = 8.f;                              // exact units: log2 units before the base moves
constexpr float kSumMin = 0x1p-100f, kSumMax = 0x1p60f;      // row sums outside: the unit is done once more, exactly

// barrier slots (8 bytes each) behind kOffBar
enum {
    kBarQFull = 0,                     // [2] loaders -> MMA, softmax   (count kLoadWarps)
    kBarQEmpty = kBarQFull + 2,        // [2] MMA commits and softmax warps (row data read) -> loaders (count kMmaWarps + kSoftmaxWarps)
    kBarKVFull = kBarQEmpty + 2,       // [kStages] loaders -> MMA      (count kLoadWarps)
    kBarKVEmpty = kBarKVFull + kStages,  // [kStages] MMA -> loaders    (count 2: one per half)
    kBarSFull = kBarKVEmpty + kStages,   // [2] MMA commit -> softmax (count 1)
    kBarSFree = kBarSFull + 2,         // [2] softmax -> MMA: S of a tile has been read (count 4: one per warp)
    kBarPFull = kBarSFree + 2,         // [2] softmax -> MMA        (count 4: one per warp)
    kBarPVDone = kBarPFull + 2,        // [2] MMA commit -> softmax: the P V of a tile is complete (count 1)
    kBarFinal = kBarPVDone + 2,        // [2]
    kBarSchedFull = kBarFinal + 2,                 // [kSchedDepth] scheduler -> every warp that follows the unit list (count 1)
    kBarSchedEmpty = kBarSchedFull + kSchedDepth,  // [kSchedDepth] those warps -> scheduler (count kSchedReaders)
    kNumBars = kBarSchedEmpty + kSchedDepth
};
static_assert(8 * kNumBars + 16 + 4 * kSchedDepth <= 512, "the barriers and the words behind them");
constexpr int kSchedReaders = kSoftmaxWarps + kMmaWarps + kLoadWarps;

// kMany: the three passes of a row-or-column plan.  (An instance of its own: the look-ups by pass cost the others up to 1 %,
// 4 x 2048 tokens 94.4 -> 95.3 us forward and backward.)
template <bool kMany>
struct Params {
    static constexpr int kV = kMany ? kViews : 2, kO = kMany ? kPasses : 1;
    __device__ static __forceinline__ int pass(int view) { return kMany ? pass_of(view) : 0; }
    // 2-D tensor maps over K and V seen as [B H N rows, 64 columns]: boxes of 128 rows, 128-byte swizzle
    CUtensorMap tmK, tmV;
    int bulk;        // 0: every tile is gathered row by row (the maps may be missing)
    int view_order;  // 1: Q, K, V, O and LSE are laid out in each head's own order (no gather, no scatter)
    const __nv_bfloat16 *Q, *K, *V;
    __nv_bfloat16 *O[kO];
    float *LSE[kO];
    ViewPlan view[kV];
    const FwdUnit *units;      // longest first
    int n_units;
    const PadChunk *pads;      // padding rows, which no unit covers
    int n_pads;
    int N, H;
    TensorRows tr;     // where (example, head) starts in the tensors
    float scale_log2;  // scale * log2(e)
    int32_t *status;
    int32_t *counters;  // [0] next unit, from kSchedWords on arrivals at the split units, 8 per unit
    uint8_t *ws;
};

// A chunk is 32 scores of one row (tile-local columns cb .. cb + 31).  A column c counts for the row
// iff c < pre or r_lo <= c < r_hi; the scores of the other columns are replaced by -inf, which the row max
// ignores and the exponential turns into an exact 0 (the scale is positive).
__device__ __forceinline__ uint32_t bits_below(int n) { return n <= 0 ? 0u : n >= 32 ? 0xffffffffu : (1u << n) - 1u; }
__device__ __forceinline__ void chunk_mask(uint32_t (&v)[32], int cb, int pre, int r_lo, int r_hi) {
    const uint32_t on = bits_below(pre - cb) | (bits_below(r_hi - cb) & ~bits_below(r_lo - cb));
#pragma unroll
    for (int e = 0; e < 32; ++e)
        if (!(on & (1u << e))) v[e] = 0xff800000u;
}
// Row max over one chunk, four partial maxima.
__device__ __forceinline__ void chunk_max(const uint32_t (&v)[32], float (&tm)[4]) {
#pragma unroll
    for (int e = 0; e < 32; e += 8) {
        tm[0] = fmax3(tm[0], __uint_as_float(v[e]), __uint_as_float(v[e + 1]));
        tm[1] = fmax3(tm[1], __uint_as_float(v[e + 2]), __uint_as_float(v[e + 3]));
        tm[2] = fmax3(tm[2], __uint_as_float(v[e + 4]), __uint_as_float(v[e + 5]));
        tm[3] = fmax3(tm[3], __uint_as_float(v[e + 6]), __uint_as_float(v[e + 7]));
    }
}
// P of one chunk: exp2(s * scale_log2 + neg_m), packed as bf16 pairs (even column in the low half); the row
// sums go to two packed pairs of partial sums.  The multiply-adds and the sums work on two columns per
// instruction (packed fp32 pairs); only the exponential is per column.
__device__ __forceinline__ void chunk_exp(const uint32_t (&v)[32], uint64_t scale2, uint64_t neg_m2, uint32_t (&packed)[16],
                                          uint64_t &l01, uint64_t &l23) {
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
        float x0, x1, x2, x3;
        unpack_f32x2(fma_f32x2(pack_f32x2(v[e], v[e + 1]), scale2, neg_m2), x0, x1);
        unpack_f32x2(fma_f32x2(pack_f32x2(v[e + 2], v[e + 3]), scale2, neg_m2), x2, x3);
        const float p0 = ex2(x0), p1 = ex2(x1), p2 = ex2(x2), p3 = ex2(x3);
        l01 = add_f32x2(l01, pack_f32x2(p0, p1));
        l23 = add_f32x2(l23, pack_f32x2(p2, p3));
        packed[e >> 1] = cvt_bf16x2(p0, p1);
        packed[(e >> 1) + 1] = cvt_bf16x2(p2, p3);
    }
}
__device__ __forceinline__ float sum_f32x2(uint64_t a, uint64_t b) {
    float a0, a1, b0, b1;
    unpack_f32x2(a, a0, a1);
    unpack_f32x2(b, b0, b1);
    return (a0 + a1) + (b0 + b1);
}

template <bool kMany>
__global__ void __launch_bounds__(kThreads, 1) tc_fwd_kernel(const __grid_constant__ Params<kMany> p) {
    launch_dependents();
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (base - raw);
    const uint32_t bars = base + kOffBar;
    volatile uint32_t *tmem_slot = (volatile uint32_t *)(sm + kOffBar + 8 * kNumBars);
    volatile int *s_abort = (volatile int *)(sm + kOffBar + 8 * kNumBars + 4);
    volatile uint32_t *s_bad = (volatile uint32_t *)(sm + kOffBar + 8 * kNumBars + 16);  // [kSchedDepth] warps that need the unit once more
    FwdUnit *s_unit = reinterpret_cast<FwdUnit *>(sm + kOffUnit);  // [kSchedDepth]; rows = 0 marks the end of the list

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = tid & 31;

    // The first loader warp hands out the units; its lanes 0-3 hold the record of the next one.  The first unit of
    // a CTA is its own index, later ones come from the shared counter, each claimed under the last tiles of the unit
    // before it.  Every CTA's last claim fails, so the claims of a
    // launch number n_units: the one that draws the last number puts the counter back to zero for the next launch.
    int4 rec = make_int4(0, 0, 0, 0);
    int u_next = blockIdx.x;  // lane 0
    auto claim = [&]() {
        if (lane == 0) u_next = atomicAdd(p.counters, 1);
    };
    auto fetch_record = [&](bool claimed) {
        if (claimed && lane == 0) {
            if (u_next == p.n_units - 1) *p.counters = 0;
            u_next += (int)gridDim.x;
        }
        const int u = __shfl_sync(0xffffffffu, u_next, 0);
        rec = make_int4(0, 0, 0, 0);  // rows = 0: the list is exhausted
        if (u < p.n_units && lane < 4) rec = __ldg(reinterpret_cast<const int4 *>(p.units + u) + lane);
    };
    if (warp == kLoadWarp0 + 1 && lane < 2) prefetch_tmap(&p.tmK + lane, p.bulk);  // both of them
    if (warp == kLoadWarp0) fetch_record(false);  // requested before the set-up below, which takes as long

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(bars + 8 * (kBarQFull + i), kLoadWarps);
            mbar_init(bars + 8 * (kBarQEmpty + i), kMmaWarps + kSoftmaxWarps);
            mbar_init(bars + 8 * (kBarSFull + i), 1);
            mbar_init(bars + 8 * (kBarSFree + i), kSoftmaxWarps / 2);
            mbar_init(bars + 8 * (kBarPFull + i), kSoftmaxWarps / 2);
            mbar_init(bars + 8 * (kBarPVDone + i), 1);
            mbar_init(bars + 8 * (kBarFinal + i), 1);
        }
        for (int i = 0; i < kStages; ++i) {
            mbar_init(bars + 8 * (kBarKVFull + i), kLoadWarps);
            mbar_init(bars + 8 * (kBarKVEmpty + i), 2);
        }
        for (int i = 0; i < kSchedDepth; ++i) {
            mbar_init(bars + 8 * (kBarSchedFull + i), 1);
            mbar_init(bars + 8 * (kBarSchedEmpty + i), kSchedReaders);
        }
        *s_abort = 0;
        for (int i = 0; i < kSchedDepth; ++i) s_bad[i] = 0;
        fence_mbar_init();
    }
    if (warp == kMmaWarp) {
        tmem_alloc(smem_u32((const void *)tmem_slot), kTmemCols);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

    // The set-up, here and in every role, may run while the kernel before still does.  Each role then waits for its end
    // (wait_prior_grid), in front of its first bounded wait: those count this kernel's own time only, and what
    // they guard comes from that kernel.

    // every wait is bounded; the first one to expire raises the abort flag, which ends all roles
    auto wait = [&](uint32_t bar, uint32_t parity) -> bool {
#pragma unroll 1
        for (uint32_t it = 0; it < kWaitLimit; ++it) {
            if (mbar_try_wait(bar, parity)) return true;
            if (*s_abort) return false;
        }
        *s_abort = 1;  // (the status word is set when the CTA ends)
        return false;
    };

#ifdef MATE_TRACE
    long long tr[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const long long tr_start = clock64();
#endif
    // The first loader warp publishes the records of the CTA's units in a small ring; every warp that
    // follows the list reads the n-th entry here and frees the slot.  false = the list is exhausted.
    auto next_unit = [&](uint32_t n, FwdUnit &u) -> bool {
        const int slot = n % kSchedDepth;
        if (!wait(bars + 8 * (kBarSchedFull + slot), (n / kSchedDepth) & 1)) return false;
        const int4 *src = reinterpret_cast<const int4 *>(s_unit + slot);
        int4 *dst = reinterpret_cast<int4 *>(&u);
#pragma unroll
        for (int i = 0; i < 4; ++i) dst[i] = src[i];
        __syncwarp();
        if (lane == 0) mbar_arrive(bars + 8 * (kBarSchedEmpty + slot));
        return u.rows != 0;
    };

    if (warp < kSoftmaxWarps) {
        // ------------------------------------------------------------------ softmax + epilogue
        reg_alloc<kRegsSoftmax>();
        const int h = warp >> 2;
        const int r = tid & 127;           // row of the half; TMEM lane
        const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
        const uint32_t tS = tmem + lane_base + h * kTile;
        const uint32_t tO = tmem + lane_base + kTmemO + h * 64;
        const uint32_t tP = tmem + lane_base + kTmemP + h * 64;
        const uint32_t bar_s = bars + 8 * (kBarSFull + h), bar_p = bars + 8 * (kBarPFull + h),
                       bar_pv = bars + 8 * (kBarPVDone + h), bar_sf = bars + 8 * (kBarSFree + h);
        uint8_t *stage = sm + kOffStage + warp * 2048;
        const uint64_t scale2 = pack_f32x2(p.scale_log2, p.scale_log2);
        uint32_t ph_s = 0, ph_pv = 0;
        bool alive = true;
        wait_prior_grid();

        for (uint32_t n = 0; alive; ++n) {
            TR_T0(t_nu);
            const int slot = n % kSchedDepth;
            if (!wait(bars + 8 * (kBarSchedFull + slot), (n / kSchedDepth) & 1)) break;
            TR_ADD(7, t_nu);
            // The record and the row data stay in shared memory until the unit is done: what is needed of
            // them is read where it is needed (registers are what this role is short of).
            const FwdUnit &un = s_unit[slot];
            if (un.rows == 0) break;
            TR_T0(t_setup);
            const int qb = QRing::buffer(n);
            if (!(alive = wait(bars + 8 * (kBarQFull + qb), QRing::full_parity(n)))) break;
            auto unit_done = [&]() {
                __syncwarp();
                if (lane == 0) {
                    mbar_arrive(bars + 8 * (kBarQEmpty + qb));
                    mbar_arrive(bars + 8 * (kBarSchedEmpty + slot));
                }
            };
            const int rows_h = un.rows_of(h);
            if (rows_h == 0) {
                unit_done();
                continue;
            }
            // this row's data: original position, key range (rows past the end shadow the last one)
            const int32_t *meta = reinterpret_cast<const int32_t *>(sm + kOffMeta) + qb * 3 * kUnitRows + h * kTile + min(r, rows_h - 1);
            // The tiles this half visits: those with positions that count for every row, then those that meet the
            // key ranges of its rows
            const int nA = un.tiles_a(), tB = un.tB & 0xff, kP = un.kP();
            const int k_lo = max(un.lo[h], un.kB0), k_hi = min(un.hi[h], un.kB_end);
            const int n_pre = nA + div_tile(kP + tB - 1, tB);
            const int b0 = max(n_pre, nA + div_tile(kP + k_lo - un.kB0, tB));
            const int n_visit = n_pre + (k_hi > k_lo ? max(nA + div_tile(kP + k_hi - un.kB0 - 1, tB) + 1 - b0, 0) : 0);
            const bool exact = (un.tB >> 8) != 0;
            const int w_lo_max = __reduce_max_sync(0xffffffffu, meta[kUnitRows]), w_hi_min = __reduce_min_sync(0xffffffffu, meta[2 * kUnitRows]);
            // The visits whose tile counts in full for every row of the warp: [0, fa) and [fb0, fb1).  (In columns of
            // range B, with the positions that count for every row in front, the rows' common range is [x_lo, x_hi).)
            const int shift = kP - un.kB0, x_lo = w_lo_max + shift, x_hi = min(w_hi_min, k_hi) + shift;
            const int fa = kP == 0 ? max(un.kA_end - un.kA0, 0) / kTile
                                   : kP / kTile + (x_lo <= kP && x_hi >= (kP / kTile + 1) * kTile);
            const int fb0 = tB == kTile ? n_pre + max((max(x_lo, 0) + kTile - 1) / kTile + nA - b0, 0) : n_visit;
            const int fb1 = n_pre + max(x_hi, 0) / kTile + nA - b0;

            TR_ADD(5, t_setup);
            float m2 = -INFINITY;                // base of the row (log2 domain, scaled)
            uint64_t l01 = 0ull, l23 = 0ull;     // row sum: packed pairs of partial sums

#pragma unroll 1
            for (int j = 0; j < n_visit; ++j) {
                TR_T0(t_ws);
                if (!(alive = wait(bar_s, ph_s))) break;
                ph_s ^= 1;
                tc_fence_after();
                TR_ADD(0, t_ws);
                TR_T0(t_p2);
                // P of the previous tile is still being read, and O written, until that tile's P V is done
                bool p_free = j == 0;
                auto wait_pv = [&]() {
                    if (p_free) return;
                    TR_T0(t_wpv);
                    alive = wait(bar_pv, ph_pv);
                    ph_pv ^= 1;
                    tc_fence_after();
                    p_free = true;
                    TR_ADD(1, t_wpv);
                };
                // Base of the row from the max t2 of this tile (the whole warp takes part).
                auto new_base = [&](float t2) {
                    if (!exact) {
                        m2 = t2 == -INFINITY ? 0.f : t2;
                        return;
                    }
                    if (!__any_sync(0xffffffffu, t2 > m2 + kRescale)) return;
                    float alpha = 1.f;
                    if (t2 > m2 + kRescale) {  // also the first finite max
                        alpha = ex2(m2 - t2);  // 0 when m2 = -inf
                        m2 = t2;
                    }
                    if (j == 0) return;
                    wait_pv();
                    const uint64_t alpha2 = pack_f32x2(alpha, alpha);
                    l01 = mul_f32x2(l01, alpha2);
                    l23 = mul_f32x2(l23, alpha2);
#pragma unroll 1
                    for (int c2 = 0; c2 < 8; ++c2) {
                        uint32_t o[8];
                        tmem_ld8(tO + c2 * 8, o);
                        tc_wait_ld();
                        reg_fence(o);
#pragma unroll
                        for (int e = 0; e < 8; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                        tmem_st8(tO + c2 * 8, o);
                    }
                };
                if (j < fa || (j >= fb0 && j < fb1)) {
                    uint32_t v[4][32];
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch) tmem_ld32(tS + ch * 32, v[ch]);
                    tc_wait_ld();
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch) reg_fence(v[ch]);
                    tc_fence_before();  // S may be overwritten
                    if (lane == 0) mbar_arrive(bar_sf);
                    if (j == 0 || exact) {  // base of the row: the max over its first tile, or, exactly, over every tile
                        float tm[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                        for (int ch = 0; ch < 4; ++ch) chunk_max(v[ch], tm);
                        new_base(fmaxf(fmaxf(tm[0], tm[1]), fmaxf(tm[2], tm[3])) * p.scale_log2);
                    }
                    const float neg_m = m2 == -INFINITY ? 0.f : -m2;  // (exact units: no score above -inf so far)
                    const uint64_t neg_m2 = pack_f32x2(neg_m, neg_m);
#pragma unroll
                    for (int ch = 0; ch < 4; ++ch) {
                        uint32_t packed[16];
                        chunk_exp(v[ch], scale2, neg_m2, packed, l01, l23);
                        if (ch == 0) wait_pv();
                        tmem_st16(tP + ch * 16, packed);
                    }
                } else {
                    // the half's MMAs touch the columns [c_begin, c1); this row counts [0, pre) and [r_lo, r_hi), and some row
                    // of the warp counts columns only there and within [e_lo, e_hi)
                    FwdUnit u = un;
                    u.tB = tB;
                    const TileInfo t = tile_info(u, j < n_pre ? j : b0 + j - n_pre, nA);
                    int c_begin, c1;
                    half_cols(un.lo[h], un.hi[h], t, c_begin, c1);
                    c_begin &= ~31;
                    const int r_lo = t.is_b ? meta[kUnitRows] - t.k0 : 0, r_hi = t.is_b ? min(meta[2 * kUnitRows] - t.k0, t.w) : 0;
                    const int e_lo = __reduce_min_sync(0xffffffffu, r_lo), e_hi = __reduce_max_sync(0xffffffffu, r_hi);
                    const int e_end = max(t.pre, e_hi > e_lo ? e_hi : 0);
                    auto off = [&](int cb) { return cb >= t.pre && (cb + 32 <= e_lo || cb >= e_hi); };
                    uint32_t v[32];
                    if (j == 0 || exact) {
                        float tm[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll 1
                        for (int cb = c_begin; cb < e_end; cb += 32) {
                            if (off(cb)) continue;
                            tmem_ld32(tS + cb, v);
                            tc_wait_ld();
                            reg_fence(v);
                            chunk_mask(v, cb, t.pre, r_lo, r_hi);
                            chunk_max(v, tm);
                        }
                        new_base(fmaxf(fmaxf(tm[0], tm[1]), fmaxf(tm[2], tm[3])) * p.scale_log2);
                    }
                    const float neg_m = m2 == -INFINITY ? 0.f : -m2;
                    const uint64_t neg_m2 = pack_f32x2(neg_m, neg_m);
                    bool held = true;  // S has not been given up yet
                    wait_pv();
#pragma unroll 1
                    for (int cb = c_begin; cb < c1; cb += 32) {
                        uint32_t packed[16];
                        if (off(cb)) {  // no row of the warp has a key here
#pragma unroll
                            for (int e = 0; e < 16; ++e) packed[e] = 0u;
                        } else {
                            tmem_ld32(tS + cb, v);
                            tc_wait_ld();
                            reg_fence(v);
                            if (cb + 32 >= e_end) {  // read for the last time
                                tc_fence_before();
                                if (lane == 0) mbar_arrive(bar_sf);
                                held = false;
                            }
                            chunk_mask(v, cb, t.pre, r_lo, r_hi);
                            chunk_exp(v, scale2, neg_m2, packed, l01, l23);
                        }
                        tmem_st16(tP + (cb >> 1), packed);
                    }
                    if (held) {
                        tc_fence_before();
                        if (lane == 0) mbar_arrive(bar_sf);
                    }
                }
                if (!alive) break;
                tc_wait_st();
                tc_fence_before();
                if (lane == 0) mbar_arrive(bar_p);
                TR_ADD(3, t_p2);
                TR_INC(4);
            }
            if (!alive) break;

            // epilogue: wait for the last P V of this half (a half may have visited no tile at all: in its part of
            // a split unit, or when its rows have no key)
            TR_T0(t_ep);
            float l = sum_f32x2(l01, l23);
            if (n_visit > 0) {
                if (!(alive = wait(bar_pv, ph_pv))) break;
                ph_pv ^= 1;
                tc_fence_after();
            }
            bool write = true;
            if (exact) {
                write = ((un.tB >> 16) >> warp) & 1;  // the others were right the first time
            } else if (n_visit > 0) {
                const bool has_keys = n_pre > 0 || min(meta[2 * kUnitRows], k_hi) > max(meta[kUnitRows], k_lo);
                if (__any_sync(0xffffffffu, r < rows_h && (!(l < kSumMax) || (l < kSumMin && has_keys)))) {
                    write = false;
                    if (lane == 0) atomicOr((uint32_t *)s_bad + slot, 1u << warp);
                }
            }
            const int n_parts = un.n_parts();
            const float4 *parts = nullptr;  // this row's column groups (of four) in the first part
            constexpr size_t kPartStride = kPartialBytes / sizeof(float4);
            if (write && n_parts > 1) {
                // Split unit: publish the un-normalised partial (groups of four columns by row, so that the
                // lanes of a warp write and read consecutive 16-byte words).  Every warp owns its 32 rows: it
                // counts the arrival, and the warp that comes last for these rows combines all parts (no wait
                // on another CTA anywhere).
                float4 *part = reinterpret_cast<float4 *>(p.ws + ((size_t)un.ws_off << 10)) + h * kTile + r;
#pragma unroll 1
                for (int c2 = 0; c2 < 4; ++c2) {
                    uint32_t o[16];
                    if (n_visit > 0) {
                        tmem_ld16(tO + c2 * 16, o);
                        tc_wait_ld();
                        reg_fence(o);
                    } else {
#pragma unroll
                        for (int e = 0; e < 16; ++e) o[e] = 0u;
                    }
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        part[(c2 * 4 + c) * kUnitRows] = make_float4(__uint_as_float(o[4 * c]), __uint_as_float(o[4 * c + 1]),
                                                                     __uint_as_float(o[4 * c + 2]), __uint_as_float(o[4 * c + 3]));
                }
                part[16 * kUnitRows] = make_float4(m2, l, 0.f, 0.f);
                __threadfence();
                __syncwarp();
                int last = 0;
                if (lane == 0) {
                    int32_t *ctr = p.counters + kSchedWords + 8 * un.ctr + warp;
                    last = atomicAdd(ctr, 1) == n_parts - 1;
                    if (last) *ctr = 0;  // ready for the next launch
                }
                write = __shfl_sync(0xffffffffu, last, 0) != 0;
                if (write) {
                    __threadfence();
                    parts = part - un.part() * kPartStride;
                    m2 = -INFINITY;
                    l = 0.f;
#pragma unroll 4
                    for (int q = 0; q < n_parts; ++q) {  // (a part in which the row has no key has the sum 0)
                        const float4 s = __ldcg(parts + q * kPartStride + 16 * kUnitRows);
                        m2 = fmaxf(m2, s.y > 0.f ? s.x : -INFINITY);
                    }
#pragma unroll 4
                    for (int q = 0; q < n_parts; ++q) {
                        const float4 s = __ldcg(parts + q * kPartStride + 16 * kUnitRows);
                        l = s.y > 0.f ? fmaf(s.y, ex2(s.x - m2), l) : l;
                    }
                }
            }
            if (write) {
                // a row without any key (possible in the passes of the row-or-column pattern) gives O = 0, LSE = -inf
                const float inv_l = l > 0.f ? 1.f / l : 0.f;
                const bool row_valid = r < rows_h;
                const int orig = p.view_order ? un.row0_of(h) + r : meta[0], dst_row = row_valid ? orig : -1;
                const size_t bh = p.tr.base(un.b, un.head());
                const int pass = p.pass(un.view());
                if (row_valid) p.LSE[pass][bh + orig] = (m2 + log2f(l)) * 0.6931471805599453f;
                // rows go through the warp's staging area, 32 columns at a time, so that a store instruction
                // writes 64 consecutive bytes of eight rows
#pragma unroll 1
                for (int c2 = 0; c2 < 2; ++c2) {
                    uint32_t o[32];
                    if (parts || n_visit == 0) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) o[e] = 0u;
#pragma unroll 2
                        for (int q = 0; q < (parts ? n_parts : 0); ++q) {  // in the order of the parts, whoever comes last
                            const float4 s = __ldcg(parts + q * kPartStride + 16 * kUnitRows);
                            const float wq = s.y > 0.f ? ex2(s.x - m2) : 0.f;
#pragma unroll
                            for (int c = 0; c < 8; ++c) {
                                const float4 x = __ldcg(parts + q * kPartStride + (c2 * 8 + c) * kUnitRows);
                                o[4 * c] = __float_as_uint(fmaf(x.x, wq, __uint_as_float(o[4 * c])));
                                o[4 * c + 1] = __float_as_uint(fmaf(x.y, wq, __uint_as_float(o[4 * c + 1])));
                                o[4 * c + 2] = __float_as_uint(fmaf(x.z, wq, __uint_as_float(o[4 * c + 2])));
                                o[4 * c + 3] = __float_as_uint(fmaf(x.w, wq, __uint_as_float(o[4 * c + 3])));
                            }
                        }
                    } else {
                        tmem_ld32(tO + c2 * 32, o);
                        tc_wait_ld();
                        reg_fence(o);
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        uint32_t w4[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            w4[e] = cvt_bf16x2(__uint_as_float(o[8 * j + 2 * e]) * inv_l, __uint_as_float(o[8 * j + 2 * e + 1]) * inv_l);
                        *reinterpret_cast<uint4 *>(stage + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4)) =
                            make_uint4(w4[0], w4[1], w4[2], w4[3]);
                    }
                    __syncwarp();
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        const int row = 8 * i + (lane >> 2), j = lane & 3;
                        const int dr = __shfl_sync(0xffffffffu, dst_row, row);
                        const uint4 x = *reinterpret_cast<const uint4 *>(stage + row * 64 + ((j ^ ((row >> 1) & 3)) << 4));
                        if (dr >= 0) *reinterpret_cast<uint4 *>(p.O[pass] + (bh + dr) * 64 + c2 * 32 + j * 8) = x;
                    }
                    __syncwarp();
                }
            }
            tc_fence_before();  // O was read; the next unit's first P V may overwrite it
            unit_done();
            TR_ADD(6, t_ep);
        }
    } else if (warp < kPadWarp0) {
        // ------------------------------------------------------------------ MMA issuers (one warp per half)
        // Per half: Q K^T of a tile -> (softmax) -> as soon as S sits in registers the Q K^T of the
        // half's next tile, and behind it the P V of the tile once its P has arrived.  A tile's ring
        // stage is released by both halves: by the commit behind the P V, or, for a tile the half
        // skips, by a plain arrival once the tile has landed.  The whole warp runs the control flow (the
        // operands stay warp-uniform: 64 / 32 clk per Q K^T / P V step, the rate of the tensor pipe,
        // against 51 clk per P V step when a single diverged thread computes them); one lane issues.
        reg_dealloc<kRegsOther>();
        const bool leader = elect_one();
        const int h = warp - kMmaWarp;
        uint32_t kv_cnt = 0, ph_p = 0, ph_sf = 0;
        bool alive = true;
        const uint32_t idesc_pv = idesc_bf16(128, 64, 0, 1);
        const uint32_t tSh0 = tmem + h * kTile, tOh = tmem + kTmemO + h * 64, tPh0 = tmem + kTmemP + h * 64;
        const uint32_t bar_p = bars + 8 * (kBarPFull + h), bar_s = bars + 8 * (kBarSFull + h),
                       bar_pv = bars + 8 * (kBarPVDone + h), bar_sf = bars + 8 * (kBarSFree + h);
        FwdUnit un;
        wait_prior_grid();

        for (uint32_t n = 0; alive; ++n) {
            if (!next_unit(n, un)) break;
            un.tB &= 0xff;
            const int nA = un.tiles_a(), nB = un.tiles_b(), n_tiles = nA + nB;
            const int qb = QRing::buffer(n);
            TR_T0(t_qf);
            if (!(alive = wait(bars + 8 * (kBarQFull + qb), QRing::full_parity(n)))) break;
            fence_proxy_async();  // the copies of 16 bytes come through the generic proxy
            tc_fence_after();
            TR_ADD(0, t_qf);
            const uint32_t q_lo = smem_desc_lo(base + kOffQ + (qb * 2 + h) * kTileBytes);
            const bool has_rows = un.rows_of(h) > 0;

            // `out`: a tile whose Q K^T has been issued and whose P V has not; one step more than there are tiles
            int o_c0 = 0, o_c1 = 0, o_stage = 0;
            bool out = false, acc = false;
#pragma unroll 1
            for (int i = 0; i <= n_tiles; ++i) {
                const TileInfo t = tile_info(un, i, nA);
                const uint32_t c = kv_cnt + i;
                const int stage = KVRing::buffer(c);
                int c0 = 0, c1 = 0;
                if (has_rows && i < n_tiles) half_cols(h ? un.lo[1] : un.lo[0], h ? un.hi[1] : un.hi[0], t, c0, c1);
                const bool visit = c1 > c0;
                if (visit) {  // the tile has landed
                    TR_T0(t_kv);
                    if (!(alive = wait(bars + 8 * (kBarKVFull + stage), KVRing::full_parity(c)))) break;
                    fence_proxy_async();
                    TR_ADD(5, t_kv);
                }
                if (out) {  // S of the outstanding tile has been read
                    TR_T0(t_sf);
                    if (!(alive = wait(bar_sf, ph_sf))) break;
                    ph_sf ^= 1;
                    TR_ADD(6, t_sf);
                }
                tc_fence_after();
                if (visit) {
                    TR_T0(t_qk);
                    const uint32_t idesc = idesc_bf16(128, c1 - c0, 0, 0);
                    const uint32_t k_lo = smem_desc_lo(base + kOffKV + stage * 2 * kTileBytes + c0 * kRowBytes);
                    const uint32_t tSh = tSh0 + c0;
                    if (leader) {
                        mma_ss_lean<0>(tSh, q_lo, k_lo, idesc);  // K = 64 as four steps of 16 (32 bytes)
                        mma_ss_lean<1>(tSh, q_lo + 2, k_lo + 2, idesc);
                        mma_ss_lean<1>(tSh, q_lo + 4, k_lo + 4, idesc);
                        mma_ss_lean<1>(tSh, q_lo + 6, k_lo + 6, idesc);
                        mma_commit(bar_s);
                    }
                    __syncwarp();
                    TR_ADD(2, t_qk);
                    TR_INC(4);
                }
                if (out) {  // P V of the previous tile, behind this tile's Q K^T: O += P V
                    TR_T0(t_wp);
                    if (!(alive = wait(bar_p, ph_p))) break;
                    TR_ADD(1, t_wp);
                    ph_p ^= 1;
                    tc_fence_after();
                    TR_T0(t_pv);
                    const int ks0 = o_c0 >> 4, n_ks = (o_c1 - o_c0) >> 4;
                    // V rows 16 ks .. 16 ks + 15 (2 KB per step), P columns 8 ks .. 8 ks + 7
                    const uint32_t v_lo = smem_desc_lo(base + kOffKV + o_stage * 2 * kTileBytes + kTileBytes + ks0 * 16 * kRowBytes);
                    const uint32_t tPh = tPh0 + ks0 * 8;
                    if (leader) {
                        mma_ts_lean_flag(tOh, tPh, v_lo, idesc_pv, acc);
#pragma unroll 1
                        for (int ks = 1; ks < n_ks; ++ks) mma_ts_lean<1>(tOh, tPh + 8 * ks, v_lo + ks * ((16 * kRowBytes) >> 4), idesc_pv);
                        mma_commit(bar_pv);
                        mma_commit(bars + 8 * (kBarKVEmpty + o_stage));
                    }
                    __syncwarp();
                    acc = true;
                    TR_ADD(3, t_pv);
                }
                if (!visit && i < n_tiles) {  // released by a plain arrival, but not before it has landed
                    if (!(alive = wait(bars + 8 * (kBarKVFull + stage), KVRing::full_parity(c)))) break;
                    fence_proxy_async();
                    if (lane == 0) mbar_arrive(bars + 8 * (kBarKVEmpty + stage));
                }
                out = visit;
                o_c0 = c0;
                o_c1 = c1;
                o_stage = stage;
            }
            kv_cnt += n_tiles;
            if (!alive) break;
            if (leader) mma_commit(bars + 8 * (kBarQEmpty + qb));
            __syncwarp();
        }
        // nothing of this CTA may still run on the tensor pipe when TMEM is freed
        if (leader) mma_commit(bars + 8 * (kBarFinal + h));
        __syncwarp();
        mbar_wait_bounded(bars + 8 * (kBarFinal + h), 0, kWaitLimit);
    } else if (warp < kLoadWarp0) {
        // ------------------------------------------------------------------ padding rows: O = 0, LSE = -inf
        reg_dealloc<kRegsOther>();
        wait_prior_grid();
#pragma unroll 1
        for (int c = blockIdx.x; c < p.n_pads; c += gridDim.x) {
            const PadChunk pc = p.pads[c];
            const ViewPlan &vp = p.view[pc.view()];
#pragma unroll 1
            for (int i = (warp - kPadWarp0) * 4 + (lane >> 3); i < pc.n; i += 4 * kPadWarps) {  // eight lanes per row
                const int t = pc.t0 + i;
                const int orig = p.view_order ? t : __ldg(vp.perm + (size_t)pc.b * p.N + t);
                if (p.tr.exists(pc.b, orig)) {
                    const size_t row = p.tr.base(pc.b, pc.head()) + orig;
                    reinterpret_cast<uint4 *>(p.O[p.pass(pc.view())] + row * 64)[lane & 7] = make_uint4(0, 0, 0, 0);
                    if ((lane & 7) == 0) p.LSE[p.pass(pc.view())][row] = -INFINITY;
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ loaders
        reg_dealloc<kRegsOther>();
        wait_prior_grid();
        const int lw = warp - kLoadWarp0;
        const bool leader = elect_one();
        uint32_t kv_cnt = 0;
        bool alive = true;
        FwdUnit un;
        uint32_t checked = 0;  // entries of the list that are known to be done
        int4 held_back = make_int4(0, 0, 0, 0);
        bool redo = false;     // the entry being loaded is one that is done once more
        auto rec_rows = [&]() { return __shfl_sync(0xffffffffu, rec.w, 0); };  // FwdUnit::rows

        for (uint32_t n = 0; alive; ++n) {
            const int slot = n % kSchedDepth;
            if (warp == kLoadWarp0) {
                // Before the n-th entry goes out, the entries up to n - kSchedDepth have to be done (their slots are
                // used again), and before the end of the list all of them: one that came out with a row sum out of
                // range goes out once more, as an exact unit for the warps concerned.
                const uint32_t done_to = rec_rows() ? n - min(n, (uint32_t)kSchedDepth - 1) : n;
                bool again = false;
                for (; checked < done_to && !again; ++checked) {
                    const int sc = checked % kSchedDepth;
                    if (!(alive = wait(bars + 8 * (kBarSchedEmpty + sc), (checked / kSchedDepth) & 1))) break;
                    const uint32_t bad = s_bad[sc];
                    if (bad) {
                        again = true;
                        held_back = rec;  // the record that was next comes after it
                        if (lane < 4) rec = reinterpret_cast<const int4 *>(s_unit + sc)[lane];
                        if (lane == 3) rec.x = (rec.x & 0xff) | 0x100 | bad << 16;
                        __syncwarp();
                        if (lane == 0) s_bad[sc] = 0;
                    }
                }
                if (!alive) break;
                if (lane < 4) reinterpret_cast<int4 *>(s_unit + slot)[lane] = rec;
                __syncwarp();
                if (lane == 0) mbar_arrive(bars + 8 * (kBarSchedFull + slot));  // release: the record is visible to the readers
                redo = again;
            }
            if (!next_unit(n, un)) break;
            un.tB &= 0xff;
            const int nA = un.tiles_a(), nB = un.tiles_b(), n_tiles = nA + nB;
            const ViewPlan &vp = p.view[un.view()];
            const size_t bn = (size_t)un.b * p.N;
            const int32_t *perm = p.view_order ? nullptr : vp.perm + bn;
            const size_t bh = p.tr.base(un.b, un.head());
            const uint8_t *Qbh = reinterpret_cast<const uint8_t *>(p.Q + bh * 64), *Kbh = reinterpret_cast<const uint8_t *>(p.K + bh * 64);
            const int64_t v_off = reinterpret_cast<const uint8_t *>(p.V) - reinterpret_cast<const uint8_t *>(p.K);
            // Rows of the order that sit in place in the tensors ([0, ident)): a K/V tile inside that range
            // (see bulk_tile) is one contiguous [128, 64] box and comes in by one bulk tensor copy per matrix
            // instead of 2 x 1024 copies of 16 bytes.  That is the prefix block's full tiles in every unit and, for a
            // row-major table, those of the row view.
            const int ident = !p.bulk ? 0 : p.view_order ? p.N : __ldg(vp.ident + un.b);
            const int qb = QRing::buffer(n);
            // steps -2, -1: the two Q halves (and the row data of the unit); steps 0 ..: the key tiles
            auto step_idx = [&](int i) {
                const TileInfo t = i < 0 ? row_tile(un.row0_of(i + 2), un.rows_of(i + 2)) : tile_info(un, i, nA);
                return t.w > 0 ? fetch_idx(perm, t, lw, lane) : 0;
            };
            int next = step_idx(-2);
#pragma unroll 1
            for (int i = -2; i < n_tiles; ++i) {
                const int now = next;
                if (i + 1 < n_tiles) next = step_idx(i + 1);
                const uint32_t c = kv_cnt + max(i, 0), stage = KVRing::buffer(c);
                const uint32_t bar_full = bars + 8 * (i < 0 ? kBarQFull + qb : kBarKVFull + stage);
                if (i != -1 && !(alive = wait(bars + 8 * (i < 0 ? kBarQEmpty + qb : kBarKVEmpty + stage),
                                              i < 0 ? QRing::wait_parity(n) : KVRing::wait_parity(c)))) break;
                TR_T0(t_cp);
                if (i == -2) {  // row data for the softmax threads: original position and key range
#pragma unroll 1
                    for (int half = 0; half < 2; ++half) {
                        const int rr = 32 * lw + lane;
                        if (rr < un.rows_of(half)) {
                            const size_t at = bn + un.row0_of(half) + rr;
                            const uint32_t meta = base + kOffMeta + (qb * 3 * kUnitRows + half * kTile + rr) * 4;
                            cp_async4(meta, vp.perm + at);
                            cp_async4(meta + kUnitRows * 4, vp.seg_lo + at);
                            cp_async4(meta + 2 * kUnitRows * 4, vp.seg_hi + at);
                        }
                    }
                }
                const TileInfo t = tile_info(un, max(i, 0), nA);
                const uint32_t dst = base + (i < 0 ? kOffQ + (qb * 2 + i + 2) * kTileBytes : kOffKV + stage * 2 * kTileBytes);
                const bool bulk = i >= 0 && bulk_tile(t, ident);
                // (rows of a Q half past its last one are never looked at: their results are not stored)
                if (!bulk) gather_rows(dst, i < 0 ? Qbh : Kbh, i >= 0, v_off, now, i < 0 ? un.rows_of(i + 2) : (t.w + 15) & ~15, lw, lane);
                if (i != -2) {
                    cp_async_arrive(bar_full);
                    __syncwarp();
                    if (bulk && lw == 0) {
                        if (leader) {
                            mbar_arrive_expect_tx(bar_full, 2 * kTileBytes);
                            tma_load_2d(dst, &p.tmK, 0, (int)bh + t.first(), bar_full);
                            tma_load_2d(dst + kTileBytes, &p.tmV, 0, (int)bh + t.first(), bar_full);
                        }
                        __syncwarp();
                    } else if (lane == 0) {
                        mbar_arrive(bar_full);
                    }
                }
                TR_ADD(2, t_cp);
                TR_INC(4);
            }
            if (warp == kLoadWarp0 && alive) {
                if (redo) {
                    rec = held_back;
                } else {
                    // The next unit is claimed when the fourth tile from the end has been read (the first tile, of a shorter unit).
                    // Claimed before that it goes to a CTA that is not the next to be free, claimed much later its loads are late.
                    // As soon as every load is under way / so / at the second tile from the end, forward alone: 8 x 512
                    // tokens 15.9 / 15.3 / 15.4 us, 4 x 2048 30.2 / 29.6 / 30.0, 1 x 8192 53.2 / 49.7 / 51.1, 2 x 4096 51.7 / 51.4 /
                    // 54.3.  Units of one tile do not wait: nothing would be left to hide the claim behind.
                    const uint32_t c = kv_cnt + max(n_tiles - 4, 0);
                    if (n_tiles > 1 && !(alive = wait(bars + 8 * (kBarKVEmpty + KVRing::buffer(c)), KVRing::wait_parity(c + kStages)))) break;
                    claim();
                    fetch_record(true);
                }
            }
            kv_cnt += n_tiles;
        }
    }

#ifdef MATE_TRACE
    if (lane == 0 && (warp == 0 || warp == 4 || warp == kMmaWarp || warp == kLoadWarp0) &&
        blockIdx.x < kTraceCtas) {  // MMA: half 0's warp
        const int role = warp == 0 ? 0 : warp == 4 ? 1 : warp == kMmaWarp ? 2 : 3;
        long long *o = g_trace + blockIdx.x * 32 + role * 8;
        for (int i = 0; i < 7; ++i) o[i] = tr[i];
        o[7] = clock64() - tr_start;
    }
#endif
    if (*s_abort)  // copies may still be on their way to shared memory: they take a few microseconds
        for (int i = 0; i < 50; ++i) __nanosleep(1000);
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && *s_abort) atomicOr(p.status + 1, 1);
    if (warp == kMmaWarp) tmem_dealloc(tmem, kTmemCols);
}


// cuTensorMapEncodeTiled, taken from the driver through the runtime (the library does not link libcuda)
using EncodeTiledFn = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                   const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn() {
    static EncodeTiledFn fn = []() -> EncodeTiledFn {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult res;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &res) != cudaSuccess ||
            res != cudaDriverEntryPointSuccess)
            return nullptr;
        return reinterpret_cast<EncodeTiledFn>(ptr);
    }();
    return fn;
}

}  // namespace

// Map over a [rows, 64] bf16 matrix (row = 128 bytes): boxes of 128 rows, written to shared memory in
// the 128-byte swizzle the tensor-core descriptors expect (16-byte chunk index XOR row & 7).
bool make_row_map(CUtensorMap *map, const void *base, size_t rows) {
    EncodeTiledFn fn = encode_tiled_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {64, (cuuint64_t)rows};
    const cuuint64_t strides[1] = {kRowBytes};
    const cuuint32_t box[2] = {64, kTile};
    const cuuint32_t elem[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, elem,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool tc_supported(int d, int dtype) { return d == 64 && dtype == MATE_BF16; }

size_t tc_fwd_workspace(const mate_plan_t *plan, int) { return plan->fwd_ws_bytes; }

namespace {
template <bool kMany>
int launch(const mate_plan_t *plan, const void *Q, const void *K, const void *V, float scale, void *const (&O)[kPasses],
           float *const (&LSE)[kPasses], void *workspace, unsigned flags, cudaStream_t stream) {
    static SmemAttrOnce attr;
    if (!(scale > 0.f)) return MATE_ERR_UNSUPPORTED;  // the row max is taken before scaling (the caller falls back)
    if (plan->fwd_grid == 0) return MATE_OK;
    if (attr.ensure((const void *)tc_fwd_kernel<kMany>, (int)kSmemBytes, plan->device) != MATE_OK) return MATE_ERR_CUDA;
    Params<kMany> p;
    const size_t rows = plan->n_rows();
    // Bulk tensor copies for the K/V tiles that are contiguous in the caller's tensors (see bulk_tile), unless the
    // caller asks for gathers or there are no maps to be had; tensors in view order always take them.  Bulk copies against gathers, back to back:
    // 4 x 2048 tokens 29.4 us against 29.5, 8 x 512 15.5 and 15.5, 2 x 4096 51.1 and 51.5, 1 x 8192 48.6 and 48.8.
    const bool want_bulk = !(flags & MATE_FLAG_GATHER_TILES) || (flags & MATE_FLAG_VIEW_ORDER);
    p.bulk = want_bulk && rows < (size_t(1) << 31) && make_row_map(&p.tmK, K, rows) && make_row_map(&p.tmV, V, rows);
    p.view_order = (flags & MATE_FLAG_VIEW_ORDER) ? 1 : 0;
    p.Q = (const __nv_bfloat16 *)Q;
    p.K = (const __nv_bfloat16 *)K;
    p.V = (const __nv_bfloat16 *)V;
    for (int i = 0; i < p.kO; ++i) {
        p.O[i] = (__nv_bfloat16 *)O[i];
        p.LSE[i] = LSE[i];
    }
    for (int v = 0; v < p.kV; ++v) p.view[v] = plan->work_view(v);
    p.units = plan->fwd_units_dev;
    p.n_units = plan->n_fwd_units;
    p.pads = plan->pads_dev;
    p.n_pads = plan->n_pads;
    p.N = plan->N;
    p.H = plan->H;
    p.tr = plan->rows();
    p.scale_log2 = scale * 1.4426950408889634f;
    p.status = plan->status_dev;
    p.counters = plan->fwd_counters_dev;
    p.ws = (uint8_t *)workspace;
    return launch_after(tc_fwd_kernel<kMany>, dim3((unsigned)plan->fwd_grid), kThreads, kSmemBytes, stream, p) == cudaSuccess ? MATE_OK
                                                                                                                      : MATE_ERR_CUDA;
}

}  // namespace

int tc_fwd(const mate_plan_t *plan, const void *Q, const void *K, const void *V, float scale, void *const (&O)[kPasses],
           float *const (&LSE)[kPasses], void *workspace, unsigned flags, cudaStream_t stream) {
    return plan->sub[0] ? launch<true>(plan, Q, K, V, scale, O, LSE, workspace, flags, stream)
                        : launch<false>(plan, Q, K, V, scale, O, LSE, workspace, flags, stream);
}

}  // namespace mate

#ifdef MATE_TRACE
// copies the cycle counters of the last forward launch to the host: [kTraceCtas CTAs][4 roles][8]
extern "C" int mate_debug_trace(long long *host_out) {
    return cudaMemcpyFromSymbol(host_out, mate::g_trace, sizeof(long long) * mate::kTraceCtas * 32) == cudaSuccess ? 0 : -4;
}
#endif
