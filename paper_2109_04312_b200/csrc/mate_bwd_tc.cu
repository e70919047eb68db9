// Tensor-core backward of multi-view attention for bf16, d = 64, on sm_100a (derived from the head
// formula of Section 3; the paper states no backward).  With P = exp(scale S - LSE) on the pattern,
// D_k = sum_e dO_ke O_ke and dS = P o (dP - D):
//     dV_j = sum_k P_kj dO_k      dP_kj = dO_k . V_j
//     dQ_k = scale sum_j dS_kj K_j      dK_j = scale sum_k dS_kj Q_k
// Work units are up to 128 rows of a head in the head's view order (Section 3.1) and the column tiles they
// meet; the pattern is symmetric, so the same units serve both sides:
//   query side  rows = queries, columns = their keys:  S = Q K^T, dP = dO V^T -> dS -> dQ += dS K
//   key side    rows = keys, columns = the queries that attend them:  S^T = K Q^T, dP^T = V dO^T
//               -> P^T, dS^T -> dV += P^T dO, dK += dS^T Q
// so no gradient is accumulated across CTAs and the result does not depend on the schedule.
//
// One persistent, warp-specialised CTA per SM; work items (unit, side) are handed out through
// a counter, longest first.
//   warps 0-7   arithmetic: two threads (r, r + 128) share row r of the 128-row tile, the lane of
//               tensor memory; each takes every other chunk of 32 columns.  S and dP (fp32) come out of
//               tensor memory, P / dS (bf16 pairs) go back into it as MMA operands.
//   warps 8-11  gradients of a finished item: tensor memory -> the rows' original positions, through a staging area so that
//               a store covers half rows of 64 bytes
//   warps 12,13 issue the tcgen05.mma (one elected lane each): S and dP of the tiles / the gradient MMAs, each as soon as
//               what it needs is there
//   warps 14,15 zero the gradients of the padding rows
//   warps 16-19 loaders: rows by view-order index, 16 bytes per lane and copy, 32 rows of every load per warp, or a column
//               tile whose rows lie in place in the tensors by one bulk tensor copy per matrix, into 128-byte swizzled shared
//               memory (row operands double buffered, column tiles in a ring of 4).  Either kind completes on the
//               tile's barrier by itself, so no warp waits for its copies in order to signal them.
// On the key side -LSE and D belong to the columns.  Read from shared memory by every arithmetic thread (32 loads of 16 bytes per
// tile) they cost 340 clk of the shared-memory pipe, and the registers they went through spilled.  They come in with the MMAs
// instead, wherever the scale can be divided by (divides): S and dP get one more K step, ones x (-LSE / scale) and ones x (-D).  Either
// number is the sum of three bf16 to its last bit; the quotient is rounded to fp32, and so are the sums in the accumulators.  Errors against
// 64 bits (2-norm) are those of the loads: over 94 batches of six shapes, 150 to 8192 tokens, dK and dV stay at 2.3e-3 to 2.9e-3 and
// the two forms' differ by (2.0 +- 1.4) and (-0.8 +- 1.5) parts in 100,000; with LSE / scale of 8192 and D of 4096 2.42e-3 and 2.41e-3.
// What bounds it.  The exponentials take 1024 clk per 128 x 128 tile and side (16 per clock and SM); what is left is the
// chain S complete -> registers -> arithmetic -> operands -> next S, about 1600 clk per tile when all pairs count, and on
// tables the loads and the cost per item.  Hence:
//   - A tile that counts in full is taken into registers whole (64 columns of S and of dP per thread), which frees S
//     and dP for the next tile's MMAs before the arithmetic begins; the operand columns are waited for behind the
//     first chunk's arithmetic.
//   - The arithmetic warps have no part in an item's end: the store warps wait for its last gradient MMAs (700 clk
//     behind the last operands) and take the gradients out of tensor memory under the next item's first tile.
//   - All loader warps take part in every load, with the look-ups a tile ahead of the copies.  (Tensor copies of four rows by
//     teams of two warps that take the loads in turn: 1 x 512 tokens 10.5 us, 4 x 2048 58.3, 1 x 8192 108.3 against 10.0, 56.1,
//     104.9.)
//   - All roles share an instruction cache of about 32 KB: waits and rare paths are rolled.  (An earlier form with gathers and
//     waits unrolled, 14 KB more, took 92 us for 4 x 2048 tokens: a warp waited for instructions 3.9 times as long as it
//     issued, instead of 0.7.)
//   - The tensor maps are fetched ahead of the first copy (4 x 2048 tokens, forward and backward, 99.4 us without, 98.0 with).
// Forward and backward back to back, 8 x 512 tokens / 4 x 2048 / 1 x 8192 / 2 x 4096: one warp for all MMAs and the epilogue in the
// arithmetic warps 47.7 / 101.8 / 176.0 / 172.9 us; with store warps and two MMA warps, gathers by tensor copies 46.4 / 98.1 /
// 165.6 / 162.7 (backward alone 23.0 / 59.6 / 107.7 / 102.1); by 16-byte copies 41.1 / 86.9 / 160.1 / 155.6 (22.1 / 57.8 / 104.3 / 99.9);
// waits without a hint 21.4 / 56.3 / 101.2 / 97.2 alone; this form, with the row dots in one wave, 21.4 / 54.6 / 98.0 / 96.6.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "load_ring.h"
#include "mate_internal.h"
#include "sm100_ptx.cuh"
#include "tc_tiles.cuh"

namespace mate {

#ifdef MATE_TRACE
__device__ long long g_trace_bwd[kTraceCtas * 32];
#endif

namespace {

using namespace ptx;

constexpr int kComputeWarps = 8;
constexpr int kStoreWarp0 = kComputeWarps;
constexpr int kStoreWarps = 4;
constexpr int kMmaWarp = kStoreWarp0 + kStoreWarps;
constexpr int kMmaWarps = 2;  // one for S and dP, one for the gradients
constexpr int kPadWarp0 = kMmaWarp + kMmaWarps;
constexpr int kPadWarps = 2;
static_assert(kPadRows == 32 * kPadWarps, "a row per lane");
constexpr int kLoadWarp0 = kPadWarp0 + kPadWarps;
constexpr int kLoadWarps = 4;
static_assert(kTile == 32 * kLoadWarps, "a row of a tile per loader thread");
constexpr int kThreads = 32 * (kLoadWarp0 + kLoadWarps);
// registers per thread after the roles have split: 256 x 160 + 128 x 56 + 128 x 40 + 128 x 64 = 61,440 = the 640 x 96 the
// CTA is launched with; 256 x 168 + 128 x 48 + 128 x 40 + 128 x 56, as many, where the arithmetic warps read the columns' data
// (!kByMma, which spills 36 bytes and reads back 80 so, 72 and 176 with the other split: 1 x 8192 tokens 108.2 instead of 116.4 us)
template <bool kByMma>
struct Regs {
    static constexpr int kCompute = kByMma ? 160 : 168, kStore = kByMma ? 56 : 48, kMma = 40, kLoad = kByMma ? 64 : 56;
    static_assert(2 * kCompute + kStore + kMma + kLoad == 480, "what the CTA is launched with");
};
constexpr int kStages = 4;  // ring of column tiles
using RowRing = LoadRing<2>;
using ColRing = LoadRing<kStages>;
constexpr int kSchedDepth = 4;
constexpr uint32_t kOffR = 0;                                    // [2 buffers] x (Ra: Q or K, Rb: dO or V), 16 KB each
constexpr uint32_t kOffC = 4 * kTileBytes;                       // [kStages] x (Ca 16 KB, Cb 16 KB)
constexpr uint32_t kOffExt = kOffC + kStages * 2 * kTileBytes;   // [kStages] x 128 rows x 16 bytes of -LSE / scale, then of -D (key side;
                                                                 // !kByMma: 128 x (-LSE log2 e), 128 x D)
constexpr uint32_t kOffOnes = kOffExt + kStages * 4096;          // 128 rows x (1, 1, 1, 0, 0, 0, 0, 0)
constexpr uint32_t kOffZero = kOffOnes + 2048;                   // 128 rows x 16 bytes of zeros
constexpr uint32_t kOffMeta = kOffZero + 2048;                   // [2 buffers] x (perm, seg_lo, seg_hi, -LSE log2 e, D) of 128 rows
constexpr uint32_t kOffStage = kOffMeta + 2 * 5 * kTile * 4;     // [store warps] x 32 rows x 64 bytes
constexpr uint32_t kOffItem = kOffStage + kStoreWarps * 2048;    // [kSchedDepth] unit records
constexpr uint32_t kOffBar = kOffItem + kSchedDepth * sizeof(FwdUnit);
constexpr uint32_t kSmemBytes = kOffBar + 512 + 1024;            // + slack for the 1024-byte alignment
static_assert(kSmemBytes <= 232448, "shared memory per CTA");
// barrier slots (8 bytes each) behind kOffBar
enum {
    kBarRFull = 0,                     // [2] loaders -> MMA, arithmetic      (count kLoadWarps)
    kBarREmpty = kBarRFull + 2,        // [2] MMA commit and arithmetic warps (row data read) -> loaders (count 1 + kComputeWarps + kStoreWarps)
    kBarCFull = kBarREmpty + 2,        // [kStages] loaders -> MMA            (count kLoadWarps)
    kBarCEmpty = kBarCFull + kStages,  // [kStages] MMA commit -> loaders     (count 1)
    kBarSFull = kBarCEmpty + kStages,  // MMA commit -> arithmetic: S and dP of a tile are complete (count 1)
    kBarAFull,         // arithmetic -> MMA: the bf16 operands of a tile are written (count: one per warp)
    kBarGDone,         // MMA commit -> arithmetic: the gradient MMAs of a tile are complete (count 1)
    kBarSTFree,        // arithmetic -> MMA: S and dP of a tile are in registers (count: one per warp)
    kBarItemDone,      // MMA commit -> store warps: every gradient MMA of an item is complete (count 1)
    kBarAccFree,       // store warps -> MMA: the gradients of an item are in registers (count: one per warp)
    kBarSchedFull,                               // [kSchedDepth] scheduler -> every warp (count 1)
    kBarSchedEmpty = kBarSchedFull + kSchedDepth,  // [kSchedDepth] every warp -> scheduler (count kSchedReaders)
    kBarFinal = kBarSchedEmpty + kSchedDepth,      // [2]
    kNumBars = kBarFinal + 2
};
static_assert(8 * kNumBars + 8 <= 512, "the barriers and two words behind them");
constexpr int kSchedReaders = kComputeWarps + kMmaWarps + kStoreWarps + kLoadWarps;
// tensor memory columns
constexpr uint32_t kTmS = 0, kTmT = 128, kTmA1 = 256, kTmA2 = 320, kTmAcc1 = 384, kTmAcc2 = 448;

// kMany: the three passes of a row-or-column plan.  (An instance of its own: the look-ups by pass cost the others up to 1 %,
// 4 x 2048 tokens 94.4 -> 95.3 us forward and backward.)
template <bool kMany>
struct Params {
    static constexpr int kV = kMany ? kViews : 2, kO = kMany ? kPasses : 1;
    __device__ static __forceinline__ int pass(int view) { return kMany ? pass_of(view) : 0; }
    CUtensorMap tmQ, tmK, tmV, tmdO;  // boxes of 128 rows, 128-byte swizzle
    int bulk;                         // 0: there are none, every tile is gathered row by row
    const __nv_bfloat16 *Q, *K, *V, *dO;
    const float *nlse, *D;  // per row, original order: -LSE log2 e, D
    const uint4 *ext;       // per row: -LSE / scale and -D, each as the sum of three bf16 (and five zeros)
    __nv_bfloat16 *dQ[kO], *dK[kO], *dV[kO];
    ViewPlan view[kV];
    const FwdUnit *units;  // one half each; item = 2 unit + (0 key side, 1 query side)
    int n_units, N, H;
    const PadChunk *pads;
    int n_pads;
    TensorRows tr;         // where (example, head) starts in the tensors
    float scale, scale_log2;
    int32_t *status;
    int32_t *counter;      // next work item (zeroed before the launch)
};

// A number as the sum of three bf16, exactly (24 bits of mantissa, 8 each): the first three of eight in a row of 16 bytes.
__device__ __forceinline__ uint4 split_bf16(float x) {
    const uint32_t h = __float_as_uint(x) & 0xffff0000u;
    float left = x - __uint_as_float(h);
    if (!(fabsf(x) <= 3.4028235e38f)) left = 0.f;  // inf and NaN as they are
    const uint32_t m = __float_as_uint(left) & 0xffff0000u;
    const uint32_t l = __float_as_uint(left - __uint_as_float(m));
    return make_uint4(h >> 16 | m, l >> 16, 0u, 0u);
}
// D_k = sum_e dO_ke O_ke and -LSE_k log2 e per row (original order), and what the MMAs of the key side add to their
// accumulators (ext), d = 64: eight threads per row, 16 bytes
// of each tensor and row per thread, all rows of a thread in flight.  HBM- or L2-bound, and in front of every backward: blocks
// of a second wave, and a row's LSE fetched behind its sum, cost 1.0 to 1.3 us at 4 x 2048 to 1 x 8192 tokens (55.9 -> 54.7 and
// 99.3 -> 98.0 us with four rows per thread instead of two), four rows where two fit 0.6 us at 8 x 512.  The first block also clears the
// work-item counter of the kernel that follows (and the rest of its 256 bytes).
// kRows: rows of a group of eight threads, 32 groups to a block.
constexpr int kRowdotBlocks = 8;  // of an SM, with one or two rows (26 and 32 registers)
// (Four rows take 48 registers with all their loads in flight.  With 40, for six blocks to an SM, backward of 4 x 2048 / 2 x 4096 tokens
// 54.9 / 95.6 us instead of 54.4 / 95.4, with 34 54.7 / 96.7.)
template <int kRows>
__global__ void __launch_bounds__(256, kRows < 4 ? kRowdotBlocks : 1) rowdot_kernel(const __nv_bfloat16 *__restrict__ dO, const __nv_bfloat16 *__restrict__ O,
                                                     const float *__restrict__ LSE, float *__restrict__ D,
                                                     float *__restrict__ nlse, uint4 *__restrict__ ext, float scale,
                                                     size_t rows, int32_t *counter) {
    launch_dependents();
    wait_prior_grid();
    if (blockIdx.x == 0 && threadIdx.x < 64) counter[threadIdx.x] = 0;
    const int part = threadIdx.x & 7;
    const size_t r0 = (size_t)blockIdx.x * (32 * kRows) + (threadIdx.x >> 3), own = r0 + 32 * part;  // own: the row this thread finishes
    uint4 a[kRows], b[kRows];
#pragma unroll
    for (int q = 0; q < kRows; ++q) {
        const size_t r = r0 + 32 * q;
        a[q] = b[q] = make_uint4(0, 0, 0, 0);
        if (r < rows) {
            a[q] = __ldg(reinterpret_cast<const uint4 *>(dO + r * 64) + part);
            b[q] = __ldg(reinterpret_cast<const uint4 *>(O + r * 64) + part);
        }
    }
    const bool finish = part < kRows && own < rows;
    const float lse = finish ? __ldg(LSE + own) : 0.f;
    float dot = 0.f;
#pragma unroll
    for (int q = 0; q < kRows; ++q) {
        const uint32_t aw[4] = {a[q].x, a[q].y, a[q].z, a[q].w}, bw[4] = {b[q].x, b[q].y, b[q].z, b[q].w};
        float acc = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const float2 fa = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&aw[i]));
            const float2 fb = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&bw[i]));
            acc = fmaf(fa.x, fb.x, acc);
            acc = fmaf(fa.y, fb.y, acc);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (part == q) dot = acc;
    }
    if (finish) {
        D[own] = dot;
        nlse[own] = lse * -1.4426950408889634f;
        // (LSE = -inf: a padding row, which is no column of any tile, or a query all of whose scores are -inf, whose weights are not
        // numbers: -inf + inf)
        ext[2 * own] = split_bf16(-lse / scale);
        ext[2 * own + 1] = split_bf16(-dot);
    }
}

// P and dS of 32 columns, as bf16 pairs (even column in the low half): p = exp2(s * scale2 + nlse), dS = p (dP - D).
// Query side: nlse and D are the row's.  Key side: they are the columns', and the accumulators hold s - LSE / scale and dP - D
// already (kByMma), or they are in shared memory, at vec and 512 bytes behind.  Columns whose bit of
// `on` is clear do not count (kMask).  Two columns per instruction except for the exponential.
template <bool kKeySide, bool kMask, bool kByMma>
__device__ __forceinline__ void math32(const uint32_t (&sv)[32], const uint32_t (&tv)[32], uint64_t scale2, uint64_t row_nlse2,
                                       uint64_t row_D2, uint32_t vec, uint32_t on, uint32_t (&pk_p)[16], uint32_t (&pk_ds)[16]) {
    uint64_t nlse2[2] = {row_nlse2, row_nlse2}, D2[2] = {row_D2, row_D2};
#pragma unroll
    for (int k = 0; k < 32; k += 2) {
        if (kKeySide && !kByMma && k % 4 == 0) {
            const float4 a = ld_shared_f4(vec + 4 * k), b = ld_shared_f4(vec + 512 + 4 * k);
            nlse2[0] = pack_f32x2(a.x, a.y), nlse2[1] = pack_f32x2(a.z, a.w);
            D2[0] = pack_f32x2(b.x, b.y), D2[1] = pack_f32x2(b.z, b.w);
        }
        const uint64_t s = pack_f32x2(sv[k], sv[k + 1]), t = pack_f32x2(tv[k], tv[k + 1]);
        const int q = k / 2 % 2;
        float x0, x1, d0, d1;
        unpack_f32x2(kKeySide && kByMma ? mul_f32x2(s, scale2) : fma_f32x2(s, scale2, nlse2[q]), x0, x1);
        float p0 = ex2(x0), p1 = ex2(x1);
        if (kMask) {
            if (!(on & (1u << k))) p0 = 0.f;
            if (!(on & (2u << k))) p1 = 0.f;
        }
        unpack_f32x2(mul_f32x2(pack_f32x2(p0, p1), kKeySide && kByMma ? t : sub_f32x2(t, D2[q])), d0, d1);
        if (kKeySide) pk_p[k >> 1] = cvt_bf16x2(p0, p1);
        pk_ds[k >> 1] = cvt_bf16x2(d0, d1);
    }
}
// Tiles of an item: nA of range A, then those of range B (all of them kTile columns wide but for the last of either).
struct ItemTiles {
    int kA0, len_a, kB0, len_b, kP, nA, n;
    __device__ __forceinline__ explicit ItemTiles(const FwdUnit &u) {
        kA0 = u.kA0;
        kB0 = u.kB0;
        kP = u.kP();
        len_a = max(u.kA_end - kA0, 0);
        len_b = kP + u.kB_end - kB0;
        nA = (len_a + kTile - 1) / kTile;
        n = nA + (len_b + kTile - 1) / kTile;
    }
    __device__ __forceinline__ TileInfo tile(int i) const {  // = tile_info
        TileInfo t;
        t.is_b = i >= nA;
        const int off = (t.is_b ? i - nA : i) * kTile;
        t.w = min((t.is_b ? len_b : len_a) - off, kTile);
        t.x0 = t.is_b ? off : kA0 + off;
        t.k0 = t.is_b ? off + kB0 - kP : t.x0;
        t.pre = t.is_b ? min(max(kP - off, 0), t.w) : t.w;
        return t;
    }
};
__device__ __forceinline__ uint32_t bits_below(int n) { return n <= 0 ? 0u : n >= 32 ? 0xffffffffu : (1u << n) - 1u; }

// kByMma: the key side's column data come in with the MMAs, which takes a scale that can be divided by (divides); otherwise
// every thread reads them from shared memory.
template <bool kMany, bool kByMma>
__global__ void __launch_bounds__(kThreads, 1) tc_bwd_kernel(const __grid_constant__ Params<kMany> p) {
    launch_dependents();
    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    const uint32_t base = (raw + 1023u) & ~1023u;
    uint8_t *sm = smem_raw + (base - raw);
    const uint32_t bars = base + kOffBar;
    volatile uint32_t *tmem_slot = (volatile uint32_t *)(sm + kOffBar + 8 * kNumBars);
    volatile int *s_abort = (volatile int *)(sm + kOffBar + 8 * kNumBars + 4);
    FwdUnit *s_item = reinterpret_cast<FwdUnit *>(sm + kOffItem);  // [kSchedDepth]; rows = 0 marks the end of the list,
                                                                   // ws_off holds the side
    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = tid & 31;

    // The first loader warp hands out the items; its lanes 0-3 hold the record of the next one.  The first item
    // of a CTA is its own index, later ones come from the shared counter, each claimed when every load of the item before is
    // under way.  (Claimed in front of the last load but one, the record fetched in front of the last: the loads wait behind
    // the look-ups; 1 x 134 tokens 7.85 us instead of 7.49, 2 x 1026 22.3 / 20.5, 8 x 512 22.2 / 21.9, 4 x 2048 56.1 / 55.5.  Claimed
    // when the fourth tile from the end has been read, as in the forward: 8 x 512 12 %, 4 x 2048 11 % slower.)
    int4 rec = make_int4(0, 0, 0, 0);
    int it_next = blockIdx.x;  // lane 0
    auto claim = [&]() {
        if (lane == 0) it_next = atomicAdd(p.counter, 1);
    };
    auto fetch_record = [&](bool claimed = true) {
        const int it = __shfl_sync(0xffffffffu, it_next, 0) + (claimed ? (int)gridDim.x : 0);
        rec = make_int4(0, 0, 0, 0);  // rows = 0: the list is exhausted
        if (it < 2 * p.n_units && lane < 4) {
            rec = __ldg(reinterpret_cast<const int4 *>(p.units + (it >> 1)) + lane);
            if (lane == 3) rec.z = it & 1;
        }
    };
    if (warp == kLoadWarp0) fetch_record(false);
    if (warp == kLoadWarp0 + 1 && lane < 4) prefetch_tmap(&p.tmQ + lane, p.bulk);  // all four of them

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(bars + 8 * (kBarRFull + i), kLoadWarps);
            mbar_init(bars + 8 * (kBarREmpty + i), 1 + kComputeWarps + kStoreWarps);
        }
        for (int i = 0; i < kStages; ++i) {
            mbar_init(bars + 8 * (kBarCFull + i), kLoadWarps);
            mbar_init(bars + 8 * (kBarCEmpty + i), 1);
        }
        mbar_init(bars + 8 * kBarSFull, 1);
        mbar_init(bars + 8 * kBarAFull, kComputeWarps);
        mbar_init(bars + 8 * kBarSTFree, kComputeWarps);
        mbar_init(bars + 8 * kBarGDone, 1);
        mbar_init(bars + 8 * kBarItemDone, 1);
        mbar_init(bars + 8 * kBarAccFree, kStoreWarps);
        for (int i = 0; i < kMmaWarps; ++i) mbar_init(bars + 8 * (kBarFinal + i), 1);
        for (int i = 0; i < kSchedDepth; ++i) {
            mbar_init(bars + 8 * (kBarSchedFull + i), 1);
            mbar_init(bars + 8 * (kBarSchedEmpty + i), kSchedReaders);
        }
        *s_abort = 0;
        fence_mbar_init();
    }
    if (tid < 256) {  // (1, 1, 1, 0 ..) and zeros: the parts of the additional K step that do not change
        *reinterpret_cast<uint4 *>(sm + kOffOnes + 16 * tid) = tid < 128 ? make_uint4(0x3f803f80u, 0x3f80u, 0u, 0u) : make_uint4(0u, 0u, 0u, 0u);
        fence_proxy_async();
    }
    if (warp == kMmaWarp) {
        tmem_alloc(smem_u32((const void *)tmem_slot), 512);
        tmem_relinquish();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = __shfl_sync(0xffffffffu, *tmem_slot, 0);

    // The set-up, here and in every role, may run while the kernel before still does.  Each role then waits for its end
    // (wait_prior_grid), in front of its first bounded wait: those count this kernel's own time only, and what
    // they guard comes from that kernel.

#ifdef MATE_TRACE
    long long tr[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    const long long tr_start = clock64();
#endif
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
    if (warp < kComputeWarps) {
        // ------------------------------------------------------------------ arithmetic + epilogue
        reg_alloc<Regs<kByMma>::kCompute>();
        const int r = tid & 127;   // row of the tile = lane of tensor memory
        const int cq = warp >> 2;  // takes the chunks cq and cq + 2 of a column tile
        const uint32_t tm = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        const uint64_t scale2 = pack_f32x2(p.scale_log2, p.scale_log2);
        uint32_t c_cnt = 0;  // tiles so far
        bool alive = true;
        wait_prior_grid();
        auto gradients_done = [&]() {  // of every tile so far (at once when there is none)
            alive = wait(bars + 8 * kBarGDone, (c_cnt - 1) & 1);
            tc_fence_after();
        };

#pragma unroll 1
        for (uint32_t n = 0; alive; ++n) {
            const int slot = n % kSchedDepth, rb = RowRing::buffer(n);
            if (!wait(bars + 8 * (kBarSchedFull + slot), (n / kSchedDepth) & 1)) break;
            // The record and the row data stay in shared memory until the item's last tile: what is needed of them is
            // read where it is needed (registers are what this role is short of).
            const FwdUnit &un = s_item[slot];
            if (un.rows == 0) break;
            const bool key_side = un.ws_off == 0;
            const ItemTiles tiles(un);
            if (!(alive = wait(bars + 8 * (kBarRFull + rb), RowRing::full_parity(n)))) break;
            // this row's data (rows past the end shadow the last one)
            const uint32_t meta = base + kOffMeta + (rb * 5 * kTile + min(r, un.rows_of(0) - 1)) * 4;
            const int w_lo_max = __reduce_max_sync(0xffffffffu, ld_shared_s32(meta + kTile * 4)),
                      w_hi_min = __reduce_min_sync(0xffffffffu, ld_shared_s32(meta + 2 * kTile * 4));

            // the tile loop is compiled once per side
            auto tile_loop = [&](auto side) {
                constexpr bool kKeySide = decltype(side)::value;
                uint64_t row_nlse2 = 0ull, row_D2 = 0ull;
                if (!kKeySide) {
                    const float nlse = __int_as_float(ld_shared_s32(meta + 3 * kTile * 4)), D = __int_as_float(ld_shared_s32(meta + 4 * kTile * 4));
                    row_nlse2 = pack_f32x2(nlse, nlse);
                    row_D2 = pack_f32x2(D, D);
                }
                TileInfo t = tiles.tile(0);
#pragma unroll 1
                for (int i = 0; i < tiles.n; ++i) {
                    const bool full = t.w == kTile && (t.pre == kTile || (w_lo_max - t.k0 <= t.pre && w_hi_min - t.k0 >= kTile));
                    const uint32_t vec = base + kOffExt + ColRing::buffer(c_cnt) * 4096;
                    TR_T0(t_ws);
                    if (!(alive = wait(bars + 8 * kBarSFull, c_cnt & 1))) break;
                    tc_fence_after();
                    TR_ADD(0, t_ws);
                    TR_T0(t_cmp);
                    auto release_st = [&]() {  // S and dP may be overwritten
                        tc_fence_before();
                        if (lane == 0) mbar_arrive(bars + 8 * kBarSTFree);
                    };
                    uint32_t pk_p[16], pk_ds[16];
                    if (full) {
                        uint32_t sv[2][32], tv[2][32];
#pragma unroll
                        for (int cc = 0; cc < 2; ++cc) {
                            tmem_ld32(tm + kTmS + cq * 32 + cc * 64, sv[cc]);
                            tmem_ld32(tm + kTmT + cq * 32 + cc * 64, tv[cc]);
                        }
                        tc_wait_ld();
#pragma unroll
                        for (int cc = 0; cc < 2; ++cc) {
                            reg_fence(sv[cc]);
                            reg_fence(tv[cc]);
                        }
                        release_st();
                        TR_ADD(4, t_cmp);
                        math32<kKeySide, false, kByMma>(sv[0], tv[0], scale2, row_nlse2, row_D2, vec + cq * 128, 0u, pk_p, pk_ds);
                        TR_T0(t_wa);
                        gradients_done();  // of the tile before: the operand columns are free
                        TR_ADD(1, t_wa);
                        if (kKeySide) tmem_st16(tm + kTmA1 + cq * 16, pk_p);
                        tmem_st16(tm + (kKeySide ? kTmA2 : kTmA1) + cq * 16, pk_ds);
                        math32<kKeySide, false, kByMma>(sv[1], tv[1], scale2, row_nlse2, row_D2, vec + 256 + cq * 128, 0u, pk_p, pk_ds);
                        if (kKeySide) tmem_st16(tm + kTmA1 + cq * 16 + 32, pk_p);
                        tmem_st16(tm + (kKeySide ? kTmA2 : kTmA1) + cq * 16 + 32, pk_ds);
                    } else {
                        // this row counts the columns [0, pre) and [r_lo, r_hi); some row of the warp counts columns only
                        // there and within [e_lo, e_hi)
                        const int r_lo = t.is_b ? ld_shared_s32(meta + kTile * 4) - t.k0 : 0, r_hi = t.is_b ? min(ld_shared_s32(meta + 2 * kTile * 4) - t.k0, t.w) : 0;
                        const int e_lo = __reduce_min_sync(0xffffffffu, r_lo), e_hi = __reduce_max_sync(0xffffffffu, r_hi);
                        const int e_end = max(t.pre, e_hi > e_lo ? e_hi : 0);
                        bool held = true, a_free = false;
#pragma unroll 1
                        for (int cb = cq * 32; cb < t.w; cb += 64) {
                            if (cb >= t.pre && (cb + 32 <= e_lo || cb >= e_hi)) {  // no row of the warp has a pair here
#pragma unroll
                                for (int e = 0; e < 16; ++e) pk_p[e] = pk_ds[e] = 0u;
                            } else {
                                uint32_t sv[32], tv[32];
                                tmem_ld32(tm + kTmS + cb, sv);
                                tmem_ld32(tm + kTmT + cb, tv);
                                tc_wait_ld();
                                reg_fence(sv);
                                reg_fence(tv);
                                if (cb + 64 >= e_end) {  // read for the last time
                                    release_st();
                                    held = false;
                                }
                                math32<kKeySide, true, kByMma>(sv, tv, scale2, row_nlse2, row_D2, vec + 4 * cb,
                                                               bits_below(t.pre - cb) | (bits_below(r_hi - cb) & ~bits_below(r_lo - cb)), pk_p, pk_ds);
                            }
                            if (!a_free) gradients_done();
                            a_free = true;
                            if (kKeySide) tmem_st16(tm + kTmA1 + (cb >> 1), pk_p);
                            tmem_st16(tm + (kKeySide ? kTmA2 : kTmA1) + (cb >> 1), pk_ds);
                        }
                        if (held) release_st();
                        // Also when nothing was written: keeps this warp's arrival below out of the barrier phase of the
                        // previous tile, which a slower warp may not have reached yet.
                        if (!a_free) gradients_done();
                    }
                    if (!alive) break;
                    ++c_cnt;
                    TR_T0(t_st);
                    tc_wait_st();
                    tc_fence_before();
                    if (lane == 0) mbar_arrive(bars + 8 * kBarAFull);
                    TR_ADD(6, t_st);
                    TR_ADD(2, t_cmp);
                    TR_INC(7);
                    t = tiles.tile(i + 1);
                }
            };
            if (key_side) tile_loop(std::true_type{});
            else tile_loop(std::false_type{});
            if (!alive) break;
            __syncwarp();
            if (lane == 0) {
                mbar_arrive(bars + 8 * (kBarREmpty + rb));
                mbar_arrive(bars + 8 * (kBarSchedEmpty + slot));
            }
        }
    } else if (warp < kMmaWarp) {
        // ------------------------------------------------------------------ gradients: tensor memory -> original positions
        reg_dealloc<Regs<kByMma>::kStore>();
        const int q4 = warp - kStoreWarp0;  // rows 32 q4 .. of the tile = lanes of tensor memory this warp can read
        static_assert(kStoreWarp0 % 4 == 0, "warp w reads the lanes 32 (w % 4) ..");
        const uint32_t acc = tmem + ((uint32_t)(q4 * 32) << 16) + kTmAcc1;
        uint8_t *stage = sm + kOffStage + q4 * 2048;
        uint32_t units = 0;
        wait_prior_grid();
#pragma unroll 1
        for (uint32_t n = 0;; ++n) {
            const int slot = n % kSchedDepth, rb = RowRing::buffer(n);
            if (!wait(bars + 8 * (kBarSchedFull + slot), (n / kSchedDepth) & 1)) break;
            const FwdUnit &un = s_item[slot];
            if (un.rows == 0) break;
            const bool key_side = un.ws_off == 0, any = ItemTiles(un).n > 0;
            const int rows_h = un.rows_of(0), pass = p.pass(un.view());
            const size_t at = p.tr.base(un.b, un.head()) * 64;
            __syncwarp();
            if (lane == 0) mbar_arrive(bars + 8 * (kBarSchedEmpty + slot));
            if (!wait(bars + 8 * (kBarRFull + rb), RowRing::full_parity(n))) break;
            const int r = q4 * 32 + lane;
            const int dst_row = r < rows_h ? (reinterpret_cast<const int32_t *>(sm + kOffMeta) + rb * 5 * kTile)[r] : -1;
            __syncwarp();
            if (lane == 0) mbar_arrive(bars + 8 * (kBarREmpty + rb));
            if (any) {
                if (!wait(bars + 8 * kBarItemDone, units++ & 1)) break;
                tc_fence_after();
            }
            // key side: dV, dK; query side: dQ.  32 columns at a time through the staging area, so that a store writes
            // 64 consecutive bytes of eight rows.
            const int n_c = key_side ? 4 : 2;
#pragma unroll 1
            for (int c = 0; c < n_c; ++c) {
                const float mul = key_side && c < 2 ? 1.f : p.scale;
                uint32_t o[32];
                if (any) {
                    tmem_ld32(acc + c * 32, o);
                    tc_wait_ld();
                    reg_fence(o);
                    if (c + 1 == n_c) {  // read for the last time
                        tc_fence_before();
                        if (lane == 0) mbar_arrive(bars + 8 * kBarAccFree);
                    }
                } else {  // rows without any pair (possible in the passes of the row-or-column pattern)
#pragma unroll
                    for (int e = 0; e < 32; ++e) o[e] = 0u;
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    uint32_t w4[4];
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        w4[e] = cvt_bf16x2(__uint_as_float(o[8 * j + 2 * e]) * mul, __uint_as_float(o[8 * j + 2 * e + 1]) * mul);
                    *reinterpret_cast<uint4 *>(stage + lane * 64 + ((j ^ ((lane >> 1) & 3)) << 4)) = make_uint4(w4[0], w4[1], w4[2], w4[3]);
                }
                __syncwarp();
                __nv_bfloat16 *out = (key_side ? (c < 2 ? p.dV[pass] : p.dK[pass]) : p.dQ[pass]) + at + (c & 1) * 32;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int row = 8 * i + (lane >> 2), j = lane & 3;
                    const int dr = __shfl_sync(0xffffffffu, dst_row, row);
                    const uint4 x = *reinterpret_cast<const uint4 *>(stage + row * 64 + ((j ^ ((row >> 1) & 3)) << 4));
                    if (dr >= 0) *reinterpret_cast<uint4 *>(out + (size_t)dr * 64 + j * 8) = x;
                }
                __syncwarp();
            }
        }
    } else if (warp < kLoadWarp0) {
        // ------------------------------------------------------------------ MMA issuers, padding rows
        // One warp issues S and dP of the tiles, the other the gradient MMAs, each as soon as what it needs is there.  The
        // whole warp runs the control flow and one lane issues; votes and shuffles keep conditions and operands
        // warp-uniform (an MMA with other operands takes 51 clk to issue, more than a gradient MMA takes to run).
        reg_dealloc<Regs<kByMma>::kMma>();
        if (warp < kMmaWarp + kMmaWarps) {
            const bool leader = elect_one();
            const bool grad = warp != kMmaWarp;
            uint32_t c_cnt = 0, units = 0;  // tiles, items with a tile
            wait_prior_grid();
            auto wait_u = [&](uint32_t bar, uint32_t parity) -> bool {
#pragma unroll 1
                for (uint32_t it = 0; it < kWaitLimit; ++it) {
                    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
                    if (__any_sync(0xffffffffu, *s_abort)) return false;
                }
                *s_abort = 1;
                return false;
            };
            bool alive = true;
#pragma unroll 1
            for (uint32_t n = 0; alive; ++n) {
                const int slot = n % kSchedDepth, rb = RowRing::buffer(n);
                if (!wait_u(bars + 8 * (kBarSchedFull + slot), (n / kSchedDepth) & 1)) break;
                const FwdUnit &un = s_item[slot];
                auto uniform = [&](int x) { return __shfl_sync(0xffffffffu, x, 0); };
                const int rows = uniform(un.rows), len_a = uniform(max(un.kA_end - un.kA0, 0)), len_b = uniform(un.kP() + un.kB_end - un.kB0);
                const bool key_side = uniform(un.ws_off) == 0;
                __syncwarp();
                if (lane == 0) mbar_arrive(bars + 8 * (kBarSchedEmpty + slot));
                if (rows == 0) break;
                const int nA = (len_a + kTile - 1) / kTile, n_tiles = nA + (len_b + kTile - 1) / kTile;
                auto steps = [&](int i) { return (min(i < nA ? len_a - i * kTile : len_b - (i - nA) * kTile, kTile) + 15) >> 4; };  // of 16 columns
                if (!grad) {
                    if (!(alive = wait_u(bars + 8 * (kBarRFull + rb), RowRing::full_parity(n)))) break;
                    fence_proxy_async();
                    const uint32_t ra = smem_desc_lo(base + kOffR) + rb * ((2 * kTileBytes) >> 4), rbb = ra + (kTileBytes >> 4);
                    const uint32_t ones = smem_desc_lo_rows16(base + kOffOnes, base + kOffZero);
#pragma unroll 1
                    for (int i = 0; i < n_tiles; ++i, ++c_cnt) {
                        const uint32_t st = ColRing::buffer(c_cnt);
                        const uint32_t idesc = idesc_bf16(128, 0, 0, 0) | (uint32_t)steps(i) << 18;  // N = 16 columns per step
                        const uint32_t ca = smem_desc_lo(base + kOffC) + st * ((2 * kTileBytes) >> 4), cb = ca + (kTileBytes >> 4);
                        const uint32_t tS = tmem + kTmS, tT = tmem + kTmT, ext = base + kOffExt + st * 4096;
                        if (!(alive = wait_u(bars + 8 * (kBarCFull + st), ColRing::full_parity(c_cnt)))) break;  // the tile has landed
                        fence_proxy_async();  // the copies of 16 bytes come through the generic proxy
                        // the tile before sits in registers (parity 1 of a barrier without a phase behind it: at once)
                        if (!(alive = wait_u(bars + 8 * kBarSTFree, (c_cnt - 1) & 1))) break;
                        tc_fence_after();
                        if (leader) {
                            mma_ss_lean<0>(tS, ra, ca, idesc);  // S = Ra Ca^T, K = 64 as four steps of 16
                            mma_ss_lean<1>(tS, ra + 2, ca + 2, idesc);
                            mma_ss_lean<1>(tS, ra + 4, ca + 4, idesc);
                            mma_ss_lean<1>(tS, ra + 6, ca + 6, idesc);
                            mma_ss_lean<0>(tT, rbb, cb, idesc);  // dP = Rb Cb^T
                            mma_ss_lean<1>(tT, rbb + 2, cb + 2, idesc);
                            mma_ss_lean<1>(tT, rbb + 4, cb + 4, idesc);
                            mma_ss_lean<1>(tT, rbb + 6, cb + 6, idesc);
                            if (kByMma && key_side) {  // - LSE / scale and - D of the columns: ones x (three bf16 per column)
                                mma_ss_rows16(tS, ones, smem_desc_lo_rows16(ext, base + kOffZero), idesc);
                                mma_ss_rows16(tT, ones, smem_desc_lo_rows16(ext + 2048, base + kOffZero), idesc);
                            }
                            mma_commit(bars + 8 * kBarSFull);
                        }
                        __syncwarp();
                    }
                    if (!alive) break;
                    if (leader) mma_commit(bars + 8 * (kBarREmpty + rb));  // the row operands are free once these MMAs are done
                    __syncwarp();
                } else {
                    constexpr uint32_t idesc = idesc_bf16(128, 64, 0, 1);  // B = 16 rows of the column tile x 64, MN-major
                    constexpr uint32_t kStep = (16 * kRowBytes) >> 4;      // 16 rows of the column tile
                    // the accumulators are free once the gradients of the item before are in the store warps' registers
                    if (n_tiles > 0 && !(alive = wait_u(bars + 8 * kBarAccFree, (units++ - 1) & 1))) break;
                    const uint32_t tA1 = tmem + kTmA1, tA2 = tmem + kTmA2, tG1 = tmem + kTmAcc1, tG2 = tmem + kTmAcc2;
#pragma unroll 1
                    for (int i = 0; i < n_tiles; ++i, ++c_cnt) {
                        const uint32_t st = ColRing::buffer(c_cnt);
                        const int ks = steps(i);
                        const uint32_t a_lo = smem_desc_lo(base + kOffC) + st * ((2 * kTileBytes) >> 4), b_lo = a_lo + (kTileBytes >> 4);
                        if (!(alive = wait_u(bars + 8 * kBarAFull, c_cnt & 1))) break;
                        tc_fence_after();
                        if (leader) {
                            if (key_side) {
                                mma_ts_lean_flag(tG1, tA1, b_lo, idesc, i > 0);  // dV += P^T dO
                                mma_ts_lean_flag(tG2, tA2, a_lo, idesc, i > 0);  // dK += dS^T Q
#pragma unroll 1
                                for (int k = 1; k < ks; ++k) {
                                    mma_ts_lean<1>(tG1, tA1 + 8 * k, b_lo + k * kStep, idesc);
                                    mma_ts_lean<1>(tG2, tA2 + 8 * k, a_lo + k * kStep, idesc);
                                }
                            } else {
                                mma_ts_lean_flag(tG1, tA1, a_lo, idesc, i > 0);  // dQ += dS K
#pragma unroll 1
                                for (int k = 1; k < ks; ++k) mma_ts_lean<1>(tG1, tA1 + 8 * k, a_lo + k * kStep, idesc);
                            }
                            mma_commit(bars + 8 * kBarGDone);
                            mma_commit(bars + 8 * (kBarCEmpty + st));
                            if (i + 1 == n_tiles) mma_commit(bars + 8 * kBarItemDone);
                        }
                        __syncwarp();
                    }
                }
            }
            // nothing of this CTA may still run on the tensor pipe when tensor memory is freed
            if (leader) mma_commit(bars + 8 * (kBarFinal + grad));
            __syncwarp();
            mbar_wait_bounded(bars + 8 * (kBarFinal + grad), 0, kWaitLimit);
        } else {
            // padding rows: zero gradients.  (Not by the store warps: until a CTA's padding is done they would hold back rows,
            // records and accumulators.)
            wait_prior_grid();
#pragma unroll 1
            for (int c = blockIdx.x; c < p.n_pads; c += gridDim.x) {
                const PadChunk pc = p.pads[c];
                const ViewPlan &vp = p.view[pc.view()];
                const int pass = p.pass(pc.view()), i = (warp - kPadWarp0) * 32 + lane;
                int row = i < pc.n ? __ldg(vp.perm + (size_t)pc.b * p.N + pc.t0 + i) : -1;  // one look-up a chunk, a row per lane
                if (row >= 0 && !p.tr.exists(pc.b, row)) row = -1;
                const size_t at = p.tr.base(pc.b, pc.head()) * 64 + (lane & 7) * 8;
#pragma unroll 1
                for (int k = lane >> 3; k < 32; k += 4) {  // eight lanes per row
                    const int r = __shfl_sync(0xffffffffu, row, k);
                    if (r < 0) continue;
                    const size_t o = at + (size_t)r * 64;
                    *reinterpret_cast<uint4 *>(p.dQ[pass] + o) = make_uint4(0, 0, 0, 0);
                    *reinterpret_cast<uint4 *>(p.dK[pass] + o) = make_uint4(0, 0, 0, 0);
                    *reinterpret_cast<uint4 *>(p.dV[pass] + o) = make_uint4(0, 0, 0, 0);
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ loaders
        reg_dealloc<Regs<kByMma>::kLoad>();
        wait_prior_grid();
        const int lw = warp - kLoadWarp0;
        const bool leader = elect_one();
        uint32_t c_cnt = 0;
        bool alive = true;
#pragma unroll 1
        for (uint32_t n = 0; alive; ++n) {
            const int slot = n % kSchedDepth, rb = RowRing::buffer(n);
            if (warp == kLoadWarp0) {
                if (!wait(bars + 8 * (kBarSchedEmpty + slot), ((n / kSchedDepth) & 1) ^ 1)) break;
                if (lane < 4) reinterpret_cast<int4 *>(s_item + slot)[lane] = rec;
                __syncwarp();
                if (lane == 0) mbar_arrive(bars + 8 * (kBarSchedFull + slot));  // release: the record is visible to the readers
            }
            if (!wait(bars + 8 * (kBarSchedFull + slot), (n / kSchedDepth) & 1)) break;
            const FwdUnit un = s_item[slot];
            __syncwarp();
            if (lane == 0) mbar_arrive(bars + 8 * (kBarSchedEmpty + slot));
            if (un.rows == 0) break;
            const bool key_side = un.ws_off == 0;
            const ItemTiles tiles(un);
            const int rows_h = un.rows_of(0);
            const ViewPlan &vp = p.view[un.view()];
            const size_t bn = (size_t)un.b * p.N;
            const int32_t *perm = vp.perm + bn;
            const size_t bh = p.tr.base(un.b, un.head());
            // column tiles inside [0, ident) of the order are contiguous in the tensors (see bulk_tile)
            const int ident = p.bulk ? __ldg(vp.ident + un.b) : 0;
            // step -1: the row operands and row data; steps 0 ..: the column tiles
            const int rr = 32 * lw + lane;  // this lane's row of a tile
            auto step_idx = [&](int i) {  // as a row of the tensors
                const TileInfo t = tiles.tile(max(i, 0));
                return (uint32_t)bh + (uint32_t)__ldg(perm + (i < 0 ? un.q0 + min(rr, rows_h - 1) : t.pos(min(rr, t.w - 1))));
            };
            uint32_t next = step_idx(-1);
#pragma unroll 1
            for (int i = -1; i < tiles.n; ++i) {
                const uint32_t now = next;
                if (i + 1 < tiles.n) next = step_idx(i + 1);
                const TileInfo t = tiles.tile(max(i, 0));
                const uint32_t c = c_cnt + max(i, 0), st = ColRing::buffer(c);
                const uint32_t bar_full = bars + 8 * (i < 0 ? kBarRFull + rb : kBarCFull + st);
                if (!(alive = wait(bars + 8 * (i < 0 ? kBarREmpty + rb : kBarCEmpty + st),
                                   i < 0 ? RowRing::wait_parity(n) : ColRing::wait_parity(c)))) break;
                if (i < 0) {  // row data for the arithmetic threads
                    if (rr < rows_h) {
                        const uint32_t meta = base + kOffMeta + rb * 5 * kTile * 4 + rr * 4;
                        const size_t at = bn + un.q0 + rr;
                        cp_async4(meta, vp.perm + at);
                        cp_async4(meta + kTile * 4, vp.seg_lo + at);
                        cp_async4(meta + 2 * kTile * 4, vp.seg_hi + at);
                        if (!key_side) {
                            cp_async4(meta + 3 * kTile * 4, p.nlse + now);
                            cp_async4(meta + 4 * kTile * 4, p.D + now);
                        }
                    }
                } else if (key_side) {  // column data
                    const uint32_t ext = base + kOffExt + st * 4096;
                    if (kByMma) {
                        cp_async16(ext + rr * 16, p.ext + 2 * (size_t)now);
                        cp_async16(ext + 2048 + rr * 16, p.ext + 2 * (size_t)now + 1);
                    } else {
                        cp_async4(ext + rr * 4, p.nlse + now);
                        cp_async4(ext + 512 + rr * 4, p.D + now);
                    }
                }
                const uint32_t dst = base + (i < 0 ? kOffR + rb * 2 * kTileBytes : kOffC + st * 2 * kTileBytes);
                const bool kv = (i < 0) == key_side;  // K and V, or Q and dO
                const bool bulk = i >= 0 && bulk_tile(t, ident);
                // (the row operands' rows past the last one are never looked at: their results are not stored)
                if (!bulk) {
                    const uint8_t *a = reinterpret_cast<const uint8_t *>(kv ? p.K : p.Q), *b = reinterpret_cast<const uint8_t *>(kv ? p.V : p.dO);
                    gather_rows(dst, a, true, b - a, now, i < 0 ? rows_h : (t.w + 15) & ~15, lw, lane);
                }
                cp_async_arrive(bar_full);
                __syncwarp();
                if (bulk && lw == 0) {
                    if (leader) {
                        mbar_arrive_expect_tx(bar_full, 2 * kTileBytes);
                        tma_load_2d(dst, kv ? &p.tmK : &p.tmQ, 0, (int)bh + t.first(), bar_full);
                        tma_load_2d(dst + kTileBytes, kv ? &p.tmV : &p.tmdO, 0, (int)bh + t.first(), bar_full);
                    }
                    __syncwarp();
                } else if (lane == 0) {
                    mbar_arrive(bar_full);
                }
            }
            if (warp == kLoadWarp0) {
                claim();
                fetch_record();
            }
            c_cnt += tiles.n;
        }
    }

#ifdef MATE_TRACE
    if (lane == 0 && (warp == 0 || warp == 4 || warp == kMmaWarp || warp == kLoadWarp0) && blockIdx.x < kTraceCtas) {
        const int role = warp == 0 ? 0 : warp == 4 ? 1 : warp == kMmaWarp ? 2 : 3;
        long long *o = g_trace_bwd + blockIdx.x * 32 + role * 8;
        for (int i = 0; i < 8; ++i) o[i] = tr[i];
        if (role == 0) o[5] = clock64() - tr_start;
    }
#endif
    if (*s_abort)  // copies may still be on their way to shared memory: they take a few microseconds
        for (int i = 0; i < 50; ++i) __nanosleep(1000);
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && *s_abort) atomicOr(p.status + 1, 1);
    if (warp == kMmaWarp) tmem_dealloc(tmem, 512);
}


inline size_t align256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

// workspace, by rows of the tensors: [256 B counters][D: a float each][-LSE log2 e: a float][the key side's column data: 32 B]
size_t tc_bwd_workspace(const mate_plan_t *plan) {
    const size_t rows = plan->n_rows();
    return 256 + 2 * align256(rows * sizeof(float)) + rows * 32;
}

namespace {
// Whether -LSE / scale is a number that three bf16 hold: with smaller scales (0 among them) it overflows, with larger ones the lowest
// of the three comes close to the smallest bf16, 2^-133.  Any other scale takes the kernel that does not divide.
bool divides(float scale) { return fabsf(scale) >= 0x1p-100f && fabsf(scale) <= 0x1p100f; }

template <bool kMany, bool kByMma>
int launch(const mate_plan_t *plan, const void *Q, const void *K, const void *V, const void *O,
           const float *LSE, const void *dO, float scale, void *const (&dQ)[kPasses], void *const (&dK)[kPasses],
           void *const (&dV)[kPasses], void *workspace, cudaStream_t stream) {
    static SmemAttrOnce attr;
    if (plan->bwd_grid == 0) return MATE_OK;
    if (attr.ensure((const void *)tc_bwd_kernel<kMany, kByMma>, (int)kSmemBytes, plan->device) != MATE_OK) return MATE_ERR_CUDA;
    const size_t rows = plan->n_rows();
    uint8_t *ws = (uint8_t *)workspace;
    float *D = (float *)(ws + 256);
    const size_t row_floats = align256(rows * sizeof(float)) / sizeof(float);
    float *nlse = D + row_floats;
    uint4 *ext = (uint4 *)(nlse + row_floats);
    Params<kMany> p;
    p.bulk = rows < (size_t(1) << 31) && make_row_map(&p.tmQ, Q, rows) && make_row_map(&p.tmK, K, rows) &&
             make_row_map(&p.tmV, V, rows) && make_row_map(&p.tmdO, dO, rows);
    p.Q = (const __nv_bfloat16 *)Q;
    p.K = (const __nv_bfloat16 *)K;
    p.V = (const __nv_bfloat16 *)V;
    p.dO = (const __nv_bfloat16 *)dO;
    p.nlse = nlse;
    p.D = D;
    p.ext = ext;
    for (int i = 0; i < p.kO; ++i) {
        p.dQ[i] = (__nv_bfloat16 *)dQ[i];
        p.dK[i] = (__nv_bfloat16 *)dK[i];
        p.dV[i] = (__nv_bfloat16 *)dV[i];
    }
    for (int v = 0; v < p.kV; ++v) p.view[v] = plan->work_view(v);
    p.units = plan->bwd_units_dev;
    p.n_units = plan->n_bwd_units;
    p.N = plan->N;
    p.H = plan->H;
    p.pads = plan->pads_dev;
    p.n_pads = plan->n_pads;
    p.tr = plan->rows();
    p.scale = scale;
    p.scale_log2 = scale * 1.4426950408889634f;
    p.status = plan->status_dev;
    p.counter = (int32_t *)ws;

    const auto rowdot = [&](auto n) {
        constexpr int kRows = decltype(n)::value;
        return launch_after(rowdot_kernel<kRows>, dim3((unsigned)((rows + 32 * kRows - 1) / (32 * kRows))), 256, 0, stream, (const __nv_bfloat16 *)dO,
                            (const __nv_bfloat16 *)O, LSE, D, nlse, ext, scale, rows, (int32_t *)ws);
    };
    // As few rows per thread as bring all blocks onto the GPU at once.  (Twice as many between 28,416 and 37,888 and between 56,832
    // and 75,776 rows, as for six blocks of each kind to an SM: backward of 4 x 680 tokens 19.1 us, 18.4 by this rule, 4 x 1400 32.1, 30.9.)
    const auto at_once = [&](int n) { return rows <= (size_t)std::max(plan->n_ctas, 1) * kRowdotBlocks * 32 * n; };
    if ((at_once(1) ? rowdot(std::integral_constant<int, 1>{}) : at_once(2) ? rowdot(std::integral_constant<int, 2>{})
                                                                            : rowdot(std::integral_constant<int, 4>{})) != cudaSuccess)
        return MATE_ERR_CUDA;
    return launch_after(tc_bwd_kernel<kMany, kByMma>, dim3((unsigned)plan->bwd_grid), kThreads, kSmemBytes, stream, p) == cudaSuccess ? MATE_OK : MATE_ERR_CUDA;
}

}  // namespace

int tc_bwd(const mate_plan_t *plan, const void *Q, const void *K, const void *V, const void *O,
           const float *LSE, const void *dO, float scale, void *const (&dQ)[kPasses], void *const (&dK)[kPasses],
           void *const (&dV)[kPasses], void *workspace, cudaStream_t stream) {
    const auto run = [&](auto many, auto by_mma) {
        return launch<many(), by_mma()>(plan, Q, K, V, O, LSE, dO, scale, dQ, dK, dV, workspace, stream);
    };
    const std::true_type yes;
    const std::false_type no;
    return plan->sub[0] ? (divides(scale) ? run(yes, yes) : run(yes, no)) : (divides(scale) ? run(no, yes) : run(no, no));
}

}  // namespace mate

#ifdef MATE_TRACE
// copies the cycle counters of the last backward launch to the host: [kTraceCtas CTAs][4 roles][8]
extern "C" int mate_debug_trace_bwd(long long *host_out) {
    return cudaMemcpyFromSymbol(host_out, mate::g_trace_bwd, sizeof(long long) * mate::kTraceCtas * 32) == cudaSuccess ? 0 : -4;
}
#endif
