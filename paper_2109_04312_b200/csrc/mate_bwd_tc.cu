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
// One persistent, warp-specialised CTA per SM (16 warps); work items (unit, side) are handed out through a
// counter, longest first.
//   warps 0-7   arithmetic: two threads (r, r + 128) share row r of the 128-row tile, the lane of
//               tensor memory; each takes every other chunk of 32 columns.  S and dP (fp32) come out of
//               tensor memory, P / dS (bf16 pairs) go back into it as MMA operands.
//   warp  8     issues every tcgen05.mma (one elected lane): S and dP of tile n + 1 as soon as those of
//               tile n sit in registers, ahead of the gradient MMAs of tile n
//   warps 9-11  zero gradients of the padding rows
//   warps 12-15 loaders: gather rows by view-order index with 16-byte cp.async into 128-byte swizzled
//               shared memory, or fetch a column tile whose rows lie in place in the tensors by one bulk
//               tensor copy per matrix (row operands double buffered, column tiles in a ring of 4)
// What bounds it: the exponentials, 1024 clk per 128 x 128 tile and side (16 per clock and SM), as far as the
// rest hides behind them.  A tile that counts in full is taken into registers whole (64 columns of S and of
// dP per thread), which frees S and dP for the next tile's MMAs before the arithmetic begins; the
// operand columns are waited for behind the first chunk's arithmetic.  Waits and rare paths are rolled (the
// instruction cache holds about 32 KB).  The gradients accumulate in tensor memory and are scattered to the
// rows' original positions in the epilogue, through a staging area so that stores cover whole sectors.
#include <cuda.h>
#include <cuda_bf16.h>

#include <type_traits>

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
constexpr int kMmaWarp = kComputeWarps;
constexpr int kPadWarp0 = kMmaWarp + 1;
constexpr int kPadWarps = 3;
constexpr int kLoadWarp0 = kPadWarp0 + kPadWarps;
constexpr int kLoadWarps = 4;
constexpr int kThreads = 32 * (kLoadWarp0 + kLoadWarps);
// registers per thread after the roles have split: 256 x 168 + 256 x 88 = 65,536 = the 512 x 128 the CTA is
// launched with
constexpr int kRegsCompute = 168, kRegsOther = 88;
constexpr int kStages = 4;  // ring of column tiles
constexpr int kLag = 2;     // loader: copy groups in flight behind the newest one
constexpr int kSchedDepth = 4;
constexpr uint32_t kOffR = 0;                                    // [2 buffers] x (Ra: Q or K, Rb: dO or V), 16 KB each
constexpr uint32_t kOffC = 4 * kTileBytes;                       // [kStages] x (Ca 16 KB, Cb 16 KB)
constexpr uint32_t kOffVec = kOffC + kStages * 2 * kTileBytes;   // [kStages] x 128 x (-LSE log2 e), 128 x D
constexpr uint32_t kOffMeta = kOffVec + kStages * 1024;          // [2 buffers] x (perm, seg_lo, seg_hi, -LSE log2 e, D) of 128 rows
constexpr uint32_t kOffStage = kOffMeta + 2 * 5 * kTile * 4;     // [arithmetic warps] x 32 rows x 64 bytes
constexpr uint32_t kOffItem = kOffStage + kComputeWarps * 2048;  // [kSchedDepth] unit records
constexpr uint32_t kOffBar = kOffItem + kSchedDepth * sizeof(FwdUnit);
constexpr uint32_t kSmemBytes = kOffBar + 256 + 1024;            // + slack for the 1024-byte alignment
static_assert(kSmemBytes <= 232448, "shared memory per CTA");
// barrier slots (8 bytes each) behind kOffBar
enum {
    kBarRFull = 0,    // [2] loaders -> MMA, arithmetic      (count: loader warps)
    kBarREmpty = 2,   // [2] MMA commit and arithmetic warps (row data read) -> loaders (count 1 + kComputeWarps)
    kBarCFull = 4,    // [kStages] loaders -> MMA            (count: loader warps)
    kBarCEmpty = 8,   // [kStages] MMA commit -> loaders     (count 1)
    kBarSFull = 12,   // MMA commit -> arithmetic: S and dP of a tile are complete (count 1)
    kBarAFull = 13,   // arithmetic -> MMA: the bf16 operands of a tile are written (count: one per warp)
    kBarGDone = 14,   // MMA commit -> arithmetic: the gradient MMAs of a tile are complete (count 1)
    kBarFinal = 15,
    kBarSchedFull = 16,   // [kSchedDepth] scheduler -> every warp (count 1)
    kBarSchedEmpty = 20,  // [kSchedDepth] every warp -> scheduler (count kSchedReaders)
    kBarSTFree = 24,      // arithmetic -> MMA: S and dP of a tile are in registers (count: one per warp)
    kNumBars = 25
};
constexpr int kSchedReaders = kComputeWarps + 1 + kLoadWarps;
// tensor memory columns
constexpr uint32_t kTmS = 0, kTmT = 128, kTmA1 = 256, kTmA2 = 320, kTmAcc1 = 384, kTmAcc2 = 448;
constexpr uint32_t kWaitLimit = 4096;  // tries (about 5 us each) before a wait gives up

struct Params {
    CUtensorMap tmQ, tmK, tmV, tmdO;  // boxes of 128 rows, 128-byte swizzle
    int use_tma;                      // 0: every tile is gathered row by row
    const __nv_bfloat16 *Q, *K, *V, *dO;
    const float *nlse, *D;  // per row, original order: -LSE log2 e, D
    __nv_bfloat16 *dQ, *dK, *dV;
    ViewPlan rowv, colv;
    const uint8_t *head_view;
    const FwdUnit *units;  // one half each; item = 2 unit + (0 key side, 1 query side)
    int n_units, N, H;
    const PadChunk *pads;
    int n_pads;
    TensorRows tr;         // where (example, head) starts in the tensors
    float scale, scale_log2;
    int32_t *status;
    int32_t *counter;      // next work item (zeroed before the launch)
};

// D_k = sum_e dO_ke O_ke and -LSE_k log2 e per row (original order), d = 64: eight threads per row, 16 bytes
// of each tensor per thread, two rows per thread in flight.  HBM-bound.  The first block also clears the
// work-item counters of the kernels that follow.
constexpr int kRowdotRows = 64;  // per block
__global__ void __launch_bounds__(256) rowdot_kernel(const __nv_bfloat16 *__restrict__ dO, const __nv_bfloat16 *__restrict__ O,
                                                     const float *__restrict__ LSE, float *__restrict__ D,
                                                     float *__restrict__ nlse, size_t rows, int32_t *counter) {
    launch_dependents();
    wait_prior_grid();
    if (blockIdx.x == 0 && threadIdx.x < 64) counter[threadIdx.x] = 0;
    const int part = threadIdx.x & 7;
    const size_t r0 = (size_t)blockIdx.x * kRowdotRows + (threadIdx.x >> 3);
    uint4 a[2], b[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const size_t r = r0 + 32 * q;
        a[q] = b[q] = make_uint4(0, 0, 0, 0);
        if (r < rows) {
            a[q] = __ldg(reinterpret_cast<const uint4 *>(dO + r * 64) + part);
            b[q] = __ldg(reinterpret_cast<const uint4 *>(O + r * 64) + part);
        }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const size_t r = r0 + 32 * q;
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
        if (part == 0 && r < rows) {
            D[r] = acc;
            nlse[r] = LSE[r] * -1.4426950408889634f;
        }
    }
}

// P and dS of 32 columns, as bf16 pairs (even column in the low half): p = exp2(s * scale2 + nlse), dS = p (dP - D).
// kKeySide: nlse and D are per column (two arrays of shared memory), otherwise per row.  Columns whose bit of
// `on` is clear do not count (kMask).  Two columns per instruction except for the exponential.
template <bool kKeySide, bool kMask>
__device__ __forceinline__ void math32(const uint32_t (&sv)[32], const uint32_t (&tv)[32], uint64_t scale2, uint64_t row_nlse2,
                                       uint64_t row_D2, const float4 *vec_nlse, const float4 *vec_D, uint32_t on,
                                       uint32_t (&pk_p)[16], uint32_t (&pk_ds)[16]) {
#pragma unroll
    for (int e = 0; e < 32; e += 4) {
        uint64_t nl[2] = {row_nlse2, row_nlse2}, Dv[2] = {row_D2, row_D2};
        if (kKeySide) {
            const float4 a = vec_nlse[e >> 2], d4 = vec_D[e >> 2];
            nl[0] = pack_f32x2(a.x, a.y);
            nl[1] = pack_f32x2(a.z, a.w);
            Dv[0] = pack_f32x2(d4.x, d4.y);
            Dv[1] = pack_f32x2(d4.z, d4.w);
        }
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int k = e + 2 * q;
            float x0, x1, d0, d1;
            unpack_f32x2(fma_f32x2(pack_f32x2(sv[k], sv[k + 1]), scale2, nl[q]), x0, x1);
            float p0 = ex2(x0), p1 = ex2(x1);
            if (kMask) {
                if (!(on & (1u << k))) p0 = 0.f;
                if (!(on & (2u << k))) p1 = 0.f;
            }
            unpack_f32x2(mul_f32x2(pack_f32x2(p0, p1), sub_f32x2(pack_f32x2(tv[k], tv[k + 1]), Dv[q])), d0, d1);
            if (kKeySide) pk_p[k >> 1] = cvt_bf16x2(p0, p1);
            pk_ds[k >> 1] = cvt_bf16x2(d0, d1);
        }
    }
}
__device__ __forceinline__ uint32_t bits_below(int n) { return n <= 0 ? 0u : n >= 32 ? 0xffffffffu : (1u << n) - 1u; }

__global__ void __launch_bounds__(kThreads, 1) tc_bwd_kernel(const __grid_constant__ Params p) {
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
    // of a CTA is its own index, later ones come from the shared counter.
    int4 rec = make_int4(0, 0, 0, 0);
    int it_next = blockIdx.x;  // lane 0
    auto claim = [&]() {
        if (lane == 0) it_next = atomicAdd(p.counter, 1) + (int)gridDim.x;
    };
    auto fetch_record = [&]() {
        const int it = __shfl_sync(0xffffffffu, it_next, 0);
        rec = make_int4(0, 0, 0, 0);  // rows = 0: the list is exhausted
        if (it < 2 * p.n_units && lane < 4) {
            rec = __ldg(reinterpret_cast<const int4 *>(p.units + (it >> 1)) + lane);
            if (lane == 3) rec.z = it & 1;
        }
    };
    if (warp == kLoadWarp0) fetch_record();

    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(bars + 8 * (kBarRFull + i), kLoadWarps);
            mbar_init(bars + 8 * (kBarREmpty + i), 1 + kComputeWarps);
        }
        for (int i = 0; i < kStages; ++i) {
            mbar_init(bars + 8 * (kBarCFull + i), kLoadWarps);
            mbar_init(bars + 8 * (kBarCEmpty + i), 1);
        }
        mbar_init(bars + 8 * kBarSFull, 1);
        mbar_init(bars + 8 * kBarAFull, kComputeWarps);
        mbar_init(bars + 8 * kBarSTFree, kComputeWarps);
        mbar_init(bars + 8 * kBarGDone, 1);
        mbar_init(bars + 8 * kBarFinal, 1);
        for (int i = 0; i < kSchedDepth; ++i) {
            mbar_init(bars + 8 * (kBarSchedFull + i), 1);
            mbar_init(bars + 8 * (kBarSchedEmpty + i), kSchedReaders);
        }
        *s_abort = 0;
        fence_mbar_init();
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
        if (mbar_test_wait(bar, parity)) return true;  // already complete: no trip through the suspending form
#pragma unroll 1
        for (uint32_t it = 0; it < kWaitLimit; ++it) {
            if (mbar_try_wait(bar, parity)) return true;
            if (*s_abort) return false;
        }
        *s_abort = 1;
        atomicOr(p.status + 1, 1);
        return false;
    };
    // n-th entry of the item list of this CTA; false = the list is exhausted
    auto next_item = [&](uint32_t n, FwdUnit &u) -> bool {
        const int slot = n % kSchedDepth;
        if (!wait(bars + 8 * (kBarSchedFull + slot), (n / kSchedDepth) & 1)) return false;
        const int4 *src = reinterpret_cast<const int4 *>(s_item + slot);
        int4 *dst = reinterpret_cast<int4 *>(&u);
#pragma unroll
        for (int i = 0; i < 4; ++i) dst[i] = src[i];
        __syncwarp();
        if (lane == 0) mbar_arrive(bars + 8 * (kBarSchedEmpty + slot));
        return u.rows != 0;
    };

    if (warp < kComputeWarps) {
        // ------------------------------------------------------------------ arithmetic + epilogue
        reg_alloc<kRegsCompute>();
        const int r = tid & 127;   // row of the tile = lane of tensor memory
        const int cq = warp >> 2;  // takes the chunks cq and cq + 2 of a column tile
        const uint32_t tm = tmem + ((uint32_t)((warp & 3) * 32) << 16);
        uint8_t *stage = sm + kOffStage + warp * 2048;
        const uint64_t scale2 = pack_f32x2(p.scale_log2, p.scale_log2);
        uint32_t ph_s = 0, ph_g = 0, c_cnt = 0, item_cnt = 0;
        bool alive = true;
        FwdUnit un;
        wait_prior_grid();

#pragma unroll 1
        for (uint32_t n = 0; alive; ++n) {
            if (!next_item(n, un)) break;
            const bool key_side = un.ws_off == 0;
            const int nA = un.tiles_a(), n_tiles = nA + ((un.kP() + un.kB_end - un.kB0 + kTile - 1) / kTile), rows_h = un.rows_of(0);
            const int rb = item_cnt & 1;
            if (!(alive = wait(bars + 8 * (kBarRFull + rb), (item_cnt >> 1) & 1))) break;
            ++item_cnt;
            // this row's data (rows past the end shadow the last one)
            const int32_t *meta = reinterpret_cast<const int32_t *>(sm + kOffMeta) + rb * 5 * kTile + min(r, rows_h - 1);
            const int dst_row = r < rows_h ? meta[0] : -1, my_lo = meta[kTile], my_hi = meta[2 * kTile];
            const float row_nlse = __int_as_float(meta[3 * kTile]), row_D = __int_as_float(meta[4 * kTile]);
            __syncwarp();
            if (lane == 0) mbar_arrive(bars + 8 * (kBarREmpty + rb));
            const int w_lo_max = __reduce_max_sync(0xffffffffu, my_lo), w_hi_min = __reduce_min_sync(0xffffffffu, my_hi);

            // the tile loop is compiled once per side
            auto tile_loop = [&](auto side) {
                constexpr bool kKeySide = decltype(side)::value;
                const uint64_t row_nlse2 = pack_f32x2(row_nlse, row_nlse), row_D2 = pack_f32x2(row_D, row_D);
#pragma unroll 1
                for (int i = 0; i < n_tiles; ++i, ++c_cnt) {
                    const TileInfo t = tile_info(un, i, nA);
                    const bool full = t.w == kTile && (t.pre == kTile || (w_lo_max - t.k0 <= t.pre && w_hi_min - t.k0 >= kTile));
                    const float4 *vec = reinterpret_cast<const float4 *>(sm + kOffVec + (c_cnt % kStages) * 1024);
                    TR_T0(t_ws);
                    if (!(alive = wait(bars + 8 * kBarSFull, ph_s))) break;
                    ph_s ^= 1;
                    tc_fence_after();
                    TR_ADD(0, t_ws);
                    TR_T0(t_cmp);
                    // the operand columns are free once the gradient MMAs of the previous tile are done
                    bool a_free = i == 0;
                    auto wait_a = [&]() {
                        if (a_free) return;
                        alive = wait(bars + 8 * kBarGDone, ph_g);
                        ph_g ^= 1;
                        tc_fence_after();
                        a_free = true;
                    };
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
#pragma unroll
                        for (int cc = 0; cc < 2; ++cc) {
                            const int cb = cq * 32 + cc * 64;
                            math32<kKeySide, false>(sv[cc], tv[cc], scale2, row_nlse2, row_D2, vec + (cb >> 2), vec + 32 + (cb >> 2),
                                                    0u, pk_p, pk_ds);
                            if (cc == 0) wait_a();
                            if (kKeySide) tmem_st16(tm + kTmA1 + (cb >> 1), pk_p);
                            tmem_st16(tm + (kKeySide ? kTmA2 : kTmA1) + (cb >> 1), pk_ds);
                        }
                    } else {
                        // this row counts the columns [0, pre) and [r_lo, r_hi); some row of the warp counts columns only
                        // there and within [e_lo, e_hi)
                        const int r_lo = t.is_b ? my_lo - t.k0 : 0, r_hi = t.is_b ? min(my_hi - t.k0, t.w) : 0;
                        const int e_lo = __reduce_min_sync(0xffffffffu, r_lo), e_hi = __reduce_max_sync(0xffffffffu, r_hi);
                        const int e_end = max(t.pre, e_hi > e_lo ? e_hi : 0);
                        bool held = true;
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
                                math32<kKeySide, true>(sv, tv, scale2, row_nlse2, row_D2, vec + (cb >> 2), vec + 32 + (cb >> 2),
                                                       bits_below(t.pre - cb) | (bits_below(r_hi - cb) & ~bits_below(r_lo - cb)), pk_p, pk_ds);
                            }
                            wait_a();
                            if (kKeySide) tmem_st16(tm + kTmA1 + (cb >> 1), pk_p);
                            tmem_st16(tm + (kKeySide ? kTmA2 : kTmA1) + (cb >> 1), pk_ds);
                        }
                        if (held) release_st();
                        // Also when nothing was written: keeps this warp's arrival below out of the barrier phase of the
                        // previous tile, which a slower warp may not have reached yet.
                        wait_a();
                    }
                    if (!alive) break;
                    tc_wait_st();
                    tc_fence_before();
                    if (lane == 0) mbar_arrive(bars + 8 * kBarAFull);
                    TR_ADD(2, t_cmp);
                    TR_INC(7);
                }
            };
            if (key_side) tile_loop(std::true_type{});
            else tile_loop(std::false_type{});
            if (!alive) break;

            // epilogue: wait for the last gradient MMAs, then scatter the rows to their original positions.  Key side:
            // one column group of the arithmetic warps stores dV, the other dK; query side: 32 columns of dQ each.
            TR_T0(t_ep);
            if (n_tiles > 0) {
                if (!(alive = wait(bars + 8 * kBarGDone, ph_g))) break;
                ph_g ^= 1;
                tc_fence_after();
            }
            __nv_bfloat16 *out = (key_side ? (cq ? p.dK : p.dV) : p.dQ + cq * 32) + p.tr.base(un.b, un.h) * 64;
            const uint32_t acc = tm + (key_side ? (cq ? kTmAcc2 : kTmAcc1) : kTmAcc1 + cq * 32);
            const float mul = key_side && cq == 0 ? 1.f : p.scale;
#pragma unroll 1
            for (int c2 = 0; c2 < (key_side ? 2 : 1); ++c2) {
                uint32_t o[32];
                if (n_tiles > 0) {
                    tmem_ld32(acc + c2 * 32, o);
                    tc_wait_ld();
                    reg_fence(o);
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
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int row = 8 * i + (lane >> 2), j = lane & 3;
                    const int dr = __shfl_sync(0xffffffffu, dst_row, row);
                    const uint4 x = *reinterpret_cast<const uint4 *>(stage + row * 64 + ((j ^ ((row >> 1) & 3)) << 4));
                    if (dr >= 0) *reinterpret_cast<uint4 *>(out + (size_t)dr * 64 + c2 * 32 + j * 8) = x;
                }
                __syncwarp();
            }
            tc_fence_before();  // the accumulators were read; the next item may overwrite them
            TR_ADD(3, t_ep);
        }
    } else if (warp == kMmaWarp) {
        // ------------------------------------------------------------------ MMA issuer
        // The whole warp runs the control flow (operands stay warp-uniform), one lane issues.
        reg_dealloc<kRegsOther>();
        const bool leader = elect_one();
        uint32_t c_cnt = 0, item_cnt = 0, ph_a = 0, ph_st = 0;
        bool alive = true;
        const uint32_t idesc_g = idesc_bf16(128, 64, 0, 1);  // B = 16 rows of the column tile x 64, MN-major
        constexpr uint32_t kStep = (16 * kRowBytes) >> 4;    // 16 rows of the column tile
        const uint32_t tA1 = tmem + kTmA1, tA2 = tmem + kTmA2, tG1 = tmem + kTmAcc1, tG2 = tmem + kTmAcc2;
        FwdUnit un;
        wait_prior_grid();
#pragma unroll 1
        for (uint32_t n = 0; alive; ++n) {
            if (!next_item(n, un)) break;
            const bool key_side = un.ws_off == 0;
            const int nA = un.tiles_a(), n_tiles = nA + ((un.kP() + un.kB_end - un.kB0 + kTile - 1) / kTile);
            const int rb = item_cnt & 1;
            if (!(alive = wait(bars + 8 * (kBarRFull + rb), (item_cnt >> 1) & 1))) break;
            tc_fence_after();
            const uint32_t ra = smem_desc_lo(base + kOffR + rb * 2 * kTileBytes), rbb = ra + (kTileBytes >> 4);
            int g_ks = 0;  // 16-column steps of the tile whose gradient MMAs are outstanding; one round more than tiles
#pragma unroll 1
            for (int i = 0; i <= n_tiles; ++i) {
                int ks = 0;
                uint32_t idesc = 0, ca = 0;
                if (i < n_tiles) {  // the tile has landed
                    const int st = c_cnt % kStages;
                    const TileInfo t = tile_info(un, i, nA);
                    ks = (t.w + 15) >> 4;
                    idesc = idesc_bf16(128, ks * 16, 0, 0);
                    ca = smem_desc_lo(base + kOffC + st * 2 * kTileBytes);
                    if (!(alive = wait(bars + 8 * (kBarCFull + st), (c_cnt / kStages) & 1))) break;
                }
                if (i > 0) {  // S and dP are free again once the previous tile's values are in registers
                    if (!(alive = wait(bars + 8 * kBarSTFree, ph_st))) break;
                    ph_st ^= 1;
                }
                tc_fence_after();
                if (i < n_tiles) {
                    const uint32_t cb = ca + (kTileBytes >> 4);
                    if (leader) {
                        mma_ss_lean<0>(tmem + kTmS, ra, ca, idesc);  // S = Ra Ca^T, K = 64 as four steps of 16
                        mma_ss_lean<1>(tmem + kTmS, ra + 2, ca + 2, idesc);
                        mma_ss_lean<1>(tmem + kTmS, ra + 4, ca + 4, idesc);
                        mma_ss_lean<1>(tmem + kTmS, ra + 6, ca + 6, idesc);
                        mma_ss_lean<0>(tmem + kTmT, rbb, cb, idesc);  // dP = Rb Cb^T
                        mma_ss_lean<1>(tmem + kTmT, rbb + 2, cb + 2, idesc);
                        mma_ss_lean<1>(tmem + kTmT, rbb + 4, cb + 4, idesc);
                        mma_ss_lean<1>(tmem + kTmT, rbb + 6, cb + 6, idesc);
                        mma_commit(bars + 8 * kBarSFull);
                    }
                    __syncwarp();
                    ++c_cnt;
                }
                if (i > 0) {  // gradient MMAs of the previous tile, behind this tile's S and dP
                    if (!(alive = wait(bars + 8 * kBarAFull, ph_a))) break;
                    ph_a ^= 1;
                    tc_fence_after();
                    const int g_st = (c_cnt - (i < n_tiles ? 2 : 1)) % kStages;
                    const uint32_t a_lo = smem_desc_lo(base + kOffC + g_st * 2 * kTileBytes), b_lo = a_lo + (kTileBytes >> 4);
                    if (leader) {
                        if (key_side) {
                            mma_ts_lean_flag(tG1, tA1, b_lo, idesc_g, i > 1);  // dV += P^T dO
                            mma_ts_lean_flag(tG2, tA2, a_lo, idesc_g, i > 1);  // dK += dS^T Q
#pragma unroll 1
                            for (int k = 1; k < g_ks; ++k) {
                                mma_ts_lean<1>(tG1, tA1 + 8 * k, b_lo + k * kStep, idesc_g);
                                mma_ts_lean<1>(tG2, tA2 + 8 * k, a_lo + k * kStep, idesc_g);
                            }
                        } else {
                            mma_ts_lean_flag(tG1, tA1, a_lo, idesc_g, i > 1);  // dQ += dS K
#pragma unroll 1
                            for (int k = 1; k < g_ks; ++k) mma_ts_lean<1>(tG1, tA1 + 8 * k, a_lo + k * kStep, idesc_g);
                        }
                        mma_commit(bars + 8 * kBarGDone);
                        mma_commit(bars + 8 * (kBarCEmpty + g_st));
                    }
                    __syncwarp();
                }
                g_ks = ks;
            }
            if (!alive) break;
            if (leader) mma_commit(bars + 8 * (kBarREmpty + rb));
            __syncwarp();
            ++item_cnt;
        }
        // nothing of this CTA may still run on the tensor pipe when tensor memory is freed
        if (leader) mma_commit(bars + 8 * kBarFinal);
        __syncwarp();
        mbar_wait_bounded(bars + 8 * kBarFinal, 0, kWaitLimit);
    } else if (warp < kLoadWarp0) {
        // ------------------------------------------------------------------ padding rows: zero gradients
        reg_dealloc<kRegsOther>();
        wait_prior_grid();
#pragma unroll 1
        for (int c = blockIdx.x; c < p.n_pads; c += gridDim.x) {
            const PadChunk pc = p.pads[c];
            const ViewPlan &vp = p.head_view[pc.h] ? p.colv : p.rowv;
#pragma unroll 2
            for (int i = (warp - kPadWarp0) * 4 + (lane >> 3); i < pc.n; i += 4 * kPadWarps) {  // eight lanes per row
                const int orig = __ldg(vp.perm + (size_t)pc.b * p.N + pc.t0 + i);
                if (p.tr.exists(pc.b, orig)) {
                    const size_t at = (p.tr.base(pc.b, pc.h) + orig) * 64 + (lane & 7) * 8;
                    *reinterpret_cast<uint4 *>(p.dQ + at) = make_uint4(0, 0, 0, 0);
                    *reinterpret_cast<uint4 *>(p.dK + at) = make_uint4(0, 0, 0, 0);
                    *reinterpret_cast<uint4 *>(p.dV + at) = make_uint4(0, 0, 0, 0);
                }
            }
        }
    } else {
        // ------------------------------------------------------------------ loaders
        reg_dealloc<kRegsOther>();
        wait_prior_grid();
        const int lw = warp - kLoadWarp0;
        uint32_t c_cnt = 0, item_cnt = 0;
        uint32_t pend[kLag];
#pragma unroll
        for (int i = 0; i < kLag; ++i) pend[i] = 0;
        bool alive = true;

        // Commits the copies issued so far as one group and signals the barrier of the group that
        // was committed kLag groups earlier (its copies have landed by then).
        auto commit_and_signal = [&](uint32_t bar) {
            cp_async_commit();
            const uint32_t oldest = pend[0];
#pragma unroll
            for (int i = 0; i + 1 < kLag; ++i) pend[i] = pend[i + 1];
            pend[kLag - 1] = bar;
            if (oldest) {
                cp_async_wait_group<kLag>();
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(oldest);
            }
        };
        // Signals every group still pending, oldest first and each as soon as its own copies have
        // landed (an older group is not held back by the latency of a newer one).  Called before
        // this warp blocks on a buffer that is not free yet: the consumers may need exactly those
        // groups to free it.
        auto flush = [&]() {
            static_assert(kLag == 2, "written out for two pending groups");
            if (pend[0]) {
                cp_async_wait_group<1>();
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(pend[0]);
                pend[0] = 0;
            }
            if (pend[1]) {
                cp_async_wait_group<0>();
                fence_proxy_async();
                __syncwarp();
                if (lane == 0) mbar_arrive(pend[1]);
                pend[1] = 0;
            }
        };
        auto wait_free = [&](uint32_t bar, uint32_t parity) -> bool {
            if (__all_sync(0xffffffffu, mbar_test_wait(bar, parity))) return true;
            flush();
            TR_T0(t_wf);
            const bool ok = wait(bar, parity);
            TR_ADD(0, t_wf);
            return ok;
        };

        FwdUnit un;
#pragma unroll 1
        for (uint32_t n = 0; alive; ++n) {
            const int slot = n % kSchedDepth;
            if (warp == kLoadWarp0) {
                if (n >= (uint32_t)kSchedDepth && !wait_free(bars + 8 * (kBarSchedEmpty + slot), ((n / kSchedDepth) & 1) ^ 1)) break;
                if (lane < 4) reinterpret_cast<int4 *>(s_item + slot)[lane] = rec;
                __syncwarp();
                if (lane == 0) mbar_arrive(bars + 8 * (kBarSchedFull + slot));  // release: the record is visible to the readers
            } else if (!wait_free(bars + 8 * (kBarSchedFull + slot), (n / kSchedDepth) & 1)) {
                break;
            }
            if (!next_item(n, un)) break;
            const bool key_side = un.ws_off == 0;
            const int nA = un.tiles_a(), n_tiles = nA + ((un.kP() + un.kB_end - un.kB0 + kTile - 1) / kTile), rows_h = un.rows_of(0);
            const ViewPlan &vp = p.head_view[un.h] ? p.colv : p.rowv;
            const size_t bn = (size_t)un.b * p.N;
            const int32_t *perm = vp.perm + bn;
            const size_t bh = p.tr.base(un.b, un.h);
            const uint8_t *row_a = reinterpret_cast<const uint8_t *>((key_side ? p.K : p.Q) + bh * 64);
            const uint8_t *col_a = reinterpret_cast<const uint8_t *>((key_side ? p.Q : p.K) + bh * 64);
            const int64_t kv = reinterpret_cast<const uint8_t *>(p.V) - reinterpret_cast<const uint8_t *>(p.K),
                          qdo = reinterpret_cast<const uint8_t *>(p.dO) - reinterpret_cast<const uint8_t *>(p.Q);
            // column tiles inside [0, ident) of the order are contiguous in the tensors (see bulk_tile)
            const int ident = p.use_tma ? __ldg(vp.ident + un.b) : 0;

            // step -1: the row operands and row data; steps 0 ..: the column tiles
            auto step_idx = [&](int i) { return fetch_idx(perm, i < 0 ? row_tile(un.q0, rows_h) : tile_info(un, i, nA), lw, lane); };
            int next = step_idx(-1);
#pragma unroll 1
            for (int i = -1; i < n_tiles; ++i) {
                const int now = next;
                if (i + 1 < n_tiles) next = step_idx(i + 1);
                else if (warp == kLoadWarp0) claim();  // the number and then the record travel under the copies
                const TileInfo t = tile_info(un, max(i, 0), nA);
                const int st = c_cnt % kStages, rb = item_cnt & 1;
                const uint32_t bar_e = i < 0 ? kBarREmpty + rb : kBarCEmpty + st, bar_full = bars + 8 * (i < 0 ? kBarRFull + rb : kBarCFull + st);
                if (!(alive = wait_free(bars + 8 * bar_e, ((i < 0 ? item_cnt >> 1 : c_cnt / kStages) & 1) ^ 1))) break;
                const uint32_t dst = base + (i < 0 ? kOffR + rb * 2 * kTileBytes : kOffC + st * 2 * kTileBytes);
                const bool bulk = i >= 0 && bulk_tile(t, ident);
                if (bulk) {
                    if (lw == 0 && lane == 0) {
                        mbar_expect_tx(bar_full, 2 * kTileBytes);
                        tma_load_2d(dst, key_side ? &p.tmQ : &p.tmK, 0, (int)bh + t.first(), bar_full);
                        tma_load_2d(dst + kTileBytes, key_side ? &p.tmdO : &p.tmV, 0, (int)bh + t.first(), bar_full);
                    }
                    __syncwarp();
                } else {
                    const bool kv_pair = (i < 0) == key_side;
                    gather_rows(dst, i < 0 ? row_a : col_a, true, kv_pair ? kv : qdo, now, i < 0 ? kTile : (t.w + 15) & ~15, lw, lane);
                }
                const int rr = 32 * lw + lane;
                if (i < 0) {  // row data for the arithmetic threads
                    const uint32_t meta = base + kOffMeta + rb * 5 * kTile * 4 + rr * 4;
                    if (rr < rows_h) {
                        const size_t at = bn + un.q0 + rr;
                        cp_async4(meta, vp.perm + at);
                        cp_async4(meta + kTile * 4, vp.seg_lo + at);
                        cp_async4(meta + 2 * kTile * 4, vp.seg_hi + at);
                        if (!key_side) {
                            cp_async4(meta + 3 * kTile * 4, p.nlse + bh + now);
                            cp_async4(meta + 4 * kTile * 4, p.D + bh + now);
                        }
                    }
                } else if (key_side) {  // column data
                    const uint32_t vec = base + kOffVec + st * 1024 + rr * 4;
                    cp_async4(vec, p.nlse + bh + now);
                    cp_async4(vec + 512, p.D + bh + now);
                }
                if (!bulk || key_side) commit_and_signal(bar_full);
                else if (lane == 0) mbar_arrive(bar_full);
                if (i + 1 == n_tiles && warp == kLoadWarp0) fetch_record();
                if (i < 0) {
                    ++item_cnt;
                } else {
                    // the very first tile of the CTA is signalled as soon as it has landed
                    if (c_cnt == 0) flush();
                    ++c_cnt;
                }
            }
        }
        flush();  // drain: signal the groups still pending
    }

#ifdef MATE_TRACE
    if (lane == 0 && (warp == 0 || warp == 4 || warp == kMmaWarp || warp == kLoadWarp0) && blockIdx.x < kTraceCtas) {
        const int role = warp == 0 ? 0 : warp == 4 ? 1 : warp == kMmaWarp ? 2 : 3;
        long long *o = g_trace_bwd + blockIdx.x * 32 + role * 8;
        for (int i = 0; i < 8; ++i) o[i] = tr[i];
        if (role == 0) o[5] = clock64() - tr_start;
    }
#endif
    tc_fence_before();
    __syncthreads();
    if (warp == kMmaWarp) tmem_dealloc(tmem, 512);
}

SmemAttrOnce g_smem_attr;

inline size_t align256(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

// workspace: [256 B counters][D: B*H*N floats][-LSE log2 e: as many]
size_t tc_bwd_workspace(const mate_plan_t *plan) {
    return 256 + 2 * align256((size_t)plan->B * plan->H * plan->N * sizeof(float));
}

// pass: which of the calls that share the workspace, O, LSE and dO this is; the row dots are formed in pass 0.
int tc_bwd(const mate_plan_t *plan, const void *Q, const void *K, const void *V, const void *O,
           const float *LSE, const void *dO, float scale, void *dQ, void *dK, void *dV, void *workspace, int pass,
           cudaStream_t stream) {
    if (plan->bwd_grid == 0) return MATE_OK;
    if (g_smem_attr.ensure((const void *)tc_bwd_kernel, (int)kSmemBytes, plan->device) != MATE_OK) return MATE_ERR_CUDA;
    const size_t rows = plan->n_rows();
    uint8_t *ws = (uint8_t *)workspace;
    float *D = (float *)(ws + 256);
    float *nlse = D + align256((size_t)plan->B * plan->H * plan->N * sizeof(float)) / sizeof(float);
    Params p;
    p.use_tma = rows < (size_t(1) << 31) && make_row_map(&p.tmQ, Q, rows) && make_row_map(&p.tmK, K, rows) &&
                make_row_map(&p.tmV, V, rows) && make_row_map(&p.tmdO, dO, rows);
    p.Q = (const __nv_bfloat16 *)Q;
    p.K = (const __nv_bfloat16 *)K;
    p.V = (const __nv_bfloat16 *)V;
    p.dO = (const __nv_bfloat16 *)dO;
    p.nlse = nlse;
    p.D = D;
    p.dQ = (__nv_bfloat16 *)dQ;
    p.dK = (__nv_bfloat16 *)dK;
    p.dV = (__nv_bfloat16 *)dV;
    p.rowv = plan->view[0];
    p.colv = plan->view[1];
    p.head_view = plan->head_view_dev;
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
    p.counter = (int32_t *)ws + 8 * pass;

    if (pass == 0 && launch_after(rowdot_kernel, dim3((unsigned)((rows + kRowdotRows - 1) / kRowdotRows)), 256, 0, stream, p.dO,
                                  (const __nv_bfloat16 *)O, LSE, D, nlse, rows, (int32_t *)ws) != cudaSuccess)
        return MATE_ERR_CUDA;
    return launch_after(tc_bwd_kernel, dim3((unsigned)plan->bwd_grid), kThreads, kSmemBytes, stream, p) == cudaSuccess ? MATE_OK : MATE_ERR_CUDA;
}

}  // namespace mate

#ifdef MATE_TRACE
// copies the cycle counters of the last backward launch to the host: [kTraceCtas CTAs][4 roles][8]
extern "C" int mate_debug_trace_bwd(long long *host_out) {
    return cudaMemcpyFromSymbol(host_out, mate::g_trace_bwd, sizeof(long long) * mate::kTraceCtas * 32) == cudaSuccess ? 0 : -4;
}
#endif
