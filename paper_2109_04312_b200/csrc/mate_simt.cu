// Kernels without tensor cores: fp32 arithmetic whatever the storage type, any head size up to 128.  They serve
// fp32 tensors and head sizes other than 64, and are the reference the tensor-core kernels were brought up
// against on the device.
//
// In a head's view order (see mate_plan) the keys of query row t are
//     [0, P)  u  [max(seg_lo[t], P), seg_hi[t])
// which is the attention pattern A of Section 3 for both table rows (own segment plus prefix) and
// prefix rows (seg_lo = 0, seg_hi = n_valid).  The pattern is symmetric, so the queries that
// attend to key t are the same two ranges; dK/dV therefore need no atomics.
//
// A block takes 32 rows of the order against tiles of 64 columns: [0, P), then the union of the rows' other
// ranges.  Two groups of 128 threads take the tiles in turn and add up what they have at the end: a table row's block has
// two or three tiles, one of the global block as many as there are columns, and those are the last to finish.  A
// thread forms 4 x 4 scores, the 16 lanes of a half warp share four rows from the scores to the results, so only the loads
// of a tile need the group to meet.  The first matrix of the next tile travels to registers under the second half of this
// one, the second under the first half.  A warp leaves out the columns that none of its eight rows counts.
// With 8 x 512 tokens (16 warps per SM at the registers this takes) the data pipe that serves shared memory is 66 % busy in the
// forward and 70 % in the backward, issue slots 59 and 58 %, the multiply-add units 36 and 37 %; what a warp waits for is shared
// memory (1.2 and 1.8 cycles per instruction), its turn (1.2, 1.0) and the group (1.0; two hand-overs per tile in the forward, three
// in the backward), hardly global memory (0.3).
// Two blocks per SM (one with heads of more than 64): three of smaller heads fit, but spill (2 x 512 tokens, heads of 32, 16.2 / 31.9 us
// with two, 19.8 / 41.4 with three; of 16 12.5 / 24.2, 13.3 / 25.9).
// 2 x 512 tokens, 12 heads of 64, forward / backward: 23.7 / 50.0 us, 23.7 / 52.5 with P of the backward in registers.  The forms before, as
// timed then: 24.4 / 53.1; with the rows' key ranges in registers 25.2 / 54.7; with the rows' look-ups directly in front of the loads
// that need them 29.4 / 62.8 (a warp waited 2.2 times as long for global memory as it issued); with 2 x 4 scores per thread,
// one group and every column of a tile 37.4 / 70.8; with one warp per row and global reads of every key 463 / 1540.
#include <cuda_bf16.h>

#include <mutex>
#include <type_traits>

#include "mate_internal.h"
#include "sm100_ptx.cuh"

namespace mate {

namespace {

// Built-in scratch of mate_attn_bwd_noalloc: one float per (example, head, position) for the row
// dots D.  It is part of the library image, so every GPU that loads the library holds these
// 4 MiB until the process exits.
constexpr size_t kNoAllocMaxRows = size_t(1) << 20;
static __device__ __align__(256) float g_noalloc_rowdot[kNoAllocMaxRows];

constexpr int kMaxD = 128;
constexpr int kRows = 32, kCols = 64, kThreads = 256;
constexpr int kGroup = 128, kMine = kRows / (kGroup / 16);  // threads that share a tile, rows of a thread
constexpr int kPStride = kCols + 4;

__device__ __forceinline__ float4 load4(const float *p) { return __ldg(reinterpret_cast<const float4 *>(p)); }
__device__ __forceinline__ float4 load4(const __nv_bfloat16 *p) {
    const uint2 x = __ldg(reinterpret_cast<const uint2 *>(p));
    const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&x.x));
    const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&x.y));
    return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void from_f(float &dst, float x) { dst = x; }
__device__ __forceinline__ void from_f(__nv_bfloat16 &dst, float x) { dst = __float2bfloat16_rn(x); }

// reductions over the 16 lanes of a half warp
__device__ __forceinline__ float half_max(float v) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
__device__ __forceinline__ float half_sum(float v) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

struct Common {
    ViewPlan rowv, colv;
    const uint8_t *head_view;
    const int32_t *n_valid, *prefix;  // prefix: length of the global block
    int N, d, view_order;
    float scale;
    TensorRows tr;
};

// First of this thread's rows of the block (both groups have all of them).
__device__ __forceinline__ int first_row() { return (int)((threadIdx.x % kGroup) >> 4) * kMine; }
__device__ __forceinline__ void group_sync() { asm volatile("bar.sync %0, %1;" ::"r"(1 + (int)threadIdx.x / kGroup), "n"(kGroup) : "memory"); }

// The rows of a block and the column tiles they meet.  What is needed once a tile stays in shared memory: registers are what the
// kernels are short of (128 with heads of 64, bytes spilled and read back: forward 8 / 8 with fp32 tensors and 20 / 16 with bf16,
// backward 4 / 4 with either).
struct RowBlock {
    struct Shared {
        int P, b_lo, b_hi, lo[kRows], hi[kRows];  // lo, hi: behind the global block
    };
    const int32_t *perm;
    const Shared *s;
    size_t bh;
    int t0, n, n_tiles;
    int w_lo, w_hi;  // all that the rows of this thread's warp count behind the global block
    __device__ __forceinline__ int orig(int t) const { return perm ? __ldg(perm + t) : t; }
    __device__ __forceinline__ int n_a() const { return (s->P + kCols - 1) / kCols; }
    // tile i: w columns from c0 on, of which [k0, k1) count for some row of this warp
    __device__ __forceinline__ void tile(int i, int &c0, int &w) const {
        const int na = n_a();
        c0 = i < na ? i * kCols : s->b_lo + (i - na) * kCols;
        w = min(kCols, (i < na ? s->P : s->b_hi) - c0);
    }
    __device__ __forceinline__ void span(int i, int c0, int w, int &k0, int &k1) const {
        const bool a = i < n_a();
        k0 = a ? 0 : max(w_lo - c0, 0);
        k1 = a ? w : min(w_hi - c0, w);
    }
    // the columns of tile i that count for a row of the block: [lo, hi)
    __device__ __forceinline__ void row_span(int i, int c0, int w, int row, int &lo, int &hi) const {
        const bool a = i < n_a();
        lo = a ? 0 : s->lo[row] - c0;
        hi = a ? w : min(s->hi[row] - c0, w);
    }
};
__device__ __forceinline__ RowBlock row_block(const Common &c, int b, int h, int blk, RowBlock::Shared *sh) {
    const ViewPlan &vp = c.head_view[h] ? c.colv : c.rowv;
    RowBlock r;
    r.perm = c.view_order ? nullptr : vp.perm + (size_t)b * c.N;
    r.s = sh;
    r.bh = c.tr.base(b, h);
    r.t0 = blk * kRows;
    const int nv = c.n_valid[b], P = min(c.prefix[b], nv);
    r.n = min(kRows, nv - r.t0);  // valid rows of the block (<= 0: padding only)
    const int32_t *slo = vp.seg_lo + (size_t)b * c.N + r.t0, *shi = vp.seg_hi + (size_t)b * c.N + r.t0;
    if (threadIdx.x < kRows) {  // (rows past the last valid one repeat it)
        const int row = min((int)threadIdx.x, r.n - 1);
        const int l = r.n > 0 ? max(slo[row], P) : 0, u = r.n > 0 ? shi[row] : 0;
        const int lmin = __reduce_min_sync(0xffffffffu, u > l ? l : 0x7fffffff), umax = __reduce_max_sync(0xffffffffu, u > l ? u : 0);
        sh->lo[threadIdx.x] = l;
        sh->hi[threadIdx.x] = u;
        if (threadIdx.x == 0) {
            sh->P = P;
            sh->b_lo = lmin;
            sh->b_hi = umax;
        }
    }
    __syncthreads();
    int w_lo = 0x7fffffff, w_hi = 0;
#pragma unroll
    for (int j = 0; j < kMine; ++j) {
        const int l = sh->lo[first_row() + j], u = sh->hi[first_row() + j];
        if (u > l) {
            w_lo = min(w_lo, l);
            w_hi = max(w_hi, u);
        }
    }
    r.w_lo = __reduce_min_sync(0xffffffffu, w_lo);
    r.w_hi = __reduce_max_sync(0xffffffffu, w_hi);
    r.n_tiles = r.n_a() + (sh->b_hi > sh->b_lo ? (sh->b_hi - sh->b_lo + kCols - 1) / kCols : 0);
    return r;
}

// kN rows of a tensor in registers (float4 chunks dealt over the threads of a group), on their way to shared memory.
template <int kN, int DP>
struct Chunks {
    static constexpr int kPer = kN * DP / 4 / kGroup;
    static_assert(kPer > 0 && kPer * kGroup * 4 == kN * DP, "every thread has the same number of chunks");
    float4 v[kPer];
    // s_at: the rows of the tensor, in shared memory
    template <typename T>
    __device__ __forceinline__ void load(const T *base, const int *s_at, int d) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int c = threadIdx.x % kGroup + i * kGroup, row = c / (DP / 4), ch = c % (DP / 4);
            v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (ch * 4 < d) v[i] = load4(base + (size_t)s_at[row] * d + ch * 4);
        }
    }
    __device__ __forceinline__ void store(float *s) const {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
            const int c = threadIdx.x % kGroup + i * kGroup, row = c / (DP / 4), ch = c % (DP / 4);
            *reinterpret_cast<float4 *>(s + row * (DP + 4) + ch * 4) = v[i];
        }
    }
};

// s[.][kQ0 .. kQ0 + kQn) = this thread's rows of A times columns tx + 16 q of B, both [., DP + 4] in shared memory
template <int DP, int kQ0, int kQn>
__device__ __forceinline__ void score_cols(float (&s)[kMine][4], const float *A, const float *B, int row0, int tx) {
#pragma unroll (DP > 64 ? 2 : 1)
    for (int e = 0; e < DP; e += 4) {
        float4 a[kMine], b[kQn];
#pragma unroll
        for (int j = 0; j < kMine; ++j) a[j] = *reinterpret_cast<const float4 *>(A + (row0 + j) * (DP + 4) + e);
#pragma unroll
        for (int c = 0; c < kQn; ++c) b[c] = *reinterpret_cast<const float4 *>(B + (tx + 16 * (kQ0 + c)) * (DP + 4) + e);
#pragma unroll
        for (int j = 0; j < kMine; ++j)
#pragma unroll
            for (int c = 0; c < kQn; ++c) {
                float &x = s[j][kQ0 + c];
                x = fmaf(a[j].x, b[c].x, x);
                x = fmaf(a[j].y, b[c].y, x);
                x = fmaf(a[j].z, b[c].z, x);
                x = fmaf(a[j].w, b[c].w, x);
            }
    }
}
// All four groups of 16 columns at once, or those that meet [k0, k1) one by one where that is half the multiply-adds
// or less (the reads of shared memory are as many for two groups alone as for four together).
template <int DP>
__device__ __forceinline__ void scores(float (&s)[kMine][4], const float *A, const float *B, int row0, int tx, int k0, int k1) {
#pragma unroll
    for (int j = 0; j < kMine; ++j)
#pragma unroll
        for (int c = 0; c < 4; ++c) s[j][c] = 0.f;
    if (((k1 + 15) >> 4) - (k0 >> 4) > 2) {
        score_cols<DP, 0, 4>(s, A, B, row0, tx);
        return;
    }
    if (k0 < 16) score_cols<DP, 0, 1>(s, A, B, row0, tx);
    if (k0 < 32 && k1 > 16) score_cols<DP, 1, 1>(s, A, B, row0, tx);
    if (k0 < 48 && k1 > 32) score_cols<DP, 2, 1>(s, A, B, row0, tx);
    if (k1 > 48) score_cols<DP, 3, 1>(s, A, B, row0, tx);
}
// The DP / 16 result columns of a thread: groups of kW at tx * kW + g * 16 * kW.
template <int DP>
struct Cols {
    static constexpr int kN = DP / 16, kW = kN < 4 ? kN : 4;
    __device__ static __forceinline__ int col(int tx, int i) { return (i / kW) * 16 * kW + tx * kW + i % kW; }
};
// acc[.][DP / 16] += rows of X ([., kPStride]) times B [64, DP + 4], over the columns [k0, k1) of X
template <int DP>
__device__ __forceinline__ void accumulate(float (&acc)[kMine][DP / 16], const float *X, const float *B, int row0, int tx, int k0, int k1) {
    constexpr int kN = Cols<DP>::kN;
#pragma unroll 2
    for (int k = k0 & ~3; k < k1; k += 4) {
        float4 x[kMine];
#pragma unroll
        for (int j = 0; j < kMine; ++j) x[j] = *reinterpret_cast<const float4 *>(X + (row0 + j) * kPStride + k);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float *brow = B + (k + q) * (DP + 4);
            float b[kN];
            if (kN >= 4) {
#pragma unroll
                for (int g = 0; g < kN / 4; ++g) *reinterpret_cast<float4 *>(b + 4 * g) = *reinterpret_cast<const float4 *>(brow + g * 64 + tx * 4);
            } else if (kN == 2) {
                *reinterpret_cast<float2 *>(b) = *reinterpret_cast<const float2 *>(brow + tx * 2);
            } else {
                b[0] = brow[tx];
            }
#pragma unroll
            for (int j = 0; j < kMine; ++j) {
                const float xv = q == 0 ? x[j].x : q == 1 ? x[j].y : q == 2 ? x[j].z : x[j].w;
#pragma unroll
                for (int i = 0; i < kN; ++i) acc[j][i] = fmaf(xv, b[i], acc[j][i]);
            }
        }
    }
}
template <typename T, int DP>
__device__ __forceinline__ void store_row(T *row, const float (&acc)[DP / 16], float mul, int tx, int d) {
#pragma unroll
    for (int i = 0; i < DP / 16; ++i) {
        const int c = Cols<DP>::col(tx, i);
        if (c < d) from_f(row[c], acc[i] * mul);
    }
}
// Rows of the block behind the valid ones: zeros (and LSE = -inf) where the row exists.
template <typename T>
__device__ __forceinline__ void pad_rows(const Common &c, const RowBlock &r, int b, T *o0, T *o1, float *lse) {
    for (int i = max(r.n, 0) * 16 + (int)threadIdx.x; i < min(kRows, c.N - r.t0) * 16; i += kThreads) {
        const int k = r.orig(r.t0 + (i >> 4));
        if (!c.tr.exists(b, k)) continue;  // packed layout: beyond the example's end there is no such row
        for (int e = i & 15; e < c.d; e += 16) {
            from_f(o0[(r.bh + k) * c.d + e], 0.f);
            if (o1) from_f(o1[(r.bh + k) * c.d + e], 0.f);
        }
        if (lse && (i & 15) == 0) lse[r.bh + k] = -INFINITY;
    }
}

// ---------------------------------------------------------------------------------- forward
template <typename T, int DP>
__global__ void __launch_bounds__(kThreads, DP <= 64 ? 2 : 1)
simt_fwd_kernel(const T *__restrict__ Q, const T *__restrict__ K, const T *__restrict__ V, T *__restrict__ O,
                float *__restrict__ LSE, const Common c, int H, int n_bh) {
    extern __shared__ __align__(16) float smem[];
    __shared__ RowBlock::Shared s_rows;
    __shared__ int s_col[2][kCols], s_own[kRows];  // original rows of each group's tile, of the block
    ptx::wait_prior_grid();
    constexpr int kC = kCols * (DP + 4), kPart = 2 * kC + kRows * kPStride;
    const int grp = threadIdx.x / kGroup;
    float *sQ = smem, *part = sQ + kRows * (DP + 4), *sK = part + grp * kPart, *sV = sK + kC, *sP = sV + kC;
    // row blocks vary slowest: the long ones (global block) come first
    const int bh = blockIdx.x % n_bh, b = bh / H, h = bh % H;
    const RowBlock r = row_block(c, b, h, blockIdx.x / n_bh, &s_rows);
    pad_rows(c, r, b, O, (T *)nullptr, LSE);
    if (r.n <= 0) return;
    const int tx = threadIdx.x & 15, row0 = first_row();
    const T *Kh = K + r.bh * c.d, *Vh = V + r.bh * c.d;

    const int tid = threadIdx.x % kGroup;
    int *at = s_col[grp];
    int c0 = 0, w = 0;
    if (grp < r.n_tiles) {
        r.tile(grp, c0, w);
        if (tid < kCols) at[tid] = r.orig(c0 + min(tid, w - 1));
    }
    if (tid >= kCols && tid < kCols + kRows && grp == 0) s_own[tid - kCols] = r.orig(r.t0 + min(tid - kCols, r.n - 1));
    __syncthreads();
    Chunks<kCols, DP> next;
    if (grp < r.n_tiles) next.load(Kh, at, c.d);
    if (grp == 0) {
        Chunks<kRows, DP> q;
        q.load(Q + r.bh * c.d, s_own, c.d);
        q.store(sQ);
    }
    __syncthreads();  // Q is there
    float m[kMine], l[kMine], acc[kMine][DP / 16];
#pragma unroll
    for (int j = 0; j < kMine; ++j) {
        m[j] = -INFINITY;
        l[j] = 0.f;
#pragma unroll
        for (int i = 0; i < DP / 16; ++i) acc[j][i] = 0.f;
    }

#pragma unroll 1
    for (int i = grp; i < r.n_tiles; i += 2) {
        const int t_c0 = c0, t_w = w;
        int k0, k1;
        r.span(i, c0, w, k0, k1);
        next.store(sK);  // (K of the tile before was read ahead of the group's last meeting)
        next.load(Vh, at, c.d);
        int next_at = 0;  // look-ups for the tile after this one, a phase ahead of the loads that need them
        if (i + 2 < r.n_tiles) {
            r.tile(i + 2, c0, w);
            if (tid < kCols) next_at = r.orig(c0 + min(tid, w - 1));
        }
        group_sync();
        float s[kMine][4];
        if (k1 > k0) scores<DP>(s, sQ, sK, row0, tx, k0, k1);
        next.store(sV);
        if (tid < kCols) at[tid] = next_at;
        group_sync();
        if (i + 2 < r.n_tiles) next.load(Kh, at, c.d);
        if (k1 <= k0) continue;
#pragma unroll
        for (int j = 0; j < kMine; ++j) {
            float mx = -INFINITY;
            int lo, hi;
            r.row_span(i, t_c0, t_w, row0 + j, lo, hi);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int col = tx + 16 * q;
                s[j][q] = col >= lo && col < hi ? c.scale * s[j][q] : -INFINITY;
                mx = fmaxf(mx, s[j][q]);
            }
            const float m_new = fmaxf(m[j], half_max(mx));
            const float base = m_new == -INFINITY ? 0.f : m_new;  // no key yet
            const float alpha = expf(m[j] - base);
            float sum = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float p = expf(s[j][q] - base);
                sP[(row0 + j) * kPStride + tx + 16 * q] = p;
                sum += p;
            }
            l[j] = l[j] * alpha + half_sum(sum);
            m[j] = m_new;
#pragma unroll
            for (int e = 0; e < DP / 16; ++e) acc[j][e] *= alpha;
        }
        __syncwarp();
        accumulate<DP>(acc, sP, sV, row0, tx, k0, k1);
        __syncwarp();
    }
    if (r.n_tiles > 1) {  // the second group's part, through its shared memory
        float *x = part + kPart + threadIdx.x % kGroup;
        __syncthreads();
        if (grp == 1) {
#pragma unroll
            for (int j = 0; j < kMine; ++j) {
                *x = m[j], x += kGroup;
                *x = l[j], x += kGroup;
#pragma unroll
                for (int e = 0; e < DP / 16; ++e) *x = acc[j][e], x += kGroup;
            }
        }
        __syncthreads();
        if (grp == 0) {
#pragma unroll
            for (int j = 0; j < kMine; ++j) {
                const float m1 = *x, m_new = fmaxf(m[j], m1), base = m_new == -INFINITY ? 0.f : m_new;
                const float f0 = expf(m[j] - base), f1 = expf(m1 - base);
                x += kGroup;
                l[j] = l[j] * f0 + *x * f1, x += kGroup;
                m[j] = m_new;
#pragma unroll
                for (int e = 0; e < DP / 16; ++e) acc[j][e] = acc[j][e] * f0 + *x * f1, x += kGroup;
            }
        }
    }
    if (grp != 0) return;
#pragma unroll
    for (int j = 0; j < kMine; ++j) {
        if (row0 + j >= r.n) continue;
        const int k = s_own[row0 + j];
        // a valid row attends at least to itself, except in the passes of the row-or-column pattern,
        // where a row may have no key at all: O = 0, LSE = -inf
        store_row<T, DP>(O + (r.bh + k) * c.d, acc[j], l[j] > 0.f ? 1.f / l[j] : 0.f, tx, c.d);
        if (tx == 0) LSE[r.bh + k] = m[j] + logf(l[j]);
    }
}

// ---------------------------------------------------------------------------------- backward
// D_k = sum_e dO_ke O_ke, original token order, 16 lanes per row.
template <typename T>
__global__ void __launch_bounds__(kThreads) simt_rowdot_kernel(const T *__restrict__ dO, const T *__restrict__ O,
                                                               float *__restrict__ D, size_t rows, int d) {
    ptx::wait_prior_grid();
    const size_t r = (size_t)blockIdx.x * (kThreads / 16) + (threadIdx.x >> 4);
    const int tx = threadIdx.x & 15;
    float acc = 0.f;
    if (r < rows)
        for (int e = tx * 4; e < d; e += 64) {
            const float4 a = load4(dO + r * d + e), b = load4(O + r * d + e);
            acc = fmaf(a.x, b.x, fmaf(a.y, b.y, fmaf(a.z, b.z, fmaf(a.w, b.w, acc))));
        }
    acc = half_sum(acc);
    if (tx == 0 && r < rows) D[r] = acc;
}

template <typename T>
struct BwdArgs {
    const T *Q, *K, *V, *dO;
    const float *LSE, *D;
    T *dQ, *dK, *dV;
    Common c;
    int H, n_bh;
};
// Even blockIdx.x: the block owns key rows and produces dV = P^T dO and dK = scale dS^T Q from the queries that attend
// to them; odd: it owns query rows and produces dQ = scale dS K.
template <typename T, int DP>
__global__ void __launch_bounds__(kThreads, DP <= 64 ? 2 : 1) simt_bwd_kernel(const BwdArgs<T> a) {
    extern __shared__ __align__(16) float smem[];
    __shared__ RowBlock::Shared s_rows;
    __shared__ int s_col[2][kCols], s_own[kRows];  // original rows of each group's tile, of the block
    __shared__ float s_row[2][kRows];                          // LSE, D of the block's rows (query side)
    constexpr int kR = kRows * (DP + 4), kC = kCols * (DP + 4), kPart = 2 * kC + kRows * kPStride + 2 * kCols;
    // P waits in shared memory for dP where it would not fit into the registers: with heads of 64 and P in registers 144 / 104 bytes are
    // spilled and read back (bf16 tensors 176 / 96) instead of 4 / 4, and 2 x 512 / 8 x 512 tokens take 52.5 / 195 us instead of 50.0 / 186;
    // heads of 16, 32 and 128, which do not spill, 22.4, 30.6 and 90.6 us with P in registers and 23.5, 31.3 and 91.2 in shared memory.
    constexpr bool kPShared = DP == 64;
    const int grp = threadIdx.x / kGroup, tid = threadIdx.x % kGroup;
    float *sRa = smem, *sRb = sRa + kR, *part = sRb + kR, *sCa = part + grp * kPart, *sCb = sCa + kC, *sX = sCb + kC,
          *sVec = sX + kRows * kPStride;
    const Common &c = a.c;
    const bool key_side = (blockIdx.x & 1) == 0;
    const int bh = (blockIdx.x >> 1) % a.n_bh, b = bh / a.H, h = bh % a.H;
    const RowBlock r = row_block(c, b, h, (blockIdx.x >> 1) / a.n_bh, &s_rows);
    ptx::wait_prior_grid();
    pad_rows(c, r, b, key_side ? a.dK : a.dQ, key_side ? a.dV : (T *)nullptr, (float *)nullptr);
    if (r.n <= 0) return;
    const int tx = threadIdx.x & 15, row0 = first_row();
    const T *Ca = (key_side ? a.Q : a.K) + r.bh * c.d, *Cb = (key_side ? a.dO : a.V) + r.bh * c.d;

    int *at = s_col[grp];
    int c0 = 0, w = 0, next_at = 0;  // next_at: original row of column tid of the next tile
    if (grp < r.n_tiles) {
        r.tile(grp, c0, w);
        if (tid < kCols) at[tid] = next_at = r.orig(c0 + min(tid, w - 1));
    }
    if (grp == 0 && tid >= kCols && tid < kCols + kRows) {
        const int row = tid - kCols, k = r.orig(r.t0 + min(row, r.n - 1));
        s_own[row] = k;
        s_row[0][row] = a.LSE[r.bh + k];
        s_row[1][row] = a.D[r.bh + k];
    }
    __syncthreads();
    Chunks<kCols, DP> next;
    float n_lse = 0.f, n_D = 0.f;  // of that row (key side)
    auto fetch = [&]() {
        next.load(Ca, at, c.d);
        if (key_side && tid < kCols) {
            n_lse = a.LSE[r.bh + next_at];
            n_D = a.D[r.bh + next_at];
        }
    };
    if (grp < r.n_tiles) fetch();
    {
        Chunks<kRows, DP> x;  // one matrix by each group
        x.load((grp ? (key_side ? a.V : a.dO) : (key_side ? a.K : a.Q)) + r.bh * c.d, s_own, c.d);
        x.store(grp ? sRb : sRa);
    }
    float acc0[kMine][DP / 16], acc1[kMine][DP / 16];
#pragma unroll
    for (int j = 0; j < kMine; ++j)
#pragma unroll
        for (int i = 0; i < DP / 16; ++i) acc0[j][i] = acc1[j][i] = 0.f;
    __syncthreads();  // the rows are there

#pragma unroll 1
    for (int i = grp; i < r.n_tiles; i += 2) {
        const int t_c0 = c0, t_w = w;
        int k0, k1;
        r.span(i, c0, w, k0, k1);
        group_sync();  // the tile before has been read
        next.store(sCa);
        if (key_side && tid < kCols) {
            sVec[tid] = n_lse;
            sVec[kCols + tid] = n_D;
        }
        next.load(Cb, at, c.d);
        if (i + 2 < r.n_tiles) {  // look-ups for the tile after this one, a phase ahead of the loads that need them
            r.tile(i + 2, c0, w);
            if (tid < kCols) next_at = r.orig(c0 + min(tid, w - 1));
        }
        group_sync();
        float s[kMine][4];
        if constexpr (kPShared) {
            if (k1 > k0) {
                scores<DP>(s, sRa, sCa, row0, tx, k0, k1);
#pragma unroll
                for (int j = 0; j < kMine; ++j) {
                    int lo, hi;
                    r.row_span(i, t_c0, t_w, row0 + j, lo, hi);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int col = tx + 16 * q;
                        const float lse = key_side ? sVec[col] : s_row[0][row0 + j];
                        sX[(row0 + j) * kPStride + col] = col >= lo && col < hi ? expf(c.scale * s[j][q] - lse) : 0.f;
                    }
                }
            }
            next.store(sCb);
            if (tid < kCols) at[tid] = next_at;
            group_sync();
            if (k1 > k0) {
                if (key_side) {
                    __syncwarp();
                    accumulate<DP>(acc1, sX, sCb, row0, tx, k0, k1);
                }
                scores<DP>(s, sRb, sCb, row0, tx, k0, k1);
                __syncwarp();
#pragma unroll
                for (int j = 0; j < kMine; ++j) {
                    int lo, hi;
                    r.row_span(i, t_c0, t_w, row0 + j, lo, hi);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int col = tx + 16 * q;
                        const float D = key_side ? sVec[kCols + col] : s_row[1][row0 + j];
                        float &x = sX[(row0 + j) * kPStride + col];
                        x = col >= lo && col < hi ? x * (s[j][q] - D) : 0.f;
                    }
                }
            }
        } else {
            float dp[kMine][4];
            if (k1 > k0) scores<DP>(s, sRa, sCa, row0, tx, k0, k1);
            next.store(sCb);
            if (tid < kCols) at[tid] = next_at;
            group_sync();
            if (k1 > k0) {
                scores<DP>(dp, sRb, sCb, row0, tx, k0, k1);
#pragma unroll
                for (int j = 0; j < kMine; ++j) {
                    int lo, hi;
                    r.row_span(i, t_c0, t_w, row0 + j, lo, hi);
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int col = tx + 16 * q;
                        const float lse = key_side ? sVec[col] : s_row[0][row0 + j], D = key_side ? sVec[kCols + col] : s_row[1][row0 + j];
                        const bool on = col >= lo && col < hi;
                        const float p = on ? expf(c.scale * s[j][q] - lse) : 0.f;
                        s[j][q] = p;
                        sX[(row0 + j) * kPStride + col] = on ? p * (dp[j][q] - D) : 0.f;
                    }
                }
            }
        }
        if (i + 2 < r.n_tiles) fetch();  // (no earlier: registers)
        if (k1 <= k0) continue;
        __syncwarp();
        accumulate<DP>(acc0, sX, sCa, row0, tx, k0, k1);
        __syncwarp();
        if (!kPShared && key_side) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
#pragma unroll
                for (int j = 0; j < kMine; ++j) sX[(row0 + j) * kPStride + tx + 16 * q] = s[j][q];
            __syncwarp();
            accumulate<DP>(acc1, sX, sCb, row0, tx, k0, k1);
            __syncwarp();
        }
    }
    if (r.n_tiles > 1) {  // the second group's part, through its shared memory
        float *x = part + kPart + tid;
        __syncthreads();
        if (grp == 1) {
#pragma unroll
            for (int j = 0; j < kMine; ++j)
#pragma unroll
                for (int e = 0; e < DP / 16; ++e, x += 2 * kGroup) x[0] = acc0[j][e], x[kGroup] = acc1[j][e];
        }
        __syncthreads();
        if (grp == 0) {
#pragma unroll
            for (int j = 0; j < kMine; ++j)
#pragma unroll
                for (int e = 0; e < DP / 16; ++e, x += 2 * kGroup) acc0[j][e] += x[0], acc1[j][e] += x[kGroup];
        }
    }
    if (grp != 0) return;
#pragma unroll
    for (int j = 0; j < kMine; ++j) {
        if (row0 + j >= r.n) continue;
        const size_t o = (r.bh + s_own[row0 + j]) * c.d;
        store_row<T, DP>((key_side ? a.dK : a.dQ) + o, acc0[j], c.scale, tx, c.d);
        if (key_side) store_row<T, DP>(a.dV + o, acc1[j], 1.f, tx, c.d);
    }
}

Common common(const mate_plan_t *pl, int d, float scale, int view_order) {
    Common c;
    c.rowv = pl->view[0];
    c.colv = pl->view[1];
    c.head_view = pl->head_view_dev;
    c.n_valid = pl->n_valid_dev;
    c.prefix = pl->global_dev;
    c.N = pl->N;
    c.d = d;
    c.view_order = view_order;
    c.scale = scale;
    c.tr = pl->rows();
    return c;
}
// Blocks of a launch per side: row blocks of every (example, head).
inline size_t n_blocks(const mate_plan_t *pl) { return (size_t)((pl->N + kRows - 1) / kRows) * pl->B * pl->H; }

template <typename T, int DP>
int fwd_launch(const mate_plan_t *pl, const void *Q, const void *K, const void *V, int d, float scale, void *O, float *LSE,
               int view_order, cudaStream_t st) {
    static SmemAttrOnce attr;
    constexpr int bytes = 4 * ((kRows + 4 * kCols) * (DP + 4) + 2 * kRows * kPStride);
    if (attr.ensure((const void *)simt_fwd_kernel<T, DP>, bytes, pl->device) != MATE_OK) return MATE_ERR_CUDA;
    return launch_after(simt_fwd_kernel<T, DP>, dim3((unsigned)n_blocks(pl)), kThreads, bytes, st, (const T *)Q, (const T *)K, (const T *)V,
                        (T *)O, LSE, common(pl, d, scale, view_order), pl->H, pl->B * pl->H) == cudaSuccess
               ? MATE_OK
               : MATE_ERR_CUDA;
}
template <typename T, int DP>
int bwd_launch(const mate_plan_t *pl, const void *Q, const void *K, const void *V, const void *O, const float *LSE, const void *dO,
               int d, float scale, void *dQ, void *dK, void *dV, float *D, int pass, cudaStream_t st) {
    static SmemAttrOnce attr;
    constexpr int bytes = 4 * (2 * (kRows + 2 * kCols) * (DP + 4) + 2 * kRows * kPStride + 4 * kCols);
    if (attr.ensure((const void *)simt_bwd_kernel<T, DP>, bytes, pl->device) != MATE_OK) return MATE_ERR_CUDA;
    const size_t rows = pl->n_rows();
    if (pass == 0 && launch_after(simt_rowdot_kernel<T>, dim3((unsigned)((rows + kThreads / 16 - 1) / (kThreads / 16))), kThreads, 0, st,
                                  (const T *)dO, (const T *)O, D, rows, d) != cudaSuccess)
        return MATE_ERR_CUDA;
    const BwdArgs<T> a{(const T *)Q, (const T *)K, (const T *)V, (const T *)dO, LSE, D, (T *)dQ, (T *)dK, (T *)dV,
                       common(pl, d, scale, 0), pl->H, pl->B * pl->H};
    return launch_after(simt_bwd_kernel<T, DP>, dim3((unsigned)(2 * n_blocks(pl))), kThreads, bytes, st, a) == cudaSuccess
               ? MATE_OK
               : MATE_ERR_CUDA;
}

// Head size padded (in shared memory, with zeros) to 16, 32, 64 or 128.
template <typename F>
int by_head_size(int d, F &&f) {
    if (d <= 16) return f(std::integral_constant<int, 16>{});
    if (d <= 32) return f(std::integral_constant<int, 32>{});
    if (d <= 64) return f(std::integral_constant<int, 64>{});
    return f(std::integral_constant<int, 128>{});
}

}  // namespace

int simt_fwd(const mate_plan_t *plan, const void *Q, const void *K, const void *V, int d, int dtype,
             float scale, void *O, float *LSE, unsigned flags, cudaStream_t stream) {
    if (d > kMaxD || 2 * n_blocks(plan) > 0x7fffffffu) return MATE_ERR_UNSUPPORTED;
    const int vo = (flags & MATE_FLAG_VIEW_ORDER) ? 1 : 0;
    if (dtype == MATE_F32)
        return by_head_size(d, [&](auto dp) { return fwd_launch<float, dp()>(plan, Q, K, V, d, scale, O, LSE, vo, stream); });
    return by_head_size(d, [&](auto dp) { return fwd_launch<__nv_bfloat16, dp()>(plan, Q, K, V, d, scale, O, LSE, vo, stream); });
}

size_t simt_bwd_workspace(const mate_plan_t *plan) {
    return sizeof(float) * (size_t)plan->B * plan->H * plan->N;
}

// pass: which of the calls that share the workspace, O and dO this is; the row dots are formed in pass 0.
int simt_bwd(const mate_plan_t *plan, const void *Q, const void *K, const void *V, const void *O,
             const float *LSE, const void *dO, int d, int dtype, float scale, void *dQ, void *dK,
             void *dV, void *workspace, int pass, cudaStream_t stream) {
    if (d > kMaxD || 2 * n_blocks(plan) > 0x7fffffffu) return MATE_ERR_UNSUPPORTED;
    float *D = (float *)workspace;
    if (dtype == MATE_F32)
        return by_head_size(d, [&](auto dp) {
            return bwd_launch<float, dp()>(plan, Q, K, V, O, LSE, dO, d, scale, dQ, dK, dV, D, pass, stream);
        });
    return by_head_size(d, [&](auto dp) {
        return bwd_launch<__nv_bfloat16, dp()>(plan, Q, K, V, O, LSE, dO, d, scale, dQ, dK, dV, D, pass, stream);
    });
}

}  // namespace mate

// Allocation-free backward (see mate.h).  The name g_noalloc_rowdot is only a host-side handle
// here; the address the kernels need comes from cudaGetSymbolAddress, looked up once per device
// with that device current.
extern "C" int mate_attn_bwd_noalloc(const mate_plan_t *plan, const void *Q, const void *K,
                                     const void *V, const void *O, const float *LSE,
                                     const void *dO, int d, int dtype, float scale, void *dQ,
                                     void *dK, void *dV, void *stream) {
    constexpr int kMaxDevices = 64;
    static std::mutex mu;
    static float *scratch_of_device[kMaxDevices] = {};

    if (!plan || !Q || !K || !V || !O || !LSE || !dO || !dQ || !dK || !dV) return MATE_ERR_INVALID_ARG;
    if (dtype != MATE_BF16 && dtype != MATE_F32) return MATE_ERR_UNSUPPORTED;
    if (d <= 0 || d % 8 != 0 || d > mate::kMaxD) return MATE_ERR_UNSUPPORTED;
    const void *ptrs[] = {Q, K, V, O, LSE, dO, dQ, dK, dV};
    for (const void *p : ptrs)
        if (reinterpret_cast<uintptr_t>(p) & 15u) return MATE_ERR_ALIGNMENT;
    if (plan->sub[0]) return MATE_ERR_UNSUPPORTED;  // row-or-column plans need the three-pass path
    const size_t rows = (size_t)plan->B * plan->H * plan->N;
    if (rows > mate::kNoAllocMaxRows) return MATE_ERR_TOO_LARGE;

    if (mate::use_plan(plan, (cudaStream_t)stream) != cudaSuccess) return MATE_ERR_CUDA;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return MATE_ERR_CUDA;
    if (dev < 0 || dev >= kMaxDevices) return MATE_ERR_UNSUPPORTED;
    if (dev != plan->device) return MATE_ERR_INVALID_ARG;  // the plan's arrays live on another device
    float *scratch = nullptr;
    {
        std::lock_guard<std::mutex> lock(mu);
        if (!scratch_of_device[dev]) {
            float *p = nullptr;
            if (cudaGetSymbolAddress((void **)&p, mate::g_noalloc_rowdot) != cudaSuccess || !p)
                return MATE_ERR_CUDA;
            scratch_of_device[dev] = p;
        }
        scratch = scratch_of_device[dev];
    }
    // every element of D that the backward kernels read is written by the row-dot kernel of the
    // same call first, so nothing in the shared array has to start at zero
    return mate::simt_bwd(plan, Q, K, V, O, LSE, dO, d, dtype, scale, dQ, dK, dV, scratch, 0,
                          (cudaStream_t)stream);
}
