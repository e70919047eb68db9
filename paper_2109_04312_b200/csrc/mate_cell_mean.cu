// Per-cell mean of token logits (cell-selection stage, Section 4.1: S(c) = avg over the tokens t of
// cell c of S(t)).  A cell is the set of table tokens that share a (row id, column id) pair.  In the
// row view of the plan the tokens of one row are contiguous, so one block takes one row: it brings the
// row's (column id, logit) pairs into shared memory, all threads loading, and thread c then reads them in the
// order of the tokens and accumulates column c (the result does not depend on the launch).  Bound by
// latency at the sizes of a table: two dependent loads, then about four instructions per token of the row.
// (One warp per row, 32 tokens at a time handed around by shuffles, took 7 us for rows of 30 tokens and 93 us
// for rows of several hundred; this takes 2.3 and 6.3.)
#include "mate_internal.h"
#include "sm100_ptx.cuh"

namespace mate {
namespace {

constexpr int kThreads = 128;
constexpr int kBuf = 1024;  // tokens of a row in shared memory at a time

__global__ void __launch_bounds__(kThreads)
cell_mean_kernel(const float *__restrict__ logits, const int32_t *__restrict__ col_ids, ViewPlan rowv, int N,
                 int n_rows, int n_cols, float *__restrict__ mean, int32_t *__restrict__ count) {
    __shared__ __align__(16) int32_t s_col[kBuf];
    __shared__ __align__(16) float s_x[kBuf];
    ptx::launch_dependents();
    ptx::wait_prior_grid();
    const int r = blockIdx.x, b = blockIdx.y;  // row id, example
    const int32_t *seg_off = rowv.seg_off + (size_t)b * (rowv.max_id + 2);
    const int lo = seg_off[r], hi = seg_off[r + 1];
    const int32_t *perm = rowv.perm + (size_t)b * N;
    const size_t out = ((size_t)b * n_rows + r) * n_cols;

    for (int c0 = 0; c0 < n_cols; c0 += kThreads) {
        const int c = c0 + (int)threadIdx.x;
        float sum = 0.f;
        int cnt = 0;
        for (int t0 = lo; t0 < hi; t0 += kBuf) {
            const int n = min(kBuf, hi - t0), n4 = (n + 3) & ~3;
            if (c0 > 0 || t0 > lo) __syncthreads();  // the buffer has been read
            for (int i = threadIdx.x; i < n4; i += kThreads) {
                const size_t at = (size_t)b * N + perm[t0 + min(i, n - 1)];
                s_col[i] = i < n ? col_ids[at] : -1;
                s_x[i] = logits[at];
            }
            __syncthreads();
            if (c < n_cols)
#pragma unroll 2
                for (int i = 0; i < n4; i += 4) {
                    const int4 k = *reinterpret_cast<const int4 *>(s_col + i);
                    const float4 x = *reinterpret_cast<const float4 *>(s_x + i);
                    if (k.x == c) sum += x.x, ++cnt;
                    if (k.y == c) sum += x.y, ++cnt;
                    if (k.z == c) sum += x.z, ++cnt;
                    if (k.w == c) sum += x.w, ++cnt;
                }
        }
        if (c < n_cols) {
            mean[out + c] = cnt ? sum / (float)cnt : 0.f;
            if (count) count[out + c] = cnt;
        }
    }
}

}  // namespace
}  // namespace mate

extern "C" int mate_cell_mean(const mate_plan_t *plan, const float *logits, const int32_t *col_ids, float *mean,
                              int32_t *count, void *stream) {
    if (!plan || !logits || !col_ids || !mean) return MATE_ERR_INVALID_ARG;
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return MATE_ERR_CUDA;
    if (dev != plan->device) return MATE_ERR_INVALID_ARG;
    if (plan->T) return MATE_ERR_UNSUPPORTED;  // packed batches: not here
    if (mate::use_plan(plan, (cudaStream_t)stream) != cudaSuccess) return MATE_ERR_CUDA;
    const int n_rows = plan->view[0].max_id + 1, n_cols = plan->view[1].max_id + 1;
    return mate::launch_after(mate::cell_mean_kernel, dim3(n_rows, plan->B), mate::kThreads, 0, (cudaStream_t)stream, logits, col_ids,
                              plan->view[0], plan->N, n_rows, n_cols, mean, count) == cudaSuccess
               ? MATE_OK
               : MATE_ERR_CUDA;
}
