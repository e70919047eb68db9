// Glue kernels of the head-independent row-or-column pattern (the pattern the paper describes for
// its closest comparison system, Section 2): the attention of a row is computed in three passes over
// disjoint key sets by the ordinary kernels; here their outputs are merged (each pass returns a
// normalised O and the logsumexp of its own keys) and their gradients summed.  HBM-bound,
// element-wise work: 16 bytes of every tensor per thread and step.
#include <cuda_bf16.h>

#include "mate_internal.h"
#include "sm100_ptx.cuh"

namespace mate {
namespace {

// 16 bytes of a tensor as floats
template <typename T>
struct Vec;
template <>
struct Vec<float> {
    static constexpr int kN = 4;
    float v[kN];
    __device__ __forceinline__ void load(const void *p, size_t i) {
        const float4 x = reinterpret_cast<const float4 *>(p)[i];
        v[0] = x.x, v[1] = x.y, v[2] = x.z, v[3] = x.w;
    }
    __device__ __forceinline__ void store(void *p, size_t i) const { reinterpret_cast<float4 *>(p)[i] = make_float4(v[0], v[1], v[2], v[3]); }
};
template <>
struct Vec<__nv_bfloat16> {
    static constexpr int kN = 8;
    float v[kN];
    __device__ __forceinline__ void load(const void *p, size_t i) {
        const uint4 x = reinterpret_cast<const uint4 *>(p)[i];
        const uint32_t w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&w[q]));
            v[2 * q] = f.x, v[2 * q + 1] = f.y;
        }
    }
    __device__ __forceinline__ void store(void *p, size_t i) const {
        reinterpret_cast<uint4 *>(p)[i] = make_uint4(ptx::cvt_bf16x2(v[0], v[1]), ptx::cvt_bf16x2(v[2], v[3]),
                                                     ptx::cvt_bf16x2(v[4], v[5]), ptx::cvt_bf16x2(v[6], v[7]));
    }
};

constexpr int kThreads = 256;
constexpr int kRowLanes = 8;  // lanes per row of the merge

// O <- sum_i w_i O_i with w_i = exp(LSE_i - LSE), LSE = log sum_i exp(LSE_i); a pass in which the row has no key
// returns LSE_i = -inf and weighs 0.  O, LSE hold pass 0 on entry.
template <typename T>
__global__ void __launch_bounds__(kThreads)
merge_kernel(void *O, float *LSE, const void *O1, const float *LSE1, const void *O2, const float *LSE2, size_t rows, int d) {
    ptx::launch_dependents();
    ptx::wait_prior_grid();
    const size_t r = (size_t)blockIdx.x * (kThreads / kRowLanes) + threadIdx.x / kRowLanes;
    const bool in = r < rows;
    const float a = in ? LSE[r] : -INFINITY, b = in ? LSE1[r] : -INFINITY, c = in ? LSE2[r] : -INFINITY;
    const float m = fmaxf(a, fmaxf(b, c));
    __syncwarp();  // all lanes of the row have read LSE
    if (m == -INFINITY) return;  // padding row: pass 0 has written O = 0, LSE = -inf
    const float wa = __expf(a - m), wb = __expf(b - m), wc = __expf(c - m);
    const float inv = 1.f / (wa + wb + wc);
    const int chunks = d / Vec<T>::kN;
    for (int e = threadIdx.x % kRowLanes; e < chunks; e += kRowLanes) {
        const size_t i = r * chunks + e;
        Vec<T> x, y, z;
        x.load(O, i);
        y.load(O1, i);
        z.load(O2, i);
#pragma unroll
        for (int q = 0; q < Vec<T>::kN; ++q) x.v[q] = (wa * x.v[q] + wb * y.v[q] + wc * z.v[q]) * inv;
        x.store(O, i);
    }
    if (threadIdx.x % kRowLanes == 0) LSE[r] = m + logf(wa + wb + wc);
}

struct Sums {
    void *a[3];
    const void *b[3], *c[3];
};
// a += b + c for three tensors of n 16-byte words (blockIdx.y: which)
template <typename T>
__global__ void __launch_bounds__(kThreads) add3_kernel(const Sums s, size_t n) {
    ptx::launch_dependents();
    ptx::wait_prior_grid();
    const size_t i = (size_t)blockIdx.x * kThreads + threadIdx.x;
    if (i >= n) return;
    // (Indexed by blockIdx.y the parameters are copied to local memory first: 72 bytes per thread, and the sums of 2 x 1024 tokens
    // with 12 heads of 64 take 4 us more in a backward of 29.2, those of 4 x 2048 12 in 156.)
    const auto which = [](auto *const(&p)[3]) { return blockIdx.y == 0 ? p[0] : blockIdx.y == 1 ? p[1] : p[2]; };
    void *const a = which(s.a);
    Vec<T> x, y, z;
    x.load(a, i);
    y.load(which(s.b), i);
    z.load(which(s.c), i);
#pragma unroll
    for (int q = 0; q < Vec<T>::kN; ++q) x.v[q] = x.v[q] + y.v[q] + z.v[q];
    x.store(a, i);
}

}  // namespace

cudaError_t launch_merge_passes(void *O, float *LSE, const void *O1, const float *LSE1, const void *O2, const float *LSE2,
                                size_t rows, int d, int dtype, cudaStream_t stream) {
    constexpr int per_block = kThreads / kRowLanes;
    const dim3 grid((unsigned)((rows + per_block - 1) / per_block));
    return launch_after(dtype == MATE_F32 ? merge_kernel<float> : merge_kernel<__nv_bfloat16>, grid, kThreads, 0, stream, O, LSE, O1, LSE1,
                        O2, LSE2, rows, d);
}

cudaError_t launch_add3(void *const (&a)[3], void *const (&b)[3], void *const (&c)[3], size_t n, int dtype, cudaStream_t stream) {
    const size_t words = n / (dtype == MATE_F32 ? Vec<float>::kN : Vec<__nv_bfloat16>::kN);  // d is a multiple of 8
    Sums s;
    for (int i = 0; i < 3; ++i) {
        s.a[i] = a[i];
        s.b[i] = b[i];
        s.c[i] = c[i];
    }
    const dim3 grid((unsigned)((words + kThreads - 1) / kThreads), 3);
    return launch_after(dtype == MATE_F32 ? add3_kernel<float> : add3_kernel<__nv_bfloat16>, grid, kThreads, 0, stream, s, words);
}

}  // namespace mate
