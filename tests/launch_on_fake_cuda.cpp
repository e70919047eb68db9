// The host side of the tensor-core kernels (csrc/mate_fwd_tc.cu, csrc/mate_bwd_tc.cu) on a CUDA runtime of plain host functions:
// a driver without tensor maps, launches that are only counted and looked at.
#include <cstring>

#include "mate_internal.h"

namespace {
int n_launches = 0;
unsigned first_grid = 0;  // of a call's first launch
size_t word_at = 0;  // of the last launch's parameters
int word = -1;
}  // namespace

extern "C" {

void **__cudaRegisterFatBinary(void *) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void **) {}
void __cudaUnregisterFatBinary(void **) {}
void __cudaRegisterFunction(void **, const char *, char *, const char *, int, uint3 *, uint3 *, dim3 *, dim3 *, int *) {}
void __cudaRegisterVar(void **, char *, char *, const char *, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, cudaStream_t) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3 *, dim3 *, size_t *, void *) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t *, const void *) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void **, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaLaunchKernel(const void *, dim3, dim3, void **, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void *, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPoint(const char *, void **fn, unsigned long long, cudaDriverEntryPointQueryResult *res) {
    *fn = nullptr;
    *res = cudaDriverEntryPointSymbolNotFound;
    return cudaErrorInvalidValue;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t *config, const void *, void **args) {
    if (++n_launches == 1) first_grid = config->gridDim.x;
    if (word_at) memcpy(&word, static_cast<const char *>(args[0]) + word_at, sizeof word);
    return cudaSuccess;
}

// status of a call, its launches and whether it asks for bulk copies (the word behind the maps)
int call(int backward, int *launches, int *bulk) {
    static char mem[256];
    mate_plan_s plan;
    plan.B = plan.H = 1;
    plan.N = 64;
    plan.fwd_grid = plan.bwd_grid = 1;
    void *t[mate::kPasses] = {mem, nullptr, nullptr};
    float *l[mate::kPasses] = {(float *)mem, nullptr, nullptr};
    n_launches = 0;
    word_at = 128 * (backward ? 4 : 2);
    const int rc = backward ? mate::tc_bwd(&plan, mem, mem, mem, mem, (float *)mem, mem, 0.125f, t, t, t, mem, nullptr)
                            : mate::tc_fwd(&plan, mem, mem, mem, 0.125f, t, l, mem, 0, nullptr);
    *launches = n_launches;
    *bulk = word;
    return rc;
}

// blocks of the row dots of H heads of N rows on a GPU of n_ctas SMs
int rowdot_grid(int H, int N, int n_ctas) {
    static char mem[256];
    mate_plan_s plan;
    plan.B = 1, plan.H = H, plan.N = N;
    plan.n_ctas = n_ctas;
    plan.bwd_grid = 1;
    void *t[mate::kPasses] = {mem, nullptr, nullptr};
    n_launches = word_at = 0;
    return mate::tc_bwd(&plan, mem, mem, mem, mem, (float *)mem, mem, 0.125f, t, t, t, mem, nullptr) == 0 ? (int)first_grid : -1;
}

// what the backward of a plan asks for (T: tokens of a packed one, N its longest example)
size_t backward_workspace(int B, int H, int N, int T) {
    mate_plan_s plan;
    plan.B = B, plan.H = H, plan.N = N, plan.T = T;
    return mate::tc_bwd_workspace(&plan);
}

}  // extern "C"
