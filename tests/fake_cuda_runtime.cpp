// The memory pool (csrc/mate_pool.cu) on a CUDA runtime of plain host functions that count, and fail on request.
// Streams are numbers; stream 0 has no id (as where the driver does not report one).
#include <cstdlib>
#include <set>

#include "mate_internal.h"

namespace {
std::set<void *> live;     // allocated and not freed
int fail_device_sync = 0, bad_frees = 0, device_syncs = 0, event_waits = 0;
mate::Block blocks[32];
}  // namespace

extern "C" {

cudaError_t cudaStreamGetId(cudaStream_t st, unsigned long long *id) {
    *id = (unsigned long long)(uintptr_t)st;
    return st ? cudaSuccess : cudaErrorNotSupported;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() {
    ++device_syncs;
    return fail_device_sync ? cudaErrorUnknown : cudaSuccess;
}
cudaError_t cudaMalloc(void **p, size_t) {
    *p = malloc(1);
    live.insert(*p);
    return cudaSuccess;
}
cudaError_t cudaFree(void *p) {
    bad_frees += live.erase(p) != 1;  // (the memory itself stays, so that no address comes twice)
    return cudaSuccess;
}
cudaError_t cudaHostAlloc(void **p, size_t n, unsigned) {
    *p = malloc(n);
    return cudaSuccess;
}
cudaError_t cudaFreeHost(void *p) {
    free(p);
    return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t *e, unsigned) {
    *e = (cudaEvent_t)1;
    return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) {
    ++event_waits;
    return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus *s) {
    *s = cudaStreamCaptureStatusNone;
    return cudaSuccess;
}
cudaError_t cudaThreadExchangeStreamCaptureMode(cudaStreamCaptureMode *) { return cudaSuccess; }

// what the tests call
void fake_fail_device_sync(int on) { fail_device_sync = on; }
int fake_bad_frees() { return bad_frees; }
int fake_device_syncs() { return device_syncs; }
int fake_live() { return (int)live.size(); }
int pool_take(int i, size_t bytes, size_t stream) { return mate::pool_take(bytes, (cudaStream_t)stream, 0, &blocks[i]); }
int pool_holds(int i) { return blocks[i].ptr != nullptr; }
int pool_is_live(int i) { return (int)live.count(blocks[i].ptr); }
void pool_give(int i, size_t stream) { mate::pool_give(blocks[i], mate::stream_id((cudaStream_t)stream)); }
// a plan made on one stream, used on another: waits for its upload
int plan_waits(size_t made_on, size_t used_on) {
    mate_plan_s plan;
    plan.stream = mate::stream_id((cudaStream_t)made_on);
    plan.ready = (cudaEvent_t)1;
    const int before = event_waits;
    return mate::use_plan(&plan, (cudaStream_t)used_on) == cudaSuccess ? event_waits - before : -1;
}

}  // extern "C"
