// Memory that outlives one plan: device blocks and pinned staging buffers.  A cudaMalloc / cudaFree pair per plan
// waits for the whole device; a training step that plans every new batch spent most of its time there.
// Bounded (kMaxBlocks blocks and kMaxBytes bytes of cached device memory, kMaxStaging buffers of at most
// kMaxStagingBytes), emptied when an allocation fails, safe with several threads and streams.
#include <algorithm>
#include <cstdlib>
#include <vector>

#include "mate_internal.h"

namespace mate {
namespace {

constexpr size_t kMaxBlocks = 16, kMaxBytes = size_t(64) << 20;
constexpr size_t kMaxStaging = 8, kMaxStagingBytes = size_t(4) << 20;

std::mutex g_mu;
std::vector<Block> g_blocks;      // free blocks, oldest first
std::vector<Staging> g_staging;   // free staging buffers

size_t granule(size_t bytes) { return (std::max<size_t>(bytes, 1) + 65535) / 65536 * 65536; }

void free_all(std::vector<Block> &blocks) {
    for (Block &b : blocks) cudaFree(b.ptr);
    blocks.clear();
}

}  // namespace

uint64_t stream_id(cudaStream_t st) {
    unsigned long long id = 0;
    if (cudaStreamGetId(st, &id) != cudaSuccess) {
        cudaGetLastError();
        return 0;  // unknown: never equal to another one
    }
    return (uint64_t)id + 1;
}

// A block for work on `st` of device `device` (the current one).  A cached block that was last used on the same
// stream is ordered behind that use; any other one waits for the device first, as freeing it would have.
bool pool_take(size_t bytes, cudaStream_t st, int device, Block *out) {
    const size_t need = granule(bytes);
    const uint64_t id = stream_id(st);
    {
        std::unique_lock<std::mutex> lock(g_mu);
        int best = -1;
        for (int i = 0; i < (int)g_blocks.size(); ++i) {
            const Block &b = g_blocks[i];
            if (b.device != device || b.bytes < need || b.bytes > 4 * need) continue;
            const auto rank = [&](const Block &x) { return std::make_pair(!(x.stream == id && id != 0), x.bytes); };
            if (best < 0 || rank(b) < rank(g_blocks[best])) best = i;
        }
        if (best >= 0) {
            *out = g_blocks[best];
            g_blocks.erase(g_blocks.begin() + best);
            lock.unlock();
            if (out->stream != id || id == 0) {
                if (cudaDeviceSynchronize() != cudaSuccess) {
                    cudaFree(out->ptr);
                    *out = Block{};  // nothing for the caller to give back
                    return false;
                }
            }
            out->stream = id;
            return true;
        }
    }
    *out = Block{nullptr, need, device, id};
    if (cudaMalloc(&out->ptr, need) == cudaSuccess) return true;
    cudaGetLastError();
    {
        std::lock_guard<std::mutex> lock(g_mu);
        free_all(g_blocks);
    }
    if (cudaMalloc(&out->ptr, need) == cudaSuccess) return true;
    cudaGetLastError();
    out->ptr = nullptr;
    return false;
}

// `stream`: id of the only stream that has used the block, 0 if there may have been others.
void pool_give(Block &b, uint64_t stream) {
    if (!b.ptr) return;
    b.stream = stream;
    std::vector<Block> drop;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        g_blocks.push_back(b);
        size_t total = 0;
        for (const Block &x : g_blocks) total += x.bytes;
        while (g_blocks.size() > kMaxBlocks || total > kMaxBytes) {
            total -= g_blocks.front().bytes;
            drop.push_back(g_blocks.front());
            g_blocks.erase(g_blocks.begin());
        }
    }
    free_all(drop);
    b = Block{};
}

// Host memory to copy from or to: pinned up to kMaxStagingBytes, ordinary memory above (the copies are then
// not asynchronous).
bool staging_take(size_t bytes, int device, Staging *out) {
    if (bytes > kMaxStagingBytes) {
        *out = Staging{malloc(bytes), bytes, device, nullptr};
        return out->ptr != nullptr;
    }
    const size_t need = granule(bytes);
    {
        std::unique_lock<std::mutex> lock(g_mu);
        for (size_t i = 0; i < g_staging.size(); ++i)
            if (g_staging[i].device == device && g_staging[i].bytes >= need) {
                *out = g_staging[i];
                g_staging.erase(g_staging.begin() + i);
                lock.unlock();
                return cudaEventSynchronize(out->event) == cudaSuccess;  // copies out of it are complete
            }
    }
    *out = Staging{nullptr, need, device, nullptr};
    if (cudaHostAlloc(&out->ptr, need, cudaHostAllocDefault) != cudaSuccess) {
        cudaGetLastError();
        out->ptr = nullptr;
        return false;
    }
    if (cudaEventCreateWithFlags(&out->event, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        cudaFreeHost(out->ptr);
        out->ptr = nullptr;
        return false;
    }
    return true;
}

// Copies out of the buffer may still be running on `st`.
void staging_give(Staging &s, cudaStream_t st) {
    if (!s.ptr) return;
    if (!s.event) {
        cudaStreamSynchronize(st);
        free(s.ptr);
    } else {
        bool keep = cudaEventRecord(s.event, st) == cudaSuccess;
        if (!keep) cudaGetLastError();
        if (keep) {
            std::lock_guard<std::mutex> lock(g_mu);
            keep = g_staging.size() < kMaxStaging;
            if (keep) g_staging.push_back(s);
        }
        if (!keep) {
            cudaStreamSynchronize(st);
            cudaEventDestroy(s.event);
            cudaFreeHost(s.ptr);
        }
    }
    s = Staging{};
}

cudaError_t use_plan(const mate_plan_t *plan, cudaStream_t st) {
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaError_t rc = cudaStreamIsCapturing(st, &capture);
    if (rc != cudaSuccess) return rc;
    if (capture == cudaStreamCaptureStatusNone && plan->stream != 0 && stream_id(st) == plan->stream) return cudaSuccess;
    plan->elsewhere = true;
    std::lock_guard<std::mutex> lock(plan->ready_mu);
    if (!plan->ready) return cudaSuccess;
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;  // a wait for work that is not part of the capture
    cudaThreadExchangeStreamCaptureMode(&mode);
    rc = cudaEventSynchronize(plan->ready);
    if (rc == cudaSuccess) {
        cudaEventDestroy(plan->ready);
        plan->ready = nullptr;
    }
    cudaThreadExchangeStreamCaptureMode(&mode);
    return rc;
}

}  // namespace mate
