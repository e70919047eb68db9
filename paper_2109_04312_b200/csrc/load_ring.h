// A ring of shared-memory buffers between the loader warps and the readers of what they load.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define MATE_HD __host__ __device__ __forceinline__
#else
#define MATE_HD inline
#endif

namespace mate {

// Load n goes into buffer n % kBuffers once the readers of load n - kBuffers are done; the buffer has one barrier for "landed"
// and one for "released", both waited for by parity.  A parity tells a phase from its neighbours only, so whoever
// waits has to know that the phase before the awaited one is over.  It is because every loader warp has a part in every load:
// it has waited for the buffer's release before, and the buffer is not read, let alone released, without its part of the load.
// (Loads dealt to two teams of warps in turn break that: a team can come to load n while load n - 2 kBuffers is still
// being read, and its wait passes for a phase too early.  tests/test_load_ring.py runs the roles of the kernels in random
// interleavings, with both.)
template <uint32_t kBuffers>
struct LoadRing {
    static_assert((kBuffers & (kBuffers - 1)) == 0, "counters wrap around");
    MATE_HD static uint32_t buffer(uint32_t n) { return n % kBuffers; }
    MATE_HD static uint32_t full_parity(uint32_t n) { return (n / kBuffers) & 1; }
    // The first kBuffers loads pass at once: parity 1 of a barrier without a phase behind it.
    MATE_HD static uint32_t wait_parity(uint32_t n) { return ((n / kBuffers) & 1) ^ 1; }
};

}  // namespace mate
