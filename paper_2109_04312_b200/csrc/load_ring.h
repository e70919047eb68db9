// Barriers of a ring of shared-memory buffers whose loads are dealt to teams of warps in turn.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define MATE_HD __host__ __device__ __forceinline__
#else
#define MATE_HD inline
#endif

namespace mate {

// Load n goes into buffer n % kBuffers once the readers of load n - kBuffers are done; readers of load n arrive on
// barrier empty(n).  A wait by parity tells a phase from its neighbours only, so whoever waits has to know that the phase before
// the awaited one is over.  A warp that does every load has waited for that phase itself; a team that does every
// other load has not, and with one barrier per buffer it can come to load n while load n - 2 kBuffers is still being
// read: the wait then passes for a phase too early.  With two barriers per buffer the phase before the awaited one is the
// release of load n - 3 kBuffers, which is over whenever load n - 2 kBuffers has been made.  That this is so
// when a team waits for load n:
//   rows (2 buffers; load n belongs to item n): record n is published when the arithmetic warps (forward: softmax
//     warps) have let record n - 4 go, which they do behind their wait for its rows.
//   tiles (4 buffers): the team's step before the one of tile c is
//     - tile c - 1 or c - 2, for which it has waited for the readers of tile c - 5 or c - 6.  They take the tiles in
//       order, so tile c - 8 had landed.
//     - or the rows of an item m, with no tile or only tile c - 1 in between.  For these it has waited until item m - 2 was
//       done with.  So tile c - 8 has landed, unless it is one of item m - 1; then at least six more tiles of that
//       item follow it, the team loaded one of the last two, and the case above applies.
// tests/test_load_ring.py runs the roles of both kernels in random interleavings; with one barrier per buffer waits pass early.
template <uint32_t kBuffers, uint32_t kBarriers = 2 * kBuffers>
struct LoadRing {
    static_assert((kBuffers & (kBuffers - 1)) == 0 && (kBarriers & (kBarriers - 1)) == 0, "counters wrap around");
    static constexpr uint32_t kEmpty = kBarriers;  // barriers on the empty side
    MATE_HD static uint32_t buffer(uint32_t n) { return n % kBuffers; }
    MATE_HD static uint32_t full_parity(uint32_t n) { return (n / kBuffers) & 1; }
    MATE_HD static uint32_t empty(uint32_t n) { return n % kEmpty; }
    // What load n waits for.  The first kBuffers loads pass at once: parity 1 of a barrier without a phase behind it.
    MATE_HD static uint32_t wait_empty(uint32_t n) { return empty(n - kBuffers); }
    MATE_HD static uint32_t wait_parity(uint32_t n) { return ((n - kBuffers) / kEmpty) & 1; }
};

}  // namespace mate
