// Internal declarations shared by the libmate translation units (not part of the C ABI).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <mutex>
#include <vector>

#include "mate.h"

namespace mate {

constexpr int kTile = 128;       // key columns per tile and query rows per half of a unit
constexpr int kSchedWords = 8;   // scheduling counters of the forward, in front of the split-unit counters
constexpr int kUnitRows = 256;   // query rows per unit of the tensor-core kernels (two halves)
// what the key range of a table row is made of (plan kernel step 4 and its host twin)
enum { kBoundsOwn = 0, kBoundsBefore = 1, kBoundsAfter = 2 };
constexpr int kTraceCtas = 256;  // CTAs whose cycle counters a -DMATE_TRACE build keeps

// x / tB for tiles of tB columns, 0 <= x.  Tiles of fewer than 128 columns come in twos (make_unit), x < 3 tB: a division would
// be 2.5 KB of code in the forward.
__host__ __device__ inline int div_tile(int x, int tB) { return tB == kTile ? x >> 7 : (x >= tB) + (x >= 2 * tB); }
static_assert(kTile == 128, "div_tile");

// A record's head and view in one word: no look-up in front of a unit's first loads.  (The kernels' grids end at 2^30 heads too.)
constexpr int kViewShift = 30;
__host__ __device__ inline int32_t pack_hv(int head, int view) { return (int32_t)((uint32_t)head | (uint32_t)view << kViewShift); }
__host__ __device__ inline int head_of(int32_t hv) { return hv & ((1 << kViewShift) - 1); }
__host__ __device__ inline int view_of(int32_t hv) { return (int)((uint32_t)hv >> kViewShift); }
// Views of a work-list: row, column, and the two further passes of a row-or-column plan, which have outputs of their own.
constexpr int kViews = 4, kPasses = 3;
__host__ __device__ inline int pass_of(int view) { return view < 2 ? 0 : view - 1; }

// One unit of work of the tensor-core kernels: up to 256 consecutive rows (view order) of one (example, head)
// in two halves of up to 128 -- half 0 = the first n0 rows, half 1 = the n1 rows behind them -- and the
// column tiles they visit, in this order:
//   range A = columns [kA0, kA_end) in tiles of 128, all of which count for every row: the global block
//             ([0, P)) for table rows, all valid positions for rows of the global block.
//   range B = the first kP positions of the order (which count for every row), then [kB0, kB_end) = the union of
//             the key ranges of the rows, in tiles of tB <= 128.  Position j of the latter counts for a row
//             iff seg_lo[row] <= j < seg_hi[row]; half h touches only the tiles that meet the first kP
//             positions or [lo[h], hi[h]) (min seg_lo / max seg_hi over its rows).
// The global block is in range A, or in front of range B (kP = P) where that takes fewer tiles.
// A unit of the forward may be split along its tiles (kP = 0) into n_parts units; each writes an un-normalised
// partial result to the workspace at ws_off (KiB); per group of 32 rows the part that finishes
// last (counted in counters[kSchedWords + 8 * ctr + row / 32]) combines them.
struct alignas(16) FwdUnit {  // (copied as four 16-byte words)
    int32_t b, hv;             // hv = pack_hv(head, view)
    int32_t q0, rows;          // rows = n0 | n1 << 8 | kP << 16; 0 ends a list
    int32_t kA0, kA_end;
    int32_t kB0, kB_end;
    int32_t lo[2], hi[2];
    int32_t tB, parts;         // parts = n_parts | part << 16 (tB: the forward keeps flags above bit 7 on its way)
    int32_t ws_off, ctr;

    __host__ __device__ int head() const { return head_of(hv); }
    __host__ __device__ int view() const { return view_of(hv); }
    __host__ __device__ int rows_of(int half) const { return half ? (rows >> 8) & 0xff : rows & 0xff; }
    __host__ __device__ int row0_of(int half) const { return half ? q0 + (rows & 0xff) : q0; }
    __host__ __device__ int kP() const { return rows >> 16; }
    __host__ __device__ int n_parts() const { return parts & 0xffff; }
    __host__ __device__ int part() const { return parts >> 16; }
    __host__ __device__ int tiles_a() const { return kA_end > kA0 ? (kA_end - kA0 + kTile - 1) / kTile : 0; }
    __host__ __device__ int tiles_b() const { return kB_end > kB0 || kP() > 0 ? div_tile(kP() + kB_end - kB0 + tB - 1, tB) : 0; }
};
static_assert(sizeof(FwdUnit) == 64, "FwdUnit is read as four 16-byte words");

// Tile i of a unit (nA = its tiles of range A): w columns (<= 128).  Column c stands for position x0 + c if c < pre
// -- these count for every row -- and for position k0 + c otherwise.
struct TileInfo {
    int x0, k0, w, pre;
    bool is_b;
    __host__ __device__ int pos(int c) const { return c < pre ? x0 + c : k0 + c; }
    // one run of positions, starting at first()
    __host__ __device__ bool contiguous() const { return pre == 0 || pre == w || k0 == x0; }
    __host__ __device__ int first() const { return pre > 0 ? x0 : k0; }
};
__host__ __device__ inline TileInfo tile_info(const FwdUnit &u, int i, int nA) {
    TileInfo t;
    t.is_b = i >= nA;
    t.x0 = t.is_b ? (i - nA) * u.tB : u.kA0 + i * kTile;
    const int kP = u.kP(), left = (t.is_b ? kP + u.kB_end - u.kB0 : u.kA_end) - t.x0, most = t.is_b ? u.tB : kTile;
    t.w = left < most ? left : most;
    t.k0 = t.is_b ? t.x0 + u.kB0 - kP : t.x0;
    t.pre = !t.is_b ? t.w : kP <= t.x0 ? 0 : kP - t.x0 < t.w ? kP - t.x0 : t.w;
    return t;
}
// Columns [c0, c1) of the tile (multiples of 16) needed by a half whose rows' key ranges span [lo, hi);
// c1 <= c0 when it skips the tile.
__host__ __device__ inline void half_cols(int lo, int hi, const TileInfo &t, int &c0, int &c1) {
    const int a = lo > t.k0 ? lo - t.k0 : 0, b = hi < t.k0 + t.w ? hi - t.k0 : t.w;
    const bool meets = t.is_b && a < b;
    c0 = t.pre > 0 ? 0 : a & ~15;
    c1 = meets && b > t.pre ? (b + 15) & ~15 : t.pre > 0 ? (t.pre + 15) & ~15 : c0;
}
// bytes of one partial result: 256 rows x (64 fp32 + base, row sum, two unused)
constexpr size_t kPartialBytes = (size_t)kUnitRows * (64 + 4) * sizeof(float);

// Up to kPadRows padding rows (view positions t0 ..) of one (example, head); zeroed by the forward
// kernel before its first unit.
constexpr int kPadRows = 64;
struct PadChunk {
    int32_t b, hv, t0, n;
    __host__ __device__ int head() const { return head_of(hv); }
    __host__ __device__ int view() const { return view_of(hv); }
};

// Where the rows of example b, head h start in the caller's tensors (in rows of d elements), and how
// far an example reaches.  Padded layout [B, H, N, d]: (b H + h) N, every example N positions long.
// Packed layout [H, T, d] (mate_plan_packed: the examples one behind the other, no padding between
// them): h T + tok_off[b], example b being len[b] positions long; positions at and beyond len[b] of
// the plan's padded view of the example do not exist in the tensors and are never written.
struct TensorRows {
    const int32_t *tok_off = nullptr;  // device [B]; null = padded layout
    const int32_t *len = nullptr;      // device [B]; null = padded layout
    int H = 0, N = 0, T = 0;
#ifdef __CUDACC__
    __device__ __forceinline__ size_t base(int b, int h) const {
        return tok_off ? (size_t)h * T + tok_off[b] : ((size_t)b * H + h) * N;
    }
    __device__ __forceinline__ bool exists(int b, int pos) const { return !len || pos < len[b]; }
#endif
};

// ---- memory pool (mate_pool.cu)
struct Block {              // device memory
    void *ptr = nullptr;
    size_t bytes = 0;
    int device = 0;
    uint64_t stream = 0;    // stream_id of the only stream that uses it (0: unknown or several)
};
struct Staging {            // host memory, pinned when `event` is set
    void *ptr = nullptr;
    size_t bytes = 0;
    int device = 0;
    cudaEvent_t event = nullptr;
};
uint64_t stream_id(cudaStream_t st);  // unique over the process's life, 0 = not to be had
bool pool_take(size_t bytes, cudaStream_t st, int device, Block *out);
void pool_give(Block &b, uint64_t stream);
bool staging_take(size_t bytes, int device, Staging *out);
void staging_give(Staging &s, cudaStream_t st);

struct ViewPlan {
    int32_t *perm = nullptr;      // [B, N]   view position -> original position
    int32_t *inv_perm = nullptr;  // [B, N]
    int32_t *seg_off = nullptr;   // [B, max_id + 2]
    int32_t *seg_lo = nullptr;    // [B, N]   per view position: first key of its own segment (bucketed
                                  //          plans: of the part of it within the adjacent buckets)
    int32_t *seg_hi = nullptr;    // [B, N]   one past the last key (prefix rows: n_valid; padding: 0)
    int32_t *cursor = nullptr;    // [B, max_id + 2] scratch of the counting sort
    int32_t *ident = nullptr;     // [B]      number of leading view positions t with perm[t] = t
    int max_id = 0;
    int n_heads = 0;
};

}  // namespace mate

struct mate_plan_s {
    int B = 0, N = 0, H = 0;
    int device = 0;                      // ordinal of the device the plan's arrays live on
    std::vector<int32_t> prefix;         // |Q| per example (host copy)
    int32_t *prefix_dev = nullptr;       // [B]
    // Length of the global block per example: the positions [0, G) of a head's order that see and are
    // seen by everything.  G = |Q| except for a bucketed plan with a longer global section.  This, not
    // |Q|, is what the attention kernels and the work-lists use; |Q| only decides the order.
    std::vector<int32_t> global;
    int32_t *global_dev = nullptr;       // [B]
    int radius = 0;                      // > 0: bucketed pattern (Section 3.1), buckets of this many positions
    int bounds_mode = 0, group = 1;      // key range of a table row (kBounds*), ids per group
    // row-or-column pattern (mate_plan_sat): this plan is the row pass; sub[0] / sub[1] are the passes
    // over the rest of the token's column in front of / behind its own cell.  The work-lists of all three are in
    // this plan's, so that the tensor-core kernels do them in one launch.
    mate_plan_s *sub[2] = {nullptr, nullptr};
    int32_t *pair_ids_dev = nullptr;     // ids of the sub-plans (in extra_block)
    // packed layout (mate_plan_packed): start and length of every example on the common token axis
    int T = 0;                           // total tokens; 0 = padded layout
    int32_t *tok_off_dev = nullptr, *len_dev = nullptr;  // [B] each (in extra_block)
    mate::TensorRows rows() const {
        mate::TensorRows r;
        r.tok_off = tok_off_dev;
        r.len = len_dev;
        r.H = H;
        r.N = N;
        r.T = T;
        return r;
    }
    size_t n_rows() const { return T ? (size_t)H * T : (size_t)B * H * N; }  // rows of a [.., d] tensor
    std::vector<uint8_t> head_view;      // host copy
    uint8_t *head_view_dev = nullptr;    // [H]
    mate::ViewPlan view[2];
    int32_t *n_valid_dev = nullptr;      // [B]
    std::vector<int32_t> n_valid;        // host copy
    std::vector<int64_t> pairs;          // [B, 2] unmasked pairs per example and view
    int32_t *status_dev = nullptr;       // device status word(s): [0] = id validation, [1] = kernel timeouts
    // device memory behind the arrays above / the work-lists below / pair_ids_dev, tok_off_dev and len_dev
    mate::Block dev_block, work_block, extra_block;
    // The stream the plan was made on, and whether it has been used on another one (or in a graph) since.  The
    // work-lists are still on their way when mate_plan returns: uses on the same stream are ordered behind the
    // copy, the first use elsewhere waits for it.
    uint64_t stream = 0;
    mutable std::atomic<bool> elsewhere{false};
    mutable std::mutex ready_mu;
    mutable cudaEvent_t ready = nullptr;  // recorded behind the copy; null once it has been waited for
    // tensor-core forward work-list, longest first; the CTAs of the persistent kernel take units through a counter
    mate::FwdUnit *fwd_units_dev = nullptr;
    mate::PadChunk *pads_dev = nullptr;
    // [kSchedWords + 8 * n_fwd_slots]: [0] next unit, then the arrival counters of the split units.
    // Zero between launches (the kernel resets what it counted), which is why two forward calls on one
    // plan must not overlap on the GPU.
    int32_t *fwd_counters_dev = nullptr;
    int n_fwd_units = 0;
    int n_pads = 0;
    int fwd_grid = 0;                     // CTAs of a forward launch
    int n_fwd_slots = 0;                  // split units
    int n_ctas = 0;                       // CTAs of the persistent kernel (SMs of the plan's device)
    size_t fwd_ws_bytes = 0;              // partial results of the split units
    std::vector<mate::FwdUnit> fwd_units; // host copies
    std::vector<mate::PadChunk> pads;
    // tensor-core backward work-list: single halves by decreasing cost; every one is done once per side
    mate::FwdUnit *bwd_units_dev = nullptr;
    int n_bwd_units = 0;
    int bwd_grid = 0;                     // CTAs of a backward launch
    std::vector<mate::FwdUnit> bwd_units;
    std::vector<int64_t> fwd_costs, bwd_costs;  // estimated clocks of the units, until the lists of three passes are joined
    const mate::ViewPlan &work_view(int v) const { return v < 2 || !sub[0] ? view[v & 1] : sub[v - 2]->view[1]; }
};

namespace mate {

// Raises a kernel's dynamic shared-memory limit once per device.  cudaFuncSetAttribute acts on the
// device that is current when it is called, so the "already done" flags are kept per device ordinal
// (under a mutex: host threads may drive different devices at the same time).
struct SmemAttrOnce {
    static constexpr int kMaxDevices = 64;
    std::mutex mu;
    bool done[kMaxDevices] = {};
    // returns MATE_OK or MATE_ERR_CUDA; `device` is the current device
    int ensure(const void *kernel, int bytes, int device) {
        std::lock_guard<std::mutex> lock(mu);
        if (device >= 0 && device < kMaxDevices && done[device]) return MATE_OK;
        if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess)
            return MATE_ERR_CUDA;
        if (device >= 0 && device < kMaxDevices) done[device] = true;
        return MATE_OK;
    }
};

// Launches a kernel that may start while the one in front of it in the stream drains: all kernels that are launched so
// wait for the one before (griddepcontrol.wait) before they read or write anything that another kernel writes or reads, and
// all but those of mate_simt.cu let the next one start early (griddepcontrol.launch_dependents; the fp32 forward takes 48.7 us
// instead of 36.8 in an earlier form, where blocks of the next kernel pile up on the SMs that finish first).  Takes the launch gap (about 2 us)
// and the set-up of the tensor-core kernels out of a layer's time.
template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream, A &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// To be called before work that uses the plan is put on `st`.
cudaError_t use_plan(const mate_plan_t *plan, cudaStream_t st);

// plan kernels (mate_plan_kernels.cu)
cudaError_t launch_plan_kernels(const int32_t *row_ids, const int32_t *col_ids, int B, int N,
                                const int32_t *prefix /* device [B] */, const int32_t *global_len /* device [B] */,
                                int radius, int bounds_mode, int group,
                                const ViewPlan &rowv, const ViewPlan &colv, int32_t *n_valid, int32_t *status,
                                cudaStream_t stream);
cudaError_t launch_unpack_ids(const int32_t *row_ids, const int32_t *col_ids, int B, int N, const int32_t *tok_off,
                              const int32_t *len, int32_t *rows_out, int32_t *cols_out, cudaStream_t stream);
cudaError_t launch_pair_ids(const int32_t *row_ids, const int32_t *col_ids, int B, int N, const int32_t *prefix,
                            int n_row_ids, int32_t *out, cudaStream_t stream);

// row-or-column pattern (mate_sat.cu): merge of the passes' outputs, sum of their gradients
cudaError_t launch_merge_passes(void *O, float *LSE, const void *O1, const float *LSE1, const void *O2, const float *LSE2,
                                size_t rows, int d, int dtype, cudaStream_t stream);
cudaError_t launch_add3(void *const (&a)[3], void *const (&b)[3], void *const (&c)[3], size_t n, int dtype, cudaStream_t stream);

// SIMT kernels (mate_simt.cu)
int simt_fwd(const mate_plan_t *plan, const void *Q, const void *K, const void *V, int d, int dtype,
             float scale, void *O, float *LSE, unsigned flags, cudaStream_t stream);
size_t simt_bwd_workspace(const mate_plan_t *plan);
int simt_bwd(const mate_plan_t *plan, const void *Q, const void *K, const void *V, const void *O,
             const float *LSE, const void *dO, int d, int dtype, float scale, void *dQ, void *dK,
             void *dV, void *workspace, int pass, cudaStream_t stream);

// tensor-core kernels (mate_fwd_tc.cu / mate_bwd_tc.cu)
bool tc_supported(int d, int dtype);
size_t tc_fwd_workspace(const mate_plan_t *plan, int d);
size_t tc_bwd_workspace(const mate_plan_t *plan);
// (outputs: one set per pass; an ordinary plan has one)
int tc_bwd(const mate_plan_t *plan, const void *Q, const void *K, const void *V, const void *O,
           const float *LSE, const void *dO, float scale, void *const (&dQ)[kPasses], void *const (&dK)[kPasses],
           void *const (&dV)[kPasses], void *workspace, cudaStream_t stream);
int tc_fwd(const mate_plan_t *plan, const void *Q, const void *K, const void *V, float scale, void *const (&O)[kPasses],
           float *const (&LSE)[kPasses], void *workspace, unsigned flags, cudaStream_t stream);

}  // namespace mate

// Optional cycle counters (compile with -DMATE_TRACE): clock64() time spent in marked regions of
// the tensor-core kernels, per CTA and role, in a local array `tr`.  Profiling aid only; compiled
// out of the library.
#ifdef MATE_TRACE
#define TR_T0(var) const long long var = clock64()
#define TR_ADD(cat, var) tr[cat] += clock64() - (var)
#define TR_INC(cat) tr[cat] += 1
#else
#define TR_T0(var)
#define TR_ADD(cat, var)
#define TR_INC(cat)
#endif
