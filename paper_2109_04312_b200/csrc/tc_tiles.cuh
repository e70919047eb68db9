// What the tensor-core forward and backward share: tiles of 128 rows of 64 bf16 in shared memory (128-byte
// swizzle), gathered by view-order position or fetched whole by a bulk tensor copy.
#pragma once
#include <cuda.h>

#include "mate_internal.h"
#include "sm100_ptx.cuh"

namespace mate {

constexpr int kRowBytes = 128;                 // 64 bf16
constexpr int kTileBytes = kTile * kRowBytes;  // 16 KB: 128 rows

// Tensor map over a [rows, 64] bf16 matrix in boxes of 128 rows (false: no tensor maps to be had).
bool make_row_map(CUtensorMap *map, const void *base, size_t rows);

// The loaders copy a tile of up to 128 rows (128 B each), warp w of the four the rows 32 w .. 32 w + 31.
// A lane looks up the original position of one row (coalesced, one latency for the whole tile, and cheap
// enough to be done a tile ahead); the copies then run four rows at a time, eight lanes per row, with the
// positions handed around by shuffle.  Rows behind the last one repeat it.
__device__ __forceinline__ int fetch_idx(const int32_t *perm, const TileInfo &t, int lw, int lane) {
    const int at = t.pos(min(32 * lw + lane, t.w - 1));
    return perm ? __ldg(perm + at) : at;  // no order given: the tensors are in view order
}
// n rows from view position q0 on, as a tile
__device__ __forceinline__ TileInfo row_tile(int q0, int n) {
    TileInfo t;
    t.x0 = t.k0 = q0;
    t.w = t.pre = n;
    t.is_b = false;
    return t;
}
// Whether a tile comes in by bulk copies: one run of positions whose rows lie in place in the tensors (`ident`: how
// many leading positions of the order do).  The box has 128 rows whatever the tile's width and the MMAs read
// whole groups of 16 rows, so a tile that ends inside a group is gathered: behind its last row the box holds
// padding or another example's tokens, whose values must not take part (the weight 0 of a masked column does not
// undo a NaN or an Inf), while a gather repeats a row of the tile.  Against bulk copies of every such tile, forward
// and backward, with earlier kernels: 8 x 512 tokens 47.8 -> 48.3 us, 4 x 2048 104.4 -> 103.8, 1 x 8192 177.3 -> 177.9.
__device__ __forceinline__ bool bulk_tile(const TileInfo &t, int ident) {
    return (t.w & 15) == 0 && t.contiguous() && t.first() + kTile <= ident;
}
// Rows [0, n_rows) of one tensor, or of two (`pair`; b_off: bytes from the first one's rows to the second's)
// -> tiles at s_a and 16 KB behind it, 128-byte swizzle.  (Four rows to a tensor copy, by two teams of two warps that took the
// loads in turn, kept a warp busy for 3700 to 4400 clk per load; these take 1000.)
__device__ __forceinline__ void gather_rows(uint32_t s_a, const uint8_t *a_bh, bool pair, int64_t b_off, uint32_t idx, int n_rows,
                                            int lw, int lane) {
    if (32 * lw >= n_rows) return;  // (rows past n_rows inside a group of 32 repeat a row that exists)
    const int sub = lane >> 3;      // row of the group of four
    a_bh += (lane & 7) * 16;
    const uint32_t d = s_a + (32 * lw + sub) * kRowBytes + (((lane & 7) ^ sub) << 4);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const uint8_t *src = a_bh + (size_t)__shfl_sync(0xffffffffu, idx, 4 * i + sub) * kRowBytes;
        const uint32_t dst = (d ^ ((i & 1) << 6)) + 4 * i * kRowBytes;
        ptx::cp_async16(dst, src);
        if (pair) ptx::cp_async16(dst + kTileBytes, src + b_off);
    }
}

}  // namespace mate
