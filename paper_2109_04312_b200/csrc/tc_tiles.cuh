// What the tensor-core forward and backward share: tiles of 128 rows of 64 bf16 in shared memory (128-byte
// swizzle), gathered by view-order position or fetched whole by a bulk tensor copy.
#pragma once
#include <cuda.h>

#include "mate_internal.h"
#include "sm100_ptx.cuh"

namespace mate {

constexpr int kRowBytes = 128;                 // 64 bf16
constexpr int kTileBytes = kTile * kRowBytes;  // 16 KB: 128 rows

// Tensor map over a [rows, 64] bf16 matrix in boxes of box_rows rows (false: no tensor maps to be had).
bool make_row_map(CUtensorMap *map, const void *base, size_t rows, int box_rows = kTile);

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
// and backward: 8 x 512 tokens 47.8 -> 48.3 us, 4 x 2048 104.4 -> 103.8, 1 x 8192 177.3 -> 177.9.
__device__ __forceinline__ bool bulk_tile(const TileInfo &t, int ident) {
    return (t.w & 15) == 0 && t.contiguous() && t.first() + kTile <= ident;
}
// Tile rows r0 .. r0 + n_rows - 1 (at most 64; up to a multiple of four) of two tensors, by index: -> tiles at s_a and 16 KB
// behind it, 128-byte swizzle, four rows per copy.  idx: the tensors' rows for tile rows r0 + lane and r0 + 32 + lane.  The
// whole warp takes part, its leader issues; the copies count on `bar` (gather_bytes per tensor).
__device__ __forceinline__ uint32_t gather_bytes(int n_rows) { return (uint32_t)((n_rows + 3) >> 2) * 4 * kRowBytes; }
template <int kUnroll>
__device__ __forceinline__ void gather_rows4(uint32_t s_a, const CUtensorMap *map_a, const CUtensorMap *map_b, const int (&idx)[2], int r0,
                                             int n_rows, bool leader, uint32_t bar) {
    s_a += r0 * kRowBytes;
#pragma unroll kUnroll
    for (int g = 0; 4 * g < n_rows; ++g, s_a += 4 * kRowBytes) {
        const int v = g < 8 ? idx[0] : idx[1], l = 4 * (g & 7);
        const int y0 = __shfl_sync(0xffffffffu, v, l), y1 = __shfl_sync(0xffffffffu, v, l + 1), y2 = __shfl_sync(0xffffffffu, v, l + 2),
                  y3 = __shfl_sync(0xffffffffu, v, l + 3);
        if (leader) {
            ptx::tma_gather4(s_a, map_a, y0, y1, y2, y3, bar);
            if (map_b) ptx::tma_gather4(s_a + kTileBytes, map_b, y0, y1, y2, y3, bar);
        }
    }
}

}  // namespace mate
