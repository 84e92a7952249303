// Size gates and row arithmetic of the library that a CPU test can check on its
// own (plain C++, no CUDA headers).
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define MDJ_HD __host__ __device__ __forceinline__
#else
#define MDJ_HD inline
#endif

namespace mdj {

// Tiles (or chunks, or blocks) of `tile` rows that n rows take.  In 64 bits: n
// + tile - 1 passes 2^32 for the last sizes of a table (nrows < 2^32), and the
// quotient would be 0.
MDJ_HD constexpr uint32_t tile_count(uint64_t n, uint32_t tile) { return (uint32_t)((n + tile - 1) / tile); }

// Tile t of n < 2^32 rows in tiles of `tile` rows: its first row and its rows.
// Kernels step over a tile with row numbers relative to row0: an absolute
// 32-bit row number wraps when a step passes 2^32, and a loop bounded by the
// tile's end then starts again at row 0 and never leaves.
struct TileRows {
  uint32_t row0, rows;
};
MDJ_HD constexpr TileRows tile_rows(uint32_t n, uint32_t tile, uint32_t t) {
  return {t * tile, n - t * tile < tile ? n - t * tile : tile};
}

// Output positions of a compaction over m candidate rows come from an
// exclusive scan of m + 1 keep flags; its last entry (the kept total) must
// fit the position type, so 32-bit positions serve only while m + 1 <= 2^32 - 1.
inline constexpr bool compaction_needs_u64_positions(uint64_t m) { return m + 1 > 0xFFFFFFFFull; }

// Chunks of `chunk` rows that n < 2^32 rows take, in 32 bits (device code).
MDJ_HD constexpr uint32_t chunk_count(uint32_t n, uint32_t chunk) { return n ? (n - 1) / chunk + 1 : 0u; }

// Elements [beg, beg + n) of a column of `es`-byte elements whose base is
// 16-byte aligned: the 16-byte-aligned interior [a, b) goes by one bulk copy,
// the head [beg, a) and tail [b, beg + n) by ordinary loads.  In shared
// memory element beg + i sits at index sh + i of the staging buffer, sh =
// beg mod (16 / es), so the interior starts on a 16-byte boundary.  beg rounded
// up may be 2^32, which wraps to 0: there is no interior then.
struct BulkPart {
  uint32_t sh, a, b;
};
MDJ_HD constexpr BulkPart bulk_part(uint32_t beg, uint32_t n, uint32_t es) {
  const uint32_t per = 16 / es, a = (beg + per - 1) / per * per, b = (beg + n) / per * per;
  if (a < beg || b <= a) return {beg % per, beg + n, beg + n};  // no aligned interior: all by ordinary loads
  return {beg % per, a, b};
}

}  // namespace mdj
