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

// Two-pass split of P partitions of S sub-buckets each: P * S1 pass-1 buckets
// of F2 sub-buckets.  S1 is fan / P (at least 1), raised where F2 would pass
// max_f2: cutting F2 instead leaves fewer buckets than the build side needs.
// At most max_buckets in all: larger inputs get sub-buckets of several tables.
// At 65 partitions, 1.4e8 x 1.4e8 rows of 4 + 4 bytes, S1 = 1 and F2 cut to 512
// left a mean of 4207 build rows a bucket, over one 4096-row table: merge 7.17
// ms; with S1 = 2 it is 5.25 (the join 2.99 -> 1.30).  The count at 72: 22.8
// -> 7.4 ms (1.5e8 rows).
struct TwoPassSplit {
  uint32_t S1, F2;
};
inline constexpr TwoPassSplit two_pass_split(uint32_t P, uint64_t S, uint32_t fan, uint32_t max_buckets,
                                             uint32_t max_f2) {
  const uint64_t most = max_buckets / P, used = S < most ? S : most;
  uint64_t S1 = fan / P, least = (used + max_f2 - 1) / max_f2;
  if (S1 < least) S1 = least;
  if (S1 < 1) S1 = 1;
  uint64_t F2 = (S + S1 - 1) / S1;
  if (F2 > max_buckets / (P * S1)) F2 = max_buckets / (P * S1);
  if (F2 > max_f2) F2 = max_f2;
  if (F2 < 1) F2 = 1;
  return {(uint32_t)S1, (uint32_t)F2};
}

// Side A's share of `full` blocks that two sides of ca and cb equal chunks
// split: the whole number that lets the longer side end first.  Rounding down
// alone left a small side's one block half as many chunks again as the others
// (1e6 + 1e8 8-byte keys counted by 152 blocks: 0.186 ms, with it 0.131).
inline constexpr uint32_t side_blocks(uint64_t full, uint64_t ca, uint64_t cb) {
  if (ca == 0 || cb == 0) return (uint32_t)(cb == 0 ? full : 0);
  uint64_t a = full * ca / (ca + cb), best = 0, time = 0;
  for (uint64_t x = a; x <= a + 1; x++) {
    const uint64_t n = x < 1 ? 1 : x > full - 1 ? full - 1 : x;
    const uint64_t ta = (ca + n - 1) / n, tb = (cb + full - n - 1) / (full - n), t = ta > tb ? ta : tb;
    if (best == 0 || t < time) best = n, time = t;
  }
  return (uint32_t)best;
}

}  // namespace mdj
