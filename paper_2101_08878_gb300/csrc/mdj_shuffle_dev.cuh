// Device code of the scatter and shuffle passes: the column set of a pass, the
// direct (unstaged) path of a tile, a shuffle tile's shared-memory layout, its
// asynchronous loads and the write-out of one column.
#pragma once

#include <string.h>

#include <algorithm>

#include "mdj_internal.cuh"

namespace mdj {
namespace {

constexpr int kNW = 16;                     // warps per scatter block
constexpr int kRPL = 8;                     // rows per lane per tile
constexpr uint32_t kTile = kNW * 32 * kRPL; // 4096 rows per tile

struct ColMove {
  const void *src[MDJ_MAX_COLS];
  void *dst[MDJ_MAX_COLS];
  int32_t width[MDJ_MAX_COLS];
  int32_t n;
  int32_t key_index;
};

// Direct path of a pass-2 tile whose rows span too many buckets for shared
// memory (tiny or very skewed pass-1 buckets): warp-aggregated reservation,
// each row written straight to its slot.  One row per lane: key k and row id
// rid of input row r (all lanes call it).
template <typename KeyT>
__device__ __forceinline__ void place_direct(KeyT k, bool valid, size_t r, uint32_t rid, const BucketSpec &bs,
                                             uint32_t *__restrict__ cursors, const ColMove &cm,
                                             uint32_t *__restrict__ rid_out) {
  const int lane = threadIdx.x & 31;
  const uint32_t fb = valid ? sub_bucket_of(fmix64(key_bits(k)), bs) : 0xFFFFFFFFu;
  const uint32_t peers = __match_any_sync(0xffffffffu, fb);
  const int leader = __ffs(peers) - 1;
  uint32_t base = 0;
  if (valid && lane == leader) base = atomicAdd(&cursors[fb], (uint32_t)__popc(peers));
  base = __shfl_sync(0xffffffffu, base, leader);
  if (!valid) return;
  const uint32_t pos = base + __popc(peers & lanemask_lt());
  for (int j = 0; j < cm.n; j++) {
    if (cm.width[j] == 8)
      ((uint64_t *)cm.dst[j])[pos] = j == cm.key_index ? (uint64_t)k : ((const uint64_t *)cm.src[j])[r];
    else
      ((uint32_t *)cm.dst[j])[pos] = j == cm.key_index ? (uint32_t)k : ((const uint32_t *)cm.src[j])[r];
  }
  if (rid_out) rid_out[pos] = rid;
}

// The stable passes' tiles: keys in registers, row ids in global memory.
template <typename KeyT>
__device__ void scatter_direct(const KeyT (&kv)[kRPL], uint32_t wrow0, uint32_t rend, const BucketSpec &bs,
                               uint32_t *__restrict__ cursors, const ColMove &cm,
                               const uint32_t *__restrict__ rid_in, uint32_t *__restrict__ rid_out) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int c = 0; c < kRPL; c++) {
    const uint32_t r = wrow0 + c * 32 + lane;
    const bool valid = r < rend;
    place_direct<KeyT>(kv[c], valid, r, valid && rid_in ? rid_in[r] : r, bs, cursors, cm, rid_out);
  }
}

// ---------------------------------------------------------------- k_shuffle
//
// Two blocks of kShNT threads per SM, each with a tile of as many rows as its
// half of the shared memory holds (of an 8-byte key and payload about 5,700 in
// pass 1, and 4,580 in pass 2 with row ids and 452 local buckets):
//   key  [tile]   the key column
//   pay  [tile]   the first non-key column (every further one in turn)
//   rid  [tile]   pass 2: row ids (none where rows carry a term)
//   perm [tile]   bucket-ordered position -> local bucket << 16 | row in tile
//   cnt, lst, gdelta [span]  per local bucket: rank counter, local start,
//                 destination - position (modulo 2^32)
//   wsum [32]     warp sums of the count scan
// Row data stays in input order, brought in by 16-byte asynchronous copies,
// so no tile data waits in registers, and only the 4-byte perm entry is
// scattered in shared memory.
//
// What bounds it: DRAM, while the runs a tile writes are long (a run is about
// tile / buckets rows; its two ends are partial 32-byte sectors).  Measured
// per 1e8 rows of 8 + 8 + 4 bytes: runs of 44 rows 0.62 ms (5.8 TB/s), of 36
// 0.65, of 28 0.71, of 19 0.80.  So the tile is as large as two blocks per SM
// allow, and the blocks' load, rank and write-out phases overlap each other.
// Before (one 1024-thread block per SM, rows held in registers and staged as
// 16-byte records): 0.83 ms in pass 1 and 0.95 ms in pass 2, now 0.62 and
// 0.77 (1e8 rows, 28.7K sub-buckets).  Three blocks of 448 threads with
// smaller tiles: 0.71 and 0.84; 640 or 768 threads: 0.62 and 0.82.
constexpr int kShNT = 512;
constexpr int kShPairs = 6;                               // row pairs per thread per tile at most
constexpr int kShBlocks = 2;                              // blocks per SM
constexpr uint32_t kShMaxTile = (uint32_t)kShNT * kShPairs * 2;
constexpr uint32_t kShSmem = 228u * 1024 / kShBlocks - 1024;  // shared memory of a block
constexpr int kShScan = (1024 + kShNT - 1) / kShNT;       // local buckets a thread scans at most
// The wide block: one per SM, with all of its shared memory (a tile of 11,000
// rows of an 8-byte key and payload).  Nothing overlaps its phases, but into
// many buckets its runs are twice as long.
constexpr int kShWideNT = 1024;
constexpr uint32_t kShWideMaxTile = (uint32_t)kShWideNT * kShPairs * 2;
constexpr uint32_t kShWideSmem = 228u * 1024 - 1024;
static_assert(kShWideMaxTile <= 65536, "perm keeps the row in tile in 16 bits");

// SH_TERM: pass 1 whose rows leave as (key, checksum term) without row ids.
enum { SH_PASS1 = 0, SH_PASS2 = 1, SH_SEG = 2, SH_TERM = 3 };
enum { TERM_F = 1, TERM_G = 2 };  // the left and the right side's term (term_f, term_g)

// Shared memory of a block for tiles of `tile` rows (a multiple of 16) and
// `span` local buckets.
struct ShLayout {
  uint32_t pay, rid, perm, cnt, total;
  __host__ __device__ ShLayout(uint32_t tile, uint32_t key_width, uint32_t pay_width, bool with_rid, uint32_t span) {
    pay = tile * key_width;
    rid = pay + tile * pay_width;
    perm = rid + (with_rid ? tile * 4 : 0u);
    cnt = perm + tile * 4;
    total = cnt + (3 * span + 32) * 4;
  }
};

// Rows of the largest tile that fits a block's shared memory.
inline uint32_t shuffle_tile_rows(uint32_t key_width, uint32_t pay_width, bool with_rid, uint32_t span,
                                  bool wide = false) {
  const uint32_t row = key_width + pay_width + (with_rid ? 4u : 0u) + 4u;
  const uint32_t rows = ((wide ? kShWideSmem : kShSmem) - (3 * span + 32) * 4) / row / 16 * 16;
  return std::min(rows, wide ? kShWideMaxTile : kShMaxTile);
}

template <int W>
__device__ __forceinline__ void cp_async(void *dst, const void *src) {
  if (W == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(dst)),
                 "l"(__cvta_generic_to_global(src))
                 : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_addr(dst)),
                 "l"(__cvta_generic_to_global(src)), "n"(W)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// `rows` elements of W bytes from src to the 16-byte-aligned dst; returns the
// first element's place.  16-byte copies where src is 16-byte aligned, else
// one copy per element.  SHIFT: 16-byte copies from any element-aligned src;
// dst (with 16 bytes of slack) takes them at src's offset within a 16-byte line.
template <int W, bool SHIFT = false, int NT = kShNT>
__device__ __forceinline__ unsigned char *load_column(unsigned char *dst, const unsigned char *src, uint32_t rows) {
  uint32_t done = 0;
  if (SHIFT) {
    const uint32_t sh = (uint32_t)((uintptr_t)src & 15), head = min(rows, ((16 - sh) & 15) / W);
    dst += sh;
    const uint32_t n16 = (rows - head) * W / 16;
    for (uint32_t c = threadIdx.x; c < n16; c += NT)
      cp_async<16>(dst + head * W + c * 16, src + head * W + (size_t)c * 16);
    if (threadIdx.x < head) cp_async<W>(dst + threadIdx.x * W, src + threadIdx.x * W);
    done = head + n16 * (16 / W);
  } else if (((uintptr_t)src & 15) == 0) {
    const uint32_t n16 = rows * W / 16;
    for (uint32_t c = threadIdx.x; c < n16; c += NT) cp_async<16>(dst + c * 16, src + (size_t)c * 16);
    done = n16 * (16 / W);
  }
  for (uint32_t i = done + threadIdx.x; i < rows; i += NT) cp_async<W>(dst + i * W, src + (size_t)i * W);
  return dst;
}

template <bool SHIFT = false, int NT = kShNT>
__device__ __forceinline__ unsigned char *load_payload(unsigned char *dst, const void *col, int width, uint32_t row0,
                                                       uint32_t rows) {
  if (width == 8) return load_column<8, SHIFT, NT>(dst, (const unsigned char *)col + (size_t)row0 * 8, rows);
  if (width == 4) return load_column<4, SHIFT, NT>(dst, (const unsigned char *)col + (size_t)row0 * 4, rows);
  return dst;
}

// Keys of the row pairs this thread ranks: rows 2q, 2q + 1 of the tile, q =
// threadIdx.x + k * NT, so that a thread reads only keys it copied itself
// (visible after its own wait, no barrier).
template <typename KeyT, int NT>
__device__ __forceinline__ void load_key_pairs(KeyT *skey, const KeyT *keys, uint32_t rows) {
  constexpr int W2 = 2 * (int)sizeof(KeyT);
  const bool al = ((uintptr_t)keys & (W2 - 1)) == 0;
#pragma unroll
  for (int k = 0; k < kShPairs; k++) {
    const uint32_t r = 2 * (threadIdx.x + k * NT);
    if (al && r + 1 < rows) {
      cp_async<W2>(skey + r, keys + r);
    } else {
      if (r < rows) cp_async<(int)sizeof(KeyT)>(skey + r, keys + r);
      if (r + 1 < rows) cp_async<(int)sizeof(KeyT)>(skey + r + 1, keys + r + 1);
    }
  }
}

// The shuffle's tiles: key and row id come from the staged tile.
template <typename KeyT, int NT>
__device__ __noinline__ void shuffle_direct(const KeyT *skey, const uint32_t *srid, uint32_t row0, uint32_t rows,
                                            const BucketSpec &bs, uint32_t *__restrict__ cursors, const ColMove &cm,
                                            uint32_t *__restrict__ rid_out) {
  const int lane = threadIdx.x & 31;
  for (uint32_t i0 = threadIdx.x & ~31u; i0 < rows; i0 += NT) {
    const uint32_t i = i0 + lane;
    const bool valid = i < rows;
    place_direct<KeyT>(valid ? skey[i] : KeyT(0), valid, (size_t)row0 + i, valid && rid_out ? srid[i] : 0u, bs, cursors,
                       cm, rid_out);
  }
}

// One column of the staged tile to its destinations: consecutive threads
// store consecutive rows of one run.
template <typename V, int NT = kShNT>
__device__ __forceinline__ void write_column(V *__restrict__ dst, const V *stage, const uint32_t *perm,
                                             const uint32_t *gdelta, uint32_t rows) {
#pragma unroll 4
  for (uint32_t p = threadIdx.x; p < rows; p += NT) {
    const uint32_t m = perm[p];
    dst[p + gdelta[m >> 16]] = stage[m & 0xFFFFu];
  }
}

}  // namespace
}  // namespace mdj
