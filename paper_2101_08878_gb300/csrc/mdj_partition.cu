// The shuffle: hash partitioning of a table on the device.
//
// In the paper the shuffle moves partition p of every worker's table to worker
// p over MPI (Sec. IV-B, the Isend/Irecv coroutines; Sec. V-B "Shuffle: True").
// On one GPU that exchange is a scatter: partition p's region of the output
// plays worker p's receive buffer.  Kernels:
//
//   k_hist       per-tile bucket histogram (shared counters); optionally also
//                the per-sub-bucket totals of a two-level plan
//   (scan)       exclusive scan of the bucket-major (bucket, tile) histogram
//                matrix = the global base of every (bucket, tile) run
//   k_partition  stable local counting sort of a tile in shared memory; the
//                columns leave as coalesced runs (one per bucket)
//   k_scatter    the same for many buckets, in smaller tiles; RESERVE variant
//                (pass 2 of the stable two-level plans): rows already grouped
//                by pass-1 bucket are split further; each tile reserves its
//                runs with one atomicAdd per (tile, bucket)
//
// Memory kernels: no tensor cores, integer hashing only.  What bounds a scatter
// is the length of the runs it writes (see k_shuffle's comments): DRAM for few
// buckets, partial sectors and the shared-memory pipe for many.
#include <stdlib.h>
#include <string.h>

#include <algorithm>

#include "mdj_internal.cuh"
#include "mdj_shuffle_dev.cuh"
#include "mdj_sizes.h"

namespace mdj {
namespace {

constexpr int kHistThreads = 512;


__host__ __device__ constexpr size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

size_t scatter_smem_bytes(uint32_t FL) {
  return (size_t)kTile * 8 + (size_t)kTile * 4 + align16((size_t)kNW * FL * 2) + (size_t)FL * 8 + 40 * 4;
}

constexpr int kHistU = 8;  // keys per thread in flight

// ------------------------------------------------------------------ k_hist
//
// hist[b * ntiles + t] = rows of bucket b in tile t.  With few buckets the
// lanes of a warp would add to the same few counters, so each counter has
// `copies` (a power of two) neighbouring copies, one per group of lanes.
// TWO: also the rows of every sub-bucket (total2), one copy of each counter.
// BLOCKS: blocks per SM, as many as the counters leave room for.  Where they
// leave room for one, the keys in flight have to come from more registers: 1e8
// + 1e8 8-byte keys in 28.9K sub-buckets 0.642 ms with 32, 0.588 with 80; 5e7 in
// 14.4K 0.228 with 32, 0.209 with 64; but 3e7 in 8.6K 0.122 with 32, 0.138 with 64.
template <typename KeyT, bool TWO, int BLOCKS>
__global__ void __launch_bounds__(kHistThreads, BLOCKS)
    k_hist(const KeyT *__restrict__ keys, uint32_t n, BucketSpec bs, uint32_t F, uint32_t copies, uint32_t tile,
           uint32_t ntiles, uint32_t *__restrict__ hist, uint32_t *__restrict__ total2, uint32_t nsub) {
  extern __shared__ uint32_t sh[];
  if (TWO) copies = 1;
  uint32_t *cnt = sh;
  uint32_t *cnt2 = sh + F * copies;
  const uint32_t mine = threadIdx.x & (copies - 1);
  if (TWO)
    for (uint32_t i = threadIdx.x; i < nsub; i += kHistThreads) cnt2[i] = 0;
  for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    for (uint32_t b = threadIdx.x; b < F * copies; b += kHistThreads) cnt[b] = 0;
    __syncthreads();
    const TileRows tr = tile_rows(n, tile, t);
    for (uint32_t i0 = 0; i0 < tr.rows; i0 += kHistThreads * kHistU) {
      const int left = (int)(tr.rows - i0) - (int)threadIdx.x;  // (a tile has few rows)
      const KeyT *__restrict__ k = keys + (tr.row0 + i0 + threadIdx.x);
      KeyT kv[kHistU];
#pragma unroll
      for (int u = 0; u < kHistU; u++) kv[u] = u * kHistThreads < left ? k[u * kHistThreads] : KeyT(0);
#pragma unroll
      for (int u = 0; u < kHistU; u++) {
        if (u * kHistThreads < left) {
          const uint64_t h = fmix64(key_bits(kv[u]));
          if (TWO) {
            const uint32_t p = mod_p(h, bs), x = (uint32_t)(h >> 32);
            atomicAdd(&cnt[p * bs.S1 + __umulhi(x, bs.S1)], 1u);
            atomicAdd(&cnt2[p * bs.S + __umulhi(x, bs.S)], 1u);
          } else {
            atomicAdd(&cnt[bucket_of(h, bs) * copies + mine], 1u);
          }
        }
      }
    }
    __syncthreads();
    if (!TWO && copies > 1) {  // F * copies <= kHistThreads: one copy per thread, neighbours summed
      const uint32_t i = threadIdx.x, all = F * copies;
      uint32_t v = i < all ? cnt[i] : 0u;
      for (uint32_t o = copies / 2; o > 0; o /= 2) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (i < all && mine == 0) hist[(size_t)(i / copies) * ntiles + t] = v;
    } else {
      for (uint32_t b = threadIdx.x; b < F; b += kHistThreads) hist[(size_t)b * ntiles + t] = cnt[b];
    }
    __syncthreads();
  }
  if (TWO) {
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < nsub; i += kHistThreads)
      if (cnt2[i]) atomicAdd(&total2[i], cnt2[i]);
  }
}

// Copies of each counter: as many as one block can sum with one thread each,
// for the few buckets of k_partition's passes.
constexpr uint32_t kPartitionMaxF = 64;  // see launch_partition
uint32_t hist_copies(uint32_t F) {
  uint32_t c = F <= kPartitionMaxF ? 32 : 1;
  while (c > 1 && F * c > kHistThreads) c /= 2;
  return c;
}

// --------------------------------------------------------------- k_scatter

// RESERVE (pass 2 of a two-level plan): the rows come grouped by pass-1 bucket
// and runs are reserved on cursors; else runs start at the scanned histogram
// entries and the scatter is stable.
template <typename KeyT, bool RESERVE>
__global__ void __launch_bounds__(kNW * 32, 2)
    k_scatter(const KeyT *__restrict__ keys, uint32_t n, BucketSpec bs, uint32_t F, uint32_t ntiles,
              const uint32_t *__restrict__ tile_base, uint32_t *__restrict__ cursors, uint32_t F2, ColMove cm,
              const uint32_t *__restrict__ rid_in, uint32_t *__restrict__ rid_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  const uint32_t FL = RESERVE ? kPass2SpanMax : F;
  uint64_t *stage64 = (uint64_t *)smem;
  uint32_t *stage32 = (uint32_t *)smem;
  uint32_t *dstmap = (uint32_t *)(smem + (size_t)kTile * 8);
  uint16_t *whist = (uint16_t *)(smem + (size_t)kTile * 12);
  uint32_t *lstart = (uint32_t *)(smem + (size_t)kTile * 12 + align16((size_t)kNW * FL * 2));
  uint32_t *gbase = lstart + FL;
  uint32_t *scratch = gbase + FL;

  const uint32_t t = blockIdx.x;
  const uint32_t row0 = t * kTile;
  const uint32_t rows = min(kTile, n - row0);
  const uint32_t rend = row0 + rows;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t wrow0 = row0 + warp * 32 * kRPL;

  KeyT kv[kRPL];
#pragma unroll
  for (int c = 0; c < kRPL; c++) {
    uint32_t r = wrow0 + c * 32 + lane;
    kv[c] = r < rend ? keys[r] : KeyT(0);
  }

  uint32_t Floc = F, lb0 = 0;
  if (RESERVE) {
    const uint32_t b1f = sub_bucket_of(fmix64(key_bits(keys[row0])), bs) / F2;
    const uint32_t b1l = sub_bucket_of(fmix64(key_bits(keys[rend - 1])), bs) / F2;
    lb0 = b1f * F2;
    Floc = (b1l - b1f + 1) * F2;
    if (Floc > kPass2SpanMax) {
      scatter_direct<KeyT>(kv, wrow0, rend, bs, cursors, cm, rid_in, rid_out);
      return;
    }
  }

  // 1. per-warp stable ranks: warp w owns rows [wrow0, wrow0 + 32*kRPL) and
  //    walks them in order, so (warp, rank) order is input order.
  for (uint32_t i = threadIdx.x; i < (kNW * Floc + 1) / 2; i += blockDim.x) ((uint32_t *)whist)[i] = 0;
  __syncthreads();
  uint32_t pk[kRPL];
  uint16_t *wh = whist + warp * Floc;
#pragma unroll
  for (int c = 0; c < kRPL; c++) {
    uint32_t r = wrow0 + c * 32 + lane;
    bool valid = r < rend;
    uint32_t b = 0xFFFFFFFFu;
    if (valid) b = bucket_of(fmix64(key_bits(kv[c])), bs) - lb0;
    uint32_t peers = __match_any_sync(0xffffffffu, b);
    uint32_t rank = __popc(peers & lanemask_lt());
    uint32_t old = valid ? wh[b] : 0u;
    __syncwarp();
    if (valid && rank == 0) wh[b] = (uint16_t)(old + __popc(peers));
    __syncwarp();
    pk[c] = (b << 16) | (old + rank);
  }
  __syncthreads();

  // 2. per bucket: warp offsets (exclusive over warps) and the tile count
  for (uint32_t b = threadIdx.x; b < Floc; b += blockDim.x) {
    uint32_t run = 0;
    for (int w = 0; w < kNW; w++) {
      uint32_t c = whist[w * Floc + b];
      whist[w * Floc + b] = (uint16_t)run;
      run += c;
    }
    lstart[b] = run;
  }
  __syncthreads();
  block_scan_array(lstart, Floc, scratch);

  // 3. global base of each bucket's run
  for (uint32_t b = threadIdx.x; b < Floc; b += blockDim.x) {
    if (!RESERVE) {
      gbase[b] = tile_base[(size_t)b * ntiles + t];
    } else {
      const uint32_t e = b + 1 < Floc ? lstart[b + 1] : rows;
      const uint32_t cnt = e - lstart[b];
      gbase[b] = cnt ? atomicAdd(&cursors[lb0 + b], cnt) : 0u;
    }
  }
  __syncthreads();

  // 4. sorted position of each row and its destination
  uint32_t lp[kRPL];
#pragma unroll
  for (int c = 0; c < kRPL; c++) {
    uint32_t r = wrow0 + c * 32 + lane;
    lp[c] = 0;
    if (r < rend) {
      uint32_t b = pk[c] >> 16, lr = pk[c] & 0xFFFFu;
      uint32_t wo = whist[warp * Floc + b];
      lp[c] = lstart[b] + wo + lr;
      dstmap[lp[c]] = gbase[b] + wo + lr;
    }
  }
  __syncthreads();

  // 5. every column: stage in sorted order, leave as runs
  for (int j = 0; j < cm.n; j++) {
    if (cm.width[j] == 8) {
      const uint64_t *src = (const uint64_t *)cm.src[j];
      uint64_t v[kRPL];
#pragma unroll
      for (int c = 0; c < kRPL; c++) {
        uint32_t r = wrow0 + c * 32 + lane;
        v[c] = j == cm.key_index ? (uint64_t)kv[c] : (r < rend ? src[r] : 0ull);
      }
#pragma unroll
      for (int c = 0; c < kRPL; c++)
        if (wrow0 + c * 32 + lane < rend) stage64[lp[c]] = v[c];
      __syncthreads();
      uint64_t *dst = (uint64_t *)cm.dst[j];
      for (uint32_t i = threadIdx.x; i < rows; i += blockDim.x) dst[dstmap[i]] = stage64[i];
      __syncthreads();
    } else {
      const uint32_t *src = (const uint32_t *)cm.src[j];
      uint32_t v[kRPL];
#pragma unroll
      for (int c = 0; c < kRPL; c++) {
        uint32_t r = wrow0 + c * 32 + lane;
        v[c] = j == cm.key_index ? (uint32_t)kv[c] : (r < rend ? src[r] : 0u);
      }
#pragma unroll
      for (int c = 0; c < kRPL; c++)
        if (wrow0 + c * 32 + lane < rend) stage32[lp[c]] = v[c];
      __syncthreads();
      uint32_t *dst = (uint32_t *)cm.dst[j];
      for (uint32_t i = threadIdx.x; i < rows; i += blockDim.x) dst[dstmap[i]] = stage32[i];
      __syncthreads();
    }
  }
  if (rid_out) {
    uint32_t v[kRPL];
#pragma unroll
    for (int c = 0; c < kRPL; c++) {
      uint32_t r = wrow0 + c * 32 + lane;
      v[c] = rid_in ? (r < rend ? rid_in[r] : 0u) : r;
    }
#pragma unroll
    for (int c = 0; c < kRPL; c++)
      if (wrow0 + c * 32 + lane < rend) stage32[lp[c]] = v[c];
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < rows; i += blockDim.x) rid_out[dstmap[i]] = stage32[i];
  }
}

// ------------------------------------------------------------- k_partition
//
// The stable scatter: persistent blocks, tiles staged in input order as in
// k_shuffle (key, first payload and row ids by asynchronous copies, a 4-byte
// permutation entry per row), two blocks per SM.  A row's stable rank: warp w
// owns rows [w * tile / 16, (w + 1) * tile / 16) and walks them 32 at a time
// (match_any among the 32, a shared counter per warp and bucket), then the
// counters become offsets over the warps; the run of (tile, bucket) starts at
// the scanned histogram entry.
//
// DRAM-bound for few buckets.  5e7 rows of 8 + 8 bytes, 8 buckets, with row
// ids: 0.407 -> 0.306 ms (5.9 TB/s).
constexpr int kPtGroups = (int)(kShMaxTile / kShNT);  // 32-row groups of a warp's rows at most
constexpr int kPtWarps = kShNT / 32;

// shift: columns are staged at their offset within a 16-byte line.
struct PtLayout {
  uint32_t pay, rid, perm, lst, whist, total;
  __host__ __device__ PtLayout(uint32_t tile, uint32_t key_width, uint32_t pay_width, bool with_rid, uint32_t F,
                               bool shift) {
    const uint32_t slack = shift ? 16 : 0;
    pay = tile * key_width + slack;
    rid = pay + tile * pay_width + slack;
    perm = rid + (with_rid ? tile * 4 : 0u);
    lst = perm + tile * 4;
    whist = lst + (2 * F + 32) * 4;
    total = whist + (kPtWarps * F * 2 + 15) / 16 * 16;
  }
};

// Tile rows (a multiple of kShNT): the most that leave room for two blocks per
// SM.
uint32_t partition_tile_rows(uint32_t key_width, uint32_t pay_width, bool with_rid, uint32_t F) {
  uint32_t tile = kShMaxTile;
  while (PtLayout(tile, key_width, pay_width, with_rid, F, true).total > kShSmem) tile -= kShNT;
  return tile;
}

template <typename KeyT, bool EXTRA, bool SHIFT>
__global__ void __launch_bounds__(kShNT, kShBlocks)
    k_partition(const KeyT *__restrict__ keys, uint32_t n, uint32_t tile, uint32_t ntiles, uint32_t pay_width,
                const __grid_constant__ BucketSpec bs, uint32_t F, const uint32_t *__restrict__ tile_base,
                const __grid_constant__ ColMove cm, int reg_col, const uint32_t *__restrict__ rid_in,
                uint32_t *__restrict__ rid_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  const PtLayout lay(tile, sizeof(KeyT), pay_width, rid_in != nullptr, F, SHIFT);
  unsigned char *spay = smem + lay.pay;
  uint32_t *srid = (uint32_t *)(smem + lay.rid);
  uint32_t *perm = (uint32_t *)(smem + lay.perm);
  uint32_t *lst = (uint32_t *)(smem + lay.lst);
  uint32_t *gdelta = lst + F;
  uint32_t *wsum = gdelta + F;
  uint16_t *whist = (uint16_t *)(smem + lay.whist);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint16_t *wh = whist + warp * F;
  const int pw = reg_col >= 0 ? cm.width[reg_col] : 0;
  KeyT *__restrict__ kdst = (KeyT *)cm.dst[cm.key_index];
  void *pdst = pw ? cm.dst[reg_col] : nullptr;
  const uint32_t wrows = tile / kPtWarps;  // rows of a warp, a multiple of 32

  for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const uint32_t row0 = t * tile, rows = min(tile, n - row0);
    const KeyT *skey =
        (const KeyT *)load_column<(int)sizeof(KeyT), SHIFT>(smem, (const unsigned char *)(keys + row0), rows);
    cp_async_commit();
    const unsigned char *pay = pw ? load_payload<SHIFT>(spay, cm.src[reg_col], pw, row0, rows) : spay;
    if (rid_in) load_column<4>((unsigned char *)srid, (const unsigned char *)(rid_in + row0), rows);
    cp_async_commit();
    for (uint32_t i = lane; i < F; i += 32) wh[i] = 0;
    cp_async_wait<1>();
    __syncthreads();
    // stable ranks inside the warp's rows
    uint32_t pk[kPtGroups];
#pragma unroll
    for (int c = 0; c < kPtGroups; c++) {
      pk[c] = 0xFFFFFFFFu;
      if (c * 32u < wrows) {  // uniform over the block
        const uint32_t i = warp * wrows + c * 32 + lane;
        const bool valid = i < rows;
        const uint32_t b = valid ? bucket_of(fmix64(key_bits(skey[i])), bs) : 0xFFFFFFFFu;
        const uint32_t peers = __match_any_sync(0xffffffffu, b);
        const uint32_t rank = __popc(peers & lanemask_lt());
        const uint32_t old = valid ? wh[b] : 0u;
        __syncwarp();
        if (valid && rank == 0) wh[b] = (uint16_t)(old + __popc(peers));
        __syncwarp();
        if (valid) pk[c] = (b << 16) | (old + rank);
      }
    }
    __syncthreads();
    // per bucket: offsets over the warps, the local start, the destination
    const uint32_t per = (F + kShNT - 1) / kShNT;
    const uint32_t s0 = min(F, threadIdx.x * per), s1 = min(F, s0 + per);
    uint32_t cb[kShScan], gb[kShScan], own = 0;
#pragma unroll
    for (int i = 0; i < kShScan; i++) {
      cb[i] = gb[i] = 0;
      if (s0 + i < s1) {
        gb[i] = tile_base[(size_t)(s0 + i) * ntiles + t];
#pragma unroll
        for (int w = 0; w < kPtWarps; w++) {
          const uint32_t c = whist[w * F + s0 + i];
          whist[w * F + s0 + i] = (uint16_t)cb[i];
          cb[i] += c;
        }
        own += cb[i];
      }
    }
    const uint32_t inc = warp_inclusive_scan(own);
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    uint32_t ex = inc - own;
#pragma unroll
    for (int w = 0; w < kPtWarps; w++)
      if (w < warp) ex += wsum[w];
#pragma unroll
    for (int i = 0; i < kShScan; i++)
      if (s0 + i < s1) {
        lst[s0 + i] = ex;
        gdelta[s0 + i] = gb[i] - ex;
        ex += cb[i];
      }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < kPtGroups; c++)
      if (pk[c] != 0xFFFFFFFFu) {
        const uint32_t b = pk[c] >> 16;
        perm[lst[b] + wh[b] + (pk[c] & 0xFFFFu)] = (b << 16) | (warp * wrows + c * 32 + lane);
      }
    cp_async_wait<0>();
    __syncthreads();
#pragma unroll 4
    for (uint32_t p = threadIdx.x; p < rows; p += kShNT) {
      const uint32_t m = perm[p], i = m & 0xFFFFu;
      const uint32_t d = p + gdelta[m >> 16];
      kdst[d] = skey[i];
      if (pw == 8) ((uint64_t *)pdst)[d] = ((const uint64_t *)pay)[i];
      if (pw == 4) ((uint32_t *)pdst)[d] = ((const uint32_t *)pay)[i];
      if (rid_out) rid_out[d] = rid_in ? srid[i] : row0 + i;
    }
    __syncthreads();
    if (EXTRA) {
#pragma unroll 1
      for (int j = 0; j < cm.n; j++) {
        if (j == cm.key_index || j == reg_col) continue;
        pay = load_payload<SHIFT>(spay, cm.src[j], cm.width[j], row0, rows);
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
        if (cm.width[j] == 8)
          write_column<uint64_t>((uint64_t *)cm.dst[j], (const uint64_t *)pay, perm, gdelta, rows);
        else
          write_column<uint32_t>((uint32_t *)cm.dst[j], (const uint32_t *)pay, perm, gdelta, rows);
        __syncthreads();
      }
    }
  }
}

// ------------------------------------------------- unstable shuffle (merge)
//
// The merge needs every row in its sub-bucket, not the input order inside a
// bucket, so its shuffle drops stability (the public partition keeps it):
//
//   k_tot      rows per final sub-bucket (shared counters, flushed with one
//              global add per counter); the next chunk's keys load while the
//              current chunk is counted
//   k_shuffle  persistent blocks: a row's rank in its bucket is a
//              shared-memory atomic, each (tile, bucket) run is reserved with
//              one global atomicAdd on the bucket's cursor, and the columns
//              leave in bucket order as runs.
//              Pass 2: rows already grouped by pass-1 bucket (sub-bucket / F2)
//              are split into their sub-buckets, as in k_scatter's RESERVE.
// A pass-1 bucket holds the rows of sub-buckets [b * F2, (b + 1) * F2)
// (pass-1 bucket = sub-bucket / F2, see BucketSpec), so the scanned counts
// of the final sub-buckets also place the pass-1 buckets.

constexpr int kTotThreads = 1024;
constexpr int kTotU = 8;                        // keys per thread per chunk
template <typename KeyT>
__device__ __forceinline__ void tot_load(const KeyT *__restrict__ keys, uint64_t base, uint32_t n, KeyT (&v)[kTotU]) {
#pragma unroll
  for (int u = 0; u < kTotU; u++) {
    const uint64_t r = base + (uint64_t)u * kTotThreads + threadIdx.x;
    v[u] = r < n ? keys[r] : KeyT(0);
  }
}

// One side of a count: `blocks` blocks add its rows per sub-bucket to tot.
struct TotSide {
  const void *keys;
  uint32_t *tot;
  uint32_t n, blocks;
};

// tot[sb] += rows of sub-bucket sb (spec bs, nsub = P * S), for one side or
// for both in one launch (the first A.blocks blocks take side A).
template <typename KeyT>
__global__ void __launch_bounds__(kTotThreads) k_tot(const TotSide A, const TotSide B, BucketSpec bs, uint32_t nsub) {
  extern __shared__ uint32_t cnt[];
  const bool first = blockIdx.x < A.blocks;
  const KeyT *__restrict__ keys = (const KeyT *)(first ? A.keys : B.keys);
  uint32_t *__restrict__ tot = first ? A.tot : B.tot;
  const uint32_t n = first ? A.n : B.n, nblk = first ? A.blocks : B.blocks;
  const uint32_t blk = first ? blockIdx.x : blockIdx.x - A.blocks;
  for (uint32_t i = threadIdx.x; i < nsub; i += kTotThreads) cnt[i] = 0;
  __syncthreads();
  const uint64_t chunk = (uint64_t)kTotThreads * kTotU, stride = chunk * nblk;
  uint64_t base = chunk * blk;
  KeyT cur[kTotU], nxt[kTotU];
  tot_load<KeyT>(keys, base, n, cur);
  for (; base < n; base += stride) {
    tot_load<KeyT>(keys, base + stride, n, nxt);
#pragma unroll
    for (int u = 0; u < kTotU; u++) {
      const uint64_t r = base + (uint64_t)u * kTotThreads + threadIdx.x;
      if (r < n) atomicAdd(&cnt[sub_bucket_of(fmix64(key_bits(cur[u])), bs)], 1u);
      cur[u] = nxt[u];
    }
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < nsub; i += kTotThreads)
    if (cnt[i]) atomicAdd(&tot[i], cnt[i]);
}

// Pass-1 cursors (the first row of every pass-1 bucket) and, for two-level
// plans, pass 2's: the first row of every sub-bucket (cur2 may be NULL).
__global__ void k_pass1_cursors(const uint32_t *__restrict__ off, uint32_t F1, uint32_t F2,
                                uint32_t *__restrict__ cur, uint32_t *__restrict__ cur2, uint32_t nsub) {
  const uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < F1) cur[b] = off[(size_t)b * F2];
  if (cur2 && b < nsub) cur2[b] = off[b];
}

// A batch of independent merges (joins: P = 1): a row of segment g with hash h
// goes to bucket base[g] + p * S[g] + floor(hi32(h) * S[g] / 2^32), p = h mod
// P[g]; nb[g] = P[g] * S[g] buckets.
struct SegArgs {
  const SegTile *tiles;  // never cross a segment
  const uint32_t *base, *nb, *P, *S;
};

// One table side of a shuffle pass: `ntiles` tiles of its n rows, run
// destinations reserved on `cursors`, row ids to rid_out (read from rid_in in
// pass 2, where both may be NULL, else the row's index).  `reg_col`: the first non-key column (-1:
// none).
struct ShSide {
  const void *keys;
  const uint32_t *rid_in;
  uint32_t *rid_out;
  uint32_t *cursors;
  ColMove cm;
  int32_t reg_col;
  int32_t term;         // SH_TERM: TERM_F or TERM_G, to term_dst
  uint64_t *term_dst;
  uint32_t n, ntiles;
};
struct ShSides {
  ShSide s[2];
};

// Persistent: block b takes tiles b, b + gridDim.x, ... (side 0's tiles
// first; only pass 1 has a side 1).  Per tile:
//   1. load: keys, then payload and row ids, by asynchronous copies;
//   2. rank: a row's rank in its bucket is a shared-memory atomicAdd;
//   3. counts: local starts by a block scan; each (tile, bucket) run's
//      destination from one atomicAdd on the bucket's cursor, whose result is
//      needed only at write-out;
//   4. perm: each row's number goes to its bucket-ordered position;
//   5. write-out: the columns are gathered through perm and leave as runs.
// `pay_width`: bytes of a row's place in the payload area.  EXTRA: further
// columns, one at a time through that area.  NT: threads, kShNT or kShWideNT.
template <typename KeyT, int MODE, bool EXTRA, int NT>
__global__ void __launch_bounds__(NT, kShNT * kShBlocks / NT)
    k_shuffle(const __grid_constant__ ShSides sides, uint32_t tile, uint32_t ntiles, uint32_t pay_width,
              const __grid_constant__ BucketSpec bs, uint32_t F, uint32_t F2, uint32_t span, const SegArgs sg) {
  constexpr int kScan = (1024 + NT - 1) / NT;  // local buckets a thread scans at most
  extern __shared__ __align__(16) unsigned char smem[];
  const bool with_rid = MODE == SH_PASS2 && sides.s[0].rid_in != nullptr;
  const ShLayout lay(tile, sizeof(KeyT), pay_width, with_rid, span);
  KeyT *skey = (KeyT *)smem;
  unsigned char *spay = smem + lay.pay;
  uint32_t *srid = (uint32_t *)(smem + lay.rid);
  uint32_t *perm = (uint32_t *)(smem + lay.perm);
  uint32_t *cnt = (uint32_t *)(smem + lay.cnt);
  uint32_t *lst = cnt + span;
  uint32_t *gdelta = lst + span;
  uint32_t *wsum = gdelta + span;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (uint32_t i = threadIdx.x; i < span; i += NT) cnt[i] = 0;
  __syncthreads();

  for (uint32_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
    const uint32_t second = MODE == SH_PASS1 && t >= sides.s[0].ntiles ? 1u : 0u;
    const ShSide &sd = sides.s[second];
    const ColMove &cm = sd.cm;
    const int reg_col = sd.reg_col;
    const int pw = reg_col >= 0 ? cm.width[reg_col] : 0;
    const KeyT *__restrict__ keys = (const KeyT *)sd.keys;
    uint32_t *__restrict__ cursors = sd.cursors;
    SegTile td = {0, 0, 0};
    if (MODE == SH_SEG) td = sg.tiles[t];
    const uint32_t row0 = MODE == SH_SEG ? td.row0 : (second ? t - sides.s[0].ntiles : t) * tile;
    const uint32_t rows = MODE == SH_SEG ? td.rows : min(tile, sd.n - row0);
    // 1. load
    load_key_pairs<KeyT, NT>(skey, keys + row0, rows);
    cp_async_commit();
    if (pw) load_payload<false, NT>(spay, cm.src[reg_col], pw, row0, rows);
    if (with_rid) load_column<4, false, NT>((unsigned char *)srid, (const unsigned char *)(sd.rid_in + row0), rows);
    cp_async_commit();
    uint32_t lb0 = 0, Floc = F;
    BucketSpec sp;
    if (MODE == SH_SEG) {
      lb0 = sg.base[td.seg];
      Floc = sg.nb[td.seg];
      sp = make_spec_dev(sg.P[td.seg]);
      sp.S = sg.S[td.seg];
    }
    if (MODE == SH_PASS2) {
      const uint32_t b1f = sub_bucket_of(fmix64(key_bits(keys[row0])), bs) / F2;
      const uint32_t b1l = sub_bucket_of(fmix64(key_bits(keys[row0 + rows - 1])), bs) / F2;
      lb0 = b1f * F2;
      Floc = (b1l - b1f + 1) * F2;
      if (Floc > span) {  // uniform over the block
        cp_async_wait<0>();
        __syncthreads();
        shuffle_direct<KeyT, NT>(skey, srid, row0, rows, bs, cursors, cm, sd.rid_out);
        __syncthreads();
        continue;
      }
    }
    // 2. rank
    cp_async_wait<1>();
    uint32_t pk[2 * kShPairs];
#pragma unroll
    for (int k = 0; k < kShPairs; k++) {
      const uint32_t r = 2 * (threadIdx.x + k * NT);
      KeyT kv[2] = {KeyT(0), KeyT(0)};
      if (r >= rows) {  // past the tile: nothing there to read
      } else if (sizeof(KeyT) == 8) {
        const longlong2 v = *(const longlong2 *)(skey + r);
        kv[0] = (KeyT)v.x, kv[1] = (KeyT)v.y;
      } else {
        const int2 v = *(const int2 *)(skey + r);
        kv[0] = (KeyT)v.x, kv[1] = (KeyT)v.y;
      }
#pragma unroll
      for (int e = 0; e < 2; e++) {
        pk[2 * k + e] = 0xFFFFFFFFu;
        if (r + e < rows) {
          const uint64_t h = fmix64(key_bits(kv[e]));
          const uint32_t lb = MODE == SH_PASS1 || MODE == SH_TERM ? bucket_of(h, bs)
                              : MODE == SH_PASS2               ? sub_bucket_of(h, bs) - lb0
                                                               : sub_bucket_of(h, sp);
          pk[2 * k + e] = (lb << 16) | atomicAdd(&cnt[lb], 1u);
        }
      }
    }
    __syncthreads();
    // 3. counts: this thread's buckets [s0, s1); its counters are cleared for the next tile
    const uint32_t per = (Floc + NT - 1) / NT;
    const uint32_t s0 = min(Floc, threadIdx.x * per), s1 = min(Floc, s0 + per);
    uint32_t cb[kScan], gb[kScan], own = 0;
#pragma unroll
    for (int i = 0; i < kScan; i++) {
      cb[i] = gb[i] = 0;
      if (s0 + i < s1) {
        cb[i] = cnt[s0 + i];
        cnt[s0 + i] = 0;
        if (cb[i]) gb[i] = atomicAdd(&cursors[lb0 + s0 + i], cb[i]);
        own += cb[i];
      }
    }
    const uint32_t inc = warp_inclusive_scan(own);
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    uint32_t ex = inc - own;
#pragma unroll
    for (int w = 0; w < NT / 32; w++)
      if (w < warp) ex += wsum[w];
#pragma unroll
    for (int i = 0; i < kScan; i++)
      if (s0 + i < s1) {
        lst[s0 + i] = ex;
        gb[i] -= ex;
        ex += cb[i];
      }
    __syncthreads();
    // 4. perm
#pragma unroll
    for (int k = 0; k < kShPairs; k++) {
#pragma unroll
      for (int e = 0; e < 2; e++) {
        const uint32_t q = pk[2 * k + e];
        if (q != 0xFFFFFFFFu)
          perm[lst[q >> 16] + (q & 0xFFFFu)] = (q & 0xFFFF0000u) | (2 * (threadIdx.x + k * NT) + e);
      }
    }
#pragma unroll
    for (int i = 0; i < kScan; i++)
      if (s0 + i < s1) gdelta[s0 + i] = gb[i];
    cp_async_wait<0>();
    __syncthreads();
    // 5. write-out
    KeyT *__restrict__ kdst = (KeyT *)cm.dst[cm.key_index];
    void *pdst = pw ? cm.dst[reg_col] : nullptr;
    uint32_t *__restrict__ rid_out = sd.rid_out;
#pragma unroll 4
    for (uint32_t p = threadIdx.x; p < rows; p += NT) {
      const uint32_t m = perm[p], i = m & 0xFFFFu;
      const uint32_t d = p + gdelta[m >> 16];
      kdst[d] = skey[i];
      if (MODE == SH_TERM) {
        const uint64_t pb = pay_bits(pw ? spay : nullptr, pw, i);
        sd.term_dst[d] = sd.term == TERM_F ? term_f(key_bits(skey[i]), row0 + i, pb) : term_g(row0 + i, pb);
        continue;
      }
      if (pw == 8) ((uint64_t *)pdst)[d] = ((const uint64_t *)spay)[i];
      if (pw == 4) ((uint32_t *)pdst)[d] = ((const uint32_t *)spay)[i];
      if (MODE != SH_PASS2)
        rid_out[d] = row0 + i;
      else if (with_rid)
        rid_out[d] = srid[i];
    }
    __syncthreads();
    if (EXTRA) {
#pragma unroll 1
      for (int j = 0; j < cm.n; j++) {
        if (j == cm.key_index || j == reg_col) continue;
        load_payload<false, NT>(spay, cm.src[j], cm.width[j], row0, rows);
        cp_async_commit();
        cp_async_wait<0>();
        __syncthreads();
        if (cm.width[j] == 8)
          write_column<uint64_t, NT>((uint64_t *)cm.dst[j], (const uint64_t *)spay, perm, gdelta, rows);
        else
          write_column<uint32_t, NT>((uint32_t *)cm.dst[j], (const uint32_t *)spay, perm, gdelta, rows);
        __syncthreads();
      }
    }
  }
}

// ------------------------------------------------------------ small kernels

// First row of every bucket, and n behind the last (as row numbers or as the
// caller's 64-bit offsets).
template <typename T>
__global__ void k_bucket_starts(const uint32_t *__restrict__ hist, uint32_t F, uint32_t ntiles, uint32_t n,
                                T *__restrict__ start) {
  uint32_t b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < F) start[b] = ntiles ? hist[(size_t)b * ntiles] : 0u;
  if (b == F) start[F] = n;
}

// offsets of partition p in rows already sorted by p: first row with p' >= p
template <typename KeyT>
__global__ void k_offsets_bsearch(const KeyT *__restrict__ keys, uint32_t n, BucketSpec bs, uint32_t P,
                                  uint32_t *__restrict__ off) {
  uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p > P) return;
  uint32_t lo = 0, hi = n;
  while (lo < hi) {
    uint32_t mid = lo + (hi - lo) / 2;
    if (mod_p(fmix64(key_bits(keys[mid])), bs) < p)
      lo = mid + 1;
    else
      hi = mid;
  }
  off[p] = lo;
}

__global__ void k_two(uint32_t *p, uint32_t a, uint32_t b) {
  p[0] = a;
  p[1] = b;
}

__global__ void k_u32_to_i64(const uint32_t *__restrict__ a, int64_t *__restrict__ b, uint32_t n) {
  uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) b[i] = (int64_t)a[i];
}

// ------------------------------------------------------------- host passes

// Histogram blocks per SM beside `smem` bytes of counters each.
int hist_blocks(size_t smem) { return smem <= 48 * 1024 ? 4 : smem <= 100 * 1024 ? 2 : 1; }

template <typename KeyT>
auto hist_kernel(bool two, int blocks) {
  if (!two) return k_hist<KeyT, false, 4>;
  return blocks == 4 ? k_hist<KeyT, true, 4> : blocks == 2 ? k_hist<KeyT, true, 2> : k_hist<KeyT, true, 1>;
}

template <typename KeyT>
auto partition_kernel(bool extra, bool shift) {
  if (shift) return extra ? k_partition<KeyT, true, true> : k_partition<KeyT, false, true>;
  return extra ? k_partition<KeyT, true, false> : k_partition<KeyT, false, false>;
}

template <typename KeyT>
int set_smem_attrs() {
  static PerDeviceOnce once;
  return once_per_device(once, [] {
    MDJ_CUDA_TRY(cudaFuncSetAttribute(k_scatter<KeyT, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)scatter_smem_bytes(kMaxFanout)));
    MDJ_CUDA_TRY(cudaFuncSetAttribute(k_scatter<KeyT, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)scatter_smem_bytes(kPass2SpanMax)));
    for (int extra = 0; extra < 2; extra++)
      for (int shift = 0; shift < 2; shift++)
        MDJ_CUDA_TRY(cudaFuncSetAttribute(partition_kernel<KeyT>(extra != 0, shift != 0),
                                          cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kShSmem));
    for (int blocks : {1, 2, 4})
      MDJ_CUDA_TRY(cudaFuncSetAttribute(hist_kernel<KeyT>(true, blocks), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        (int)((kMaxFanout + kMaxSubBuckets) * 4)));
    return (int)MDJ_OK;
  });
}

// kPartitionMaxF: buckets up to which a stable pass runs as k_partition, above
// as k_scatter.
// 5e7 rows, k_partition against k_scatter (whole mdj_partition call, us):
// 8 + 8 bytes: 32 buckets 499 / 568, 100 655 / 661, 256 693 / 688, 1000 1319 /
// 1009; 4 + 4 bytes: 32 434 / 493, 100 571 / 601, 256 663 / 612; three columns:
// 32 580 / 633, 100 748 / 732, 256 888 / 760.  Above, k_partition's counters
// per warp and bucket shorten its tile, and with it the runs.
uint32_t stable_tile_rows(uint32_t key_width, uint32_t pay_width, bool with_rid, uint32_t F) {
  return F > kPartitionMaxF ? kTile : partition_tile_rows(key_width, pay_width, with_rid, F);
}

// Launches of a stable pass over n > 0 rows into F <= kMaxFanout buckets with
// a given tile and histogram matrix: the histogram, then (the matrix scanned
// in between) the scatter.
template <typename KeyT>
void launch_hist(const KeyT *keys, uint32_t n, const BucketSpec &bs, uint32_t F, uint32_t tile, uint32_t ntiles,
                 uint32_t *hist, uint32_t *total2, uint32_t nsub, cudaStream_t s) {
  const uint32_t copies = total2 ? 1u : hist_copies(F);
  const size_t hsmem = (size_t)(F * copies + (total2 ? nsub : 0)) * 4;
  TraceScope tr("hist", s);
  const int blocks = hist_blocks(hsmem);
  const unsigned hgrid = std::min(ntiles, (uint32_t)(num_sms() * blocks));
  auto kernel = hist_kernel<KeyT>(total2 != nullptr, blocks);
  kernel<<<hgrid, kHistThreads, hsmem, s>>>(keys, n, bs, F, copies, tile, ntiles, hist, total2, nsub);
}

template <typename KeyT>
void launch_partition(const KeyT *keys, uint32_t n, const BucketSpec &bs, uint32_t F, uint32_t tile, uint32_t ntiles,
                      uint32_t pay_width, const uint32_t *hist, const ColMove &cm, const uint32_t *rid_in,
                      uint32_t *rid_out, cudaStream_t s) {
  TraceScope tr("scatter_stable", s);
  if (F > kPartitionMaxF) {
    k_scatter<KeyT, false><<<ntiles, kNW * 32, scatter_smem_bytes(F), s>>>(keys, n, bs, F, ntiles, hist, nullptr, 1, cm,
                                                                           rid_in, rid_out);
    return;
  }
  // Columns off 16-byte boundaries take a kernel that stages them at their own
  // offset.  5e7 rows of 8 + 8 bytes, 8 buckets, one element off: 0.430 ms copied
  // element by element, 0.323 so (aligned columns 0.308; 0.316 with this kernel).
  uintptr_t bases = 0;
  for (int j = 0; j < cm.n; j++) bases |= (uintptr_t)cm.src[j];
  const bool shift = (bases & 15) != 0;
  const uint32_t sm = PtLayout(tile, sizeof(KeyT), pay_width, rid_in != nullptr, F, shift).total;
  const uint32_t most = (uint32_t)num_sms() * kShBlocks;
  const int reg_col = cm.n < 2 ? -1 : (cm.key_index == 0 ? 1 : 0);
  auto kernel = partition_kernel<KeyT>(cm.n > 2, shift);
  kernel<<<std::min(ntiles, most), kShNT, sm, s>>>(keys, n, tile, ntiles, pay_width, bs, F, hist, cm, reg_col, rid_in,
                                                   rid_out);
}

// Payload bytes a row takes in a tile of the columns of `cm`.
uint32_t move_pay_width(const ColMove &cm) {
  if (cm.n > 2) return 8;  // any column may pass through
  return cm.n < 2 ? 0u : (uint32_t)cm.width[1 - cm.key_index];
}

// One stable scatter pass over n rows into F <= kMaxFanout buckets.  If
// `start` (row numbers) or `start64` (64-bit offsets) is given it receives the
// F+1 bucket start positions.  If `total2` is given, the pass also counts rows
// per sub-bucket (nsub entries, zeroed by the caller) for a following RESERVE
// pass.
template <typename KeyT>
int stable_pass(Workspace &ws, const KeyT *keys, uint32_t n, const BucketSpec &bs, uint32_t F, const ColMove &cm,
                const uint32_t *rid_in, uint32_t *rid_out, uint32_t *start, int64_t *start64, uint32_t *total2,
                uint32_t nsub) {
  cudaStream_t s = ws.stream();
  MDJ_TRY(set_smem_attrs<KeyT>());
  if (n == 0) {
    if (start) MDJ_CUDA_TRY(cudaMemsetAsync(start, 0, (size_t)(F + 1) * 4, s));
    if (start64) MDJ_CUDA_TRY(cudaMemsetAsync(start64, 0, (size_t)(F + 1) * 8, s));
    return MDJ_OK;
  }
  const uint32_t pw = move_pay_width(cm);
  const uint32_t tile = stable_tile_rows(sizeof(KeyT), pw, rid_in != nullptr, F);
  const uint32_t ntiles = tile_count(n, tile);
  uint32_t *hist = (uint32_t *)ws.get((size_t)F * ntiles * 4);
  if (!hist) return MDJ_ERR_OOM;
  launch_hist<KeyT>(keys, n, bs, F, tile, ntiles, hist, total2, nsub, s);
  MDJ_LAUNCH_CHECK();
  MDJ_TRY(exclusive_scan_u32(ws, hist, hist, (size_t)F * ntiles));
  if (start || start64) {
    TraceScope tr("bucket_starts", s);
    if (start) k_bucket_starts<uint32_t><<<(F + 1 + 255) / 256, 256, 0, s>>>(hist, F, ntiles, n, start);
    if (start64) k_bucket_starts<int64_t><<<(F + 1 + 255) / 256, 256, 0, s>>>(hist, F, ntiles, n, start64);
  }
  MDJ_LAUNCH_CHECK();
  launch_partition<KeyT>(keys, n, bs, F, tile, ntiles, pw, hist, cm, rid_in, rid_out, s);
  MDJ_LAUNCH_CHECK();
  ws.give_back(hist);
  return MDJ_OK;
}

// Pass 2 of a two-level plan: rows grouped by pass-1 bucket (sb / F2) are
// split into final sub-buckets sb with atomic run reservation.
template <typename KeyT>
int reserve_pass(Workspace &ws, const KeyT *keys, uint32_t n, const BucketSpec &bs_sub, uint32_t F2,
                 uint32_t *cursors, const ColMove &cm, const uint32_t *rid_in, uint32_t *rid_out) {
  cudaStream_t s = ws.stream();
  MDJ_TRY(set_smem_attrs<KeyT>());
  const uint32_t ntiles = tile_count(n, kTile);
  if (ntiles == 0) return MDJ_OK;
  {
    TraceScope tr("scatter_reserve", s);
    k_scatter<KeyT, true><<<ntiles, kNW * 32, scatter_smem_bytes(kPass2SpanMax), s>>>(
        keys, n, bs_sub, 0, ntiles, nullptr, cursors, F2, cm, rid_in, rid_out);
  }
  MDJ_LAUNCH_CHECK();
  return MDJ_OK;
}

// Buffers of one partitioned copy of a table: every column and the row ids
// carved from one allocation (each part 256-byte aligned).
struct TableBufs {
  void *cols[MDJ_MAX_COLS];
  uint32_t *rid;
  void *block;
};

int alloc_table_bufs(Workspace &ws, const mdj_table *t, TableBufs *b, bool with_rid) {
  const size_t n = t->nrows;
  auto part = [](size_t bytes) { return (bytes + 255) & ~(size_t)255; };
  size_t total = with_rid ? part(n * 4) : 0;
  for (int j = 0; j < t->ncols; j++) total += part(n * dtype_width(t->cols[j].dtype));
  b->block = ws.get(total ? total : 256);
  if (!b->block) return MDJ_ERR_OOM;
  unsigned char *p = (unsigned char *)b->block;
  for (int j = 0; j < t->ncols; j++) {
    b->cols[j] = p;
    p += part(n * dtype_width(t->cols[j].dtype));
  }
  b->rid = with_rid ? (uint32_t *)p : nullptr;
  return MDJ_OK;
}

void release_table_bufs(Workspace &ws, const mdj_table *, TableBufs *b) { ws.give_back(b->block); }

ColMove make_move(const mdj_table *t, int32_t key_col, const void *const *src, void *const *dst) {
  ColMove cm;
  memset(&cm, 0, sizeof cm);
  cm.n = t->ncols;
  cm.key_index = key_col;
  for (int j = 0; j < t->ncols; j++) {
    cm.src[j] = src[j];
    cm.dst[j] = dst[j];
    cm.width[j] = dtype_width(t->cols[j].dtype);
  }
  return cm;
}

// ------------------------------------------------ unstable shuffle (host)

// MDJ_STABLE_SHUFFLE=1 makes the merge use the stable passes (for comparison).
bool fast_shuffle_enabled() {
  const char *e = getenv("MDJ_STABLE_SHUFFLE");
  return !(e && e[0] == '1');
}

template <typename KeyT>
auto shuffle_kernel(int mode, bool extra, bool wide) {
  constexpr int N = kShNT, W = kShWideNT;
  if (mode == SH_PASS2) return extra ? k_shuffle<KeyT, SH_PASS2, true, N> : k_shuffle<KeyT, SH_PASS2, false, N>;
  if (mode == SH_SEG) return extra ? k_shuffle<KeyT, SH_SEG, true, N> : k_shuffle<KeyT, SH_SEG, false, N>;
  if (mode == SH_TERM) return k_shuffle<KeyT, SH_TERM, false, N>;
  if (wide) return extra ? k_shuffle<KeyT, SH_PASS1, true, W> : k_shuffle<KeyT, SH_PASS1, false, W>;
  return extra ? k_shuffle<KeyT, SH_PASS1, true, N> : k_shuffle<KeyT, SH_PASS1, false, N>;
}

template <typename KeyT>
int set_shuffle_attrs() {
  static PerDeviceOnce once;
  return once_per_device(once, [] {
    const int sm = (int)kShSmem;
    for (int extra = 0; extra < 2; extra++) {
      for (int mode = 0; mode < 4; mode++)
        MDJ_CUDA_TRY(cudaFuncSetAttribute(shuffle_kernel<KeyT>(mode, extra != 0, false),
                                          cudaFuncAttributeMaxDynamicSharedMemorySize, sm));
      MDJ_CUDA_TRY(cudaFuncSetAttribute(shuffle_kernel<KeyT>(SH_PASS1, extra != 0, true),
                                        cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kShWideSmem));
    }
    MDJ_CUDA_TRY(cudaFuncSetAttribute(k_tot<KeyT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)(kMaxSubBuckets * 4)));
    return (int)MDJ_OK;
  });
}

// Payload bytes a row takes in a shuffle tile.
uint32_t shuffle_pay_width(const mdj_table *t, int32_t key_col) {
  if (t->ncols > 2) return 8;  // any column may pass through
  return t->ncols < 2 ? 0u : (uint32_t)dtype_width(t->cols[1 - key_col].dtype);
}

// One side of a pass; ntiles is set by shuffle_pass.
ShSide shuffle_side(const mdj_table *t, int32_t key_col, const void *const *src, void *const *dst,
                    const uint32_t *rid_in, uint32_t *rid_out, uint32_t *cursors) {
  ShSide sd;
  memset(&sd, 0, sizeof sd);
  sd.cm = make_move(t, key_col, src, dst);
  sd.keys = src[key_col];
  sd.rid_in = rid_in;
  sd.rid_out = rid_out;
  sd.cursors = cursors;
  sd.reg_col = t->ncols < 2 ? -1 : (key_col == 0 ? 1 : 0);
  sd.n = (uint32_t)t->nrows;
  return sd;
}

// One unstable shuffle pass (see k_shuffle) in tiles of `tile` rows; cursors:
// pass 1 one per pass-1 bucket, pass 2 and segments one per sub-bucket.  With
// segments the tiles are sg's (ntiles of them), else the sides' (both may
// have rows in pass 1 only).
template <typename KeyT>
int shuffle_pass(Workspace &ws, int mode, ShSides &sides, uint32_t tile, uint32_t pay_width, uint32_t ntiles,
                 const BucketSpec &bs, uint32_t F, uint32_t F2, uint32_t span, const SegArgs &sg, bool wide = false) {
  bool extra = false;
  for (ShSide &sd : sides.s) {
    sd.ntiles = tile_count(sd.n, tile);
    if (mode != SH_SEG) ntiles += sd.ntiles;
    extra = extra || (mode != SH_TERM && sd.cm.n > 2);
  }
  if (ntiles == 0) return MDJ_OK;
  const bool with_rid = mode == SH_PASS2 && sides.s[0].rid_in;
  const uint32_t sm = ShLayout(tile, sizeof(KeyT), pay_width, with_rid, span).total;
  const uint32_t most = (uint32_t)num_sms() * (wide ? 1 : kShBlocks);
  TraceScope tr(mode == SH_SEG ? "seg_scatter" : (mode == SH_PASS2 ? "shuffle_pass2" : "shuffle_pass1"), ws.stream());
  shuffle_kernel<KeyT>(mode, extra, wide)<<<std::min(ntiles, most), wide ? kShWideNT : kShNT, sm, ws.stream()>>>(
      sides, tile, ntiles, pay_width, bs, F, F2, span, sg);
  MDJ_LAUNCH_CHECK();
  return MDJ_OK;
}

// Tile rows of a pass over n rows (wide: in wide blocks): the largest tile, or,
// where that leaves the last wave of blocks part empty, the same number of
// waves of equal tiles (1024 rows at least: a tile has fixed costs of its own).
uint32_t balanced_tile(uint64_t n, uint32_t largest, bool wide = false) {
  const uint64_t slots = (uint64_t)num_sms() * (wide ? 1 : kShBlocks);
  const uint64_t waves = std::max<uint64_t>(1, (n + slots * largest - 1) / (slots * largest));
  const uint64_t even = ((n + slots * waves - 1) / (slots * waves) + 15) / 16 * 16;
  return (uint32_t)std::min<uint64_t>(largest, std::max<uint64_t>(even, 1024));
}

// Whether a pass 1 of n rows into F buckets runs in wide blocks: where two
// blocks per SM leave runs of 11 rows and fewer, and from 300 buckets on where
// there are many rows with a payload.  1e8 rows of 8 + 8 bytes, two blocks
// against one wide: 304 buckets 0.802 / 0.709 ms, 489 0.939 / 0.766, 604 1.094 /
// 0.781, 862 1.317 / 0.849, 1006 1.426 / 0.889 (before the two blocks: 0.793,
// 0.918, 0.961, 1.138, 1.233).  7e6 rows of 4 + 4 bytes: 304 0.041 / 0.044, 489
// 0.056 / 0.056, 604 0.072 / 0.060, 862 0.094 / 0.069; 1e6 at 604 0.027 / 0.024;
// 4e7 lone 8-byte keys: 374 0.217 / 0.232, 604 0.281 / 0.254.
bool wide_pass(uint32_t F, uint64_t n, uint32_t pay_width) {
  return F > 512 || (F >= 300 && pay_width > 0 && n >= (1u << 25));
}

// Rows per sub-bucket of one or both sides (n = 0: none) added to their tot.
template <typename KeyT>
int count_rows(Workspace &ws, TotSide A, TotSide B, const BucketSpec &bs, uint32_t nsub) {
  const size_t smem = (size_t)nsub * 4;
  int per_sm = 0;
  MDJ_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_tot<KeyT>, kTotThreads, smem));
  const uint64_t full = (uint64_t)num_sms() * std::max(per_sm, 1);
  const uint64_t chunk = (uint64_t)kTotThreads * kTotU;
  const uint64_t ca = (A.n + chunk - 1) / chunk, cb = (B.n + chunk - 1) / chunk;
  if (ca + cb == 0) return MDJ_OK;
  A.blocks = (uint32_t)ca;
  B.blocks = (uint32_t)cb;
  if (ca + cb > full) {  // resident blocks
    A.blocks = side_blocks(full, ca, cb);
    B.blocks = (uint32_t)full - A.blocks;
  }
  TraceScope tr("hist", ws.stream());
  k_tot<KeyT><<<A.blocks + B.blocks, kTotThreads, smem, ws.stream()>>>(A, B, bs, nsub);
  MDJ_LAUNCH_CHECK();
  return MDJ_OK;
}

// The merge's partition of one side with the unstable passes, first half:
// count the final sub-buckets, scan them into `off`, then the only pass
// (F2 == 1) or pass 1 (two-level plans) into freshly allocated `out`.
// cur2 (two-level plans): pass 2's cursors, allocated here and filled from
// the offsets by the same kernel as pass 1's.
template <typename KeyT>
int shuffle_count_pass1_t(Workspace &ws, const mdj_table *t, int32_t key_col, const Plan &plan, uint32_t *off,
                          TableBufs *out, uint32_t **cur2 = nullptr, int term = 0) {
  cudaStream_t s = ws.stream();
  MDJ_TRY(set_shuffle_attrs<KeyT>());
  const uint32_t n = (uint32_t)t->nrows;
  const uint32_t nsub = plan.nbuckets;
  const uint32_t F1 = plan.F2 == 1 ? nsub : plan.F1;
  const void *src[MDJ_MAX_COLS];
  for (int j = 0; j < t->ncols; j++) src[j] = t->cols[j].data;
  const KeyT *keys = (const KeyT *)src[key_col];
  const BucketSpec sub = make_spec(plan.P, plan.S, 1);

  MDJ_CUDA_TRY(cudaMemsetAsync(off, 0, (size_t)(nsub + 1) * 4, s));
  // with a term the rows leave as two columns, the key and the term
  const mdj_col term_cols[2] = {{nullptr, t->cols[key_col].dtype}, {nullptr, MDJ_U64}};
  const mdj_table term_table = {(mdj_col *)term_cols, 2, t->nrows};
  MDJ_TRY(alloc_table_bufs(ws, term ? &term_table : t, out, !term));
  if (n == 0) return MDJ_OK;
  uint32_t *cur = (uint32_t *)ws.get((size_t)(nsub + 1) * 4);
  if (!cur) return MDJ_ERR_OOM;
  if (cur2 && !(*cur2 = (uint32_t *)ws.get((size_t)(nsub + 1) * 4))) return MDJ_ERR_OOM;
  MDJ_TRY(count_rows<KeyT>(ws, TotSide{keys, off, n, 0}, TotSide{nullptr, nullptr, 0, 0}, sub, nsub));
  MDJ_TRY(exclusive_scan_u32(ws, off, off, (size_t)nsub + 1));
  {
    // pass-1 cursors: the first row of every pass-1 bucket
    TraceScope tr("pass1_cursors", s);
    const uint32_t nk = cur2 ? (F1 > nsub ? F1 : nsub) : F1;
    k_pass1_cursors<<<(nk + 255) / 256, 256, 0, s>>>(off, F1, plan.F2, cur, cur2 ? *cur2 : nullptr, nsub);
  }
  MDJ_LAUNCH_CHECK();
  const BucketSpec spec1 = plan.F2 == 1 ? sub : make_spec(plan.P, plan.S, plan.F2);
  const int32_t pay_col = t->ncols < 2 ? -1 : (key_col == 0 ? 1 : 0);
  const uint32_t pw = !term ? shuffle_pay_width(t, key_col) : pay_col < 0 ? 0u : dtype_width(t->cols[pay_col].dtype);
  const bool wide = !term && wide_pass(F1, n, pw);
  const uint32_t tile = balanced_tile(n, shuffle_tile_rows(sizeof(KeyT), pw, false, F1, wide), wide);
  ShSides sides;
  memset(&sides, 0, sizeof sides);
  if (term) {
    void *dst[MDJ_MAX_COLS] = {};
    dst[key_col] = out->cols[0];
    sides.s[0] = shuffle_side(t, key_col, src, dst, nullptr, nullptr, cur);
    sides.s[0].term = term;
    sides.s[0].term_dst = (uint64_t *)out->cols[1];
  } else {
    sides.s[0] = shuffle_side(t, key_col, src, out->cols, nullptr, out->rid, cur);
  }
  MDJ_TRY(shuffle_pass<KeyT>(ws, term ? SH_TERM : SH_PASS1, sides, tile, pw, 0, spec1, F1, plan.F2, F1, SegArgs{},
                             wide));
  ws.give_back(cur);
  return MDJ_OK;
}

// Second half of a two-level plan: pass 2 from the pass-1 copy `p1` into
// freshly allocated `fin` (sub-bucket offsets `off` from the first half).
template <typename KeyT>
int shuffle_pass2_t(Workspace &ws, const mdj_table *t, int32_t key_col, const Plan &plan, uint32_t *cur,
                    const TableBufs &p1, TableBufs *fin) {
  const uint32_t n = (uint32_t)t->nrows;
  MDJ_TRY(alloc_table_bufs(ws, t, fin, p1.rid != nullptr));
  if (n == 0) return MDJ_OK;
  // local buckets of a tile: the pass-1 buckets it is expected to touch (two
  // at least); a tile that touches more (a run of small ones) goes direct
  const uint64_t touched = 2 + (uint64_t)kShMaxTile * plan.F1 / n;
  const uint32_t span = (uint32_t)std::min<uint64_t>(touched * plan.F2, kPass2SpanMax);
  const uint32_t pw = shuffle_pay_width(t, key_col);
  const uint32_t tile = balanced_tile(n, shuffle_tile_rows(sizeof(KeyT), pw, p1.rid != nullptr, span));
  ShSides sides;
  memset(&sides, 0, sizeof sides);
  sides.s[0] = shuffle_side(t, key_col, p1.cols, fin->cols, p1.rid, fin->rid, cur);
  MDJ_TRY(shuffle_pass<KeyT>(ws, SH_PASS2, sides, tile, pw, 0, make_spec(plan.P, plan.S, 1), 0, plan.F2, span,
                             SegArgs{}));
  ws.give_back(cur);
  return MDJ_OK;
}

template <typename KeyT>
int shuffle_side_t(Workspace &ws, const mdj_table *t, int32_t key_col, const Plan &plan, uint32_t *off,
                   TableBufs *fin) {
  if (plan.F2 == 1) return shuffle_count_pass1_t<KeyT>(ws, t, key_col, plan, off, fin);
  TableBufs p1;
  uint32_t *cur2 = nullptr;
  MDJ_TRY(shuffle_count_pass1_t<KeyT>(ws, t, key_col, plan, off, &p1, &cur2));
  MDJ_TRY(shuffle_pass2_t<KeyT>(ws, t, key_col, plan, cur2, p1, fin));
  release_table_bufs(ws, t, &p1);
  return MDJ_OK;
}

// Both sides of a single-pass plan: the shuffle in one launch.
template <typename KeyT>
int shuffle_both_t(Workspace &ws, const mdj_table *left, int32_t lk, const mdj_table *right, int32_t rk,
                   const Plan &plan, uint32_t *curL, uint32_t *curR, TableBufs *fl, TableBufs *fr) {
  MDJ_TRY(set_shuffle_attrs<KeyT>());
  MDJ_TRY(alloc_table_bufs(ws, left, fl, true));
  MDJ_TRY(alloc_table_bufs(ws, right, fr, true));
  const void *src[2][MDJ_MAX_COLS];
  for (int j = 0; j < left->ncols; j++) src[0][j] = left->cols[j].data;
  for (int j = 0; j < right->ncols; j++) src[1][j] = right->cols[j].data;
  const uint32_t F = plan.nbuckets, pw = std::max(shuffle_pay_width(left, lk), shuffle_pay_width(right, rk));
  const bool wide = wide_pass(F, left->nrows + right->nrows, pw);
  const uint32_t tile =
      balanced_tile(left->nrows + right->nrows, shuffle_tile_rows(sizeof(KeyT), pw, false, F, wide), wide);
  ShSides sides;
  sides.s[0] = shuffle_side(left, lk, src[0], fl->cols, nullptr, fl->rid, curL);
  sides.s[1] = shuffle_side(right, rk, src[1], fr->cols, nullptr, fr->rid, curR);
  return shuffle_pass<KeyT>(ws, SH_PASS1, sides, tile, pw, 0, make_spec(plan.P, plan.S, 1), F, 1, F, SegArgs{}, wide);
}

// Stable partition by p with P > kMaxFanout: two stable LSD digit passes
// (p mod 1024, then p / 1024), which sort stably by p.  Writes into `dst`
// buffers; `off` (device u32[P+1]) receives the partition offsets.
template <typename KeyT>
int lsd_partition(Workspace &ws, const mdj_table *t, int32_t key_col, uint32_t P, void *const *dst_cols,
                  uint32_t *dst_rid, uint32_t *off) {
  const uint32_t n = (uint32_t)t->nrows;
  const void *src[MDJ_MAX_COLS];
  for (int j = 0; j < t->ncols; j++) src[j] = t->cols[j].data;
  TableBufs mid;
  MDJ_TRY(alloc_table_bufs(ws, t, &mid, true));
  const uint32_t d0 = kMaxFanout, d1 = (P + kMaxFanout - 1) / kMaxFanout;
  ColMove cm0 = make_move(t, key_col, src, mid.cols);
  MDJ_TRY(stable_pass<KeyT>(ws, (const KeyT *)src[key_col], n, make_digit_spec(P, 1, d0), d0, cm0, nullptr, mid.rid,
                            nullptr, nullptr, nullptr, 0));
  ColMove cm1 = make_move(t, key_col, mid.cols, dst_cols);
  MDJ_TRY(stable_pass<KeyT>(ws, (const KeyT *)mid.cols[key_col], n, make_digit_spec(P, d0, d1), d1, cm1, mid.rid,
                            dst_rid, nullptr, nullptr, nullptr, 0));
  release_table_bufs(ws, t, &mid);
  {
    TraceScope tr("offsets_bsearch", ws.stream());
    k_offsets_bsearch<KeyT><<<(P + 1 + 255) / 256, 256, 0, ws.stream()>>>((const KeyT *)dst_cols[key_col], n,
                                                                         make_spec(P, 1, 1), P, off);
  }
  MDJ_LAUNCH_CHECK();
  return MDJ_OK;
}

template <typename KeyT>
int stable_partition_t(Workspace &ws, const mdj_table *t, int32_t key_col, uint32_t P, void *const *out_cols,
                       uint32_t *out_rid, int64_t *out_offsets) {
  cudaStream_t s = ws.stream();
  const uint32_t n = (uint32_t)t->nrows;
  if (P <= kMaxFanout) {
    const void *src[MDJ_MAX_COLS];
    for (int j = 0; j < t->ncols; j++) src[j] = t->cols[j].data;
    ColMove cm = make_move(t, key_col, src, out_cols);
    return stable_pass<KeyT>(ws, (const KeyT *)src[key_col], n, make_spec(P, 1, 1), P, cm, nullptr, out_rid, nullptr,
                             out_offsets, nullptr, 0);
  }
  uint32_t *off = (uint32_t *)ws.get((size_t)(P + 1) * 4);
  if (!off) return MDJ_ERR_OOM;
  if (n == 0) {
    MDJ_CUDA_TRY(cudaMemsetAsync(off, 0, (size_t)(P + 1) * 4, s));
  } else {
    uint32_t *rid = out_rid ? out_rid : (uint32_t *)ws.get((size_t)n * 4);
    if (!rid) return MDJ_ERR_OOM;
    MDJ_TRY(lsd_partition<KeyT>(ws, t, key_col, P, out_cols, rid, off));
  }
  {
    TraceScope tr("offsets_i64", s);
    k_u32_to_i64<<<(P + 1 + 255) / 256, 256, 0, s>>>(off, out_offsets, P + 1);
  }
  MDJ_LAUNCH_CHECK();
  return MDJ_OK;
}

template <typename KeyT>
int partition_side_t(Workspace &ws, const mdj_table *t, int32_t key_col, const Plan &plan, Side *out) {
  cudaStream_t s = ws.stream();
  const uint32_t n = (uint32_t)t->nrows;
  const void *src[MDJ_MAX_COLS];
  for (int j = 0; j < t->ncols; j++) src[j] = t->cols[j].data;

  uint32_t *off = (uint32_t *)ws.get((size_t)(plan.nbuckets + 1) * 4);
  if (!off) return MDJ_ERR_OOM;
  TableBufs fin;
  fin.rid = nullptr;
  const void *key = src[key_col];
  const void *const *cols = src;
  const uint32_t *rid = nullptr;

  if (!plan.partition) {
    TraceScope tr("offsets_whole", s);
    k_two<<<1, 1, 0, s>>>(off, 0u, n);
    MDJ_LAUNCH_CHECK();
  } else if (!plan.lsd && !plan.stable && fast_shuffle_enabled()) {
    MDJ_TRY(shuffle_side_t<KeyT>(ws, t, key_col, plan, off, &fin));
    key = fin.cols[key_col];
    cols = fin.cols;
    rid = fin.rid;
  } else if (plan.lsd) {
    MDJ_TRY(alloc_table_bufs(ws, t, &fin, true));
    MDJ_TRY(lsd_partition<KeyT>(ws, t, key_col, plan.P, fin.cols, fin.rid, off));
    key = fin.cols[key_col];
    cols = fin.cols;
    rid = fin.rid;
  } else if (plan.F2 == 1) {
    MDJ_TRY(alloc_table_bufs(ws, t, &fin, true));
    ColMove cm = make_move(t, key_col, src, fin.cols);
    MDJ_TRY(stable_pass<KeyT>(ws, (const KeyT *)key, n, make_spec(plan.P, plan.S, 1), plan.nbuckets, cm, nullptr,
                              fin.rid, off, nullptr, nullptr, 0));
    key = fin.cols[key_col];
    cols = fin.cols;
    rid = fin.rid;
  } else {
    // pass 1: F1 = P*S/F2 stable buckets, counting the final sub-buckets too
    uint32_t *cur = (uint32_t *)ws.get((size_t)(plan.nbuckets + 1) * 4);
    if (!cur) return MDJ_ERR_OOM;
    MDJ_CUDA_TRY(cudaMemsetAsync(off, 0, (size_t)(plan.nbuckets + 1) * 4, s));
    TableBufs p1;
    MDJ_TRY(alloc_table_bufs(ws, t, &p1, true));
    ColMove cm1 = make_move(t, key_col, src, p1.cols);
    MDJ_TRY(stable_pass<KeyT>(ws, (const KeyT *)key, n, make_spec(plan.P, plan.S, plan.F2), plan.F1, cm1, nullptr,
                              p1.rid, nullptr, nullptr, off, plan.nbuckets));
    MDJ_TRY(exclusive_scan_u32(ws, off, off, plan.nbuckets + 1));
    MDJ_CUDA_TRY(cudaMemcpyAsync(cur, off, (size_t)plan.nbuckets * 4, cudaMemcpyDeviceToDevice, s));
    // pass 2
    MDJ_TRY(alloc_table_bufs(ws, t, &fin, true));
    ColMove cm2 = make_move(t, key_col, p1.cols, fin.cols);
    MDJ_TRY(reserve_pass<KeyT>(ws, (const KeyT *)p1.cols[key_col], n, make_spec(plan.P, plan.S, 1), plan.F2, cur,
                               cm2, p1.rid, fin.rid));
    release_table_bufs(ws, t, &p1);
    ws.give_back(cur);
    key = fin.cols[key_col];
    cols = fin.cols;
    rid = fin.rid;
  }

  out->key = key;
  out->key_dtype = t->cols[key_col].dtype;
  out->ncols = 0;
  for (int j = 0; j < t->ncols; j++) {
    if (j == key_col) continue;
    out->cols[out->ncols] = cols[j];
    out->widths[out->ncols] = dtype_width(t->cols[j].dtype);
    out->dtypes[out->ncols] = t->cols[j].dtype;
    out->ncols++;
  }
  out->rid = rid;
  out->off = off;
  out->nrows = n;
  return MDJ_OK;
}

}  // namespace

Plan make_plan(uint64_t n_build, uint32_t P, uint32_t cap, bool force_partition, bool stable) {
  Plan pl;
  pl.stable = stable;
  const bool stable_passes = stable || !fast_shuffle_enabled();
  pl.P = P;
  pl.cap = cap;
  // target mean build rows per sub-bucket: ~85% of a table, so that hash
  // variance rarely overflows one table
  uint64_t target = (uint64_t)cap * 85 / 100;
  // small build sides: enough sub-buckets for every resident block of the join,
  // the count and the grouping (two per SM), of at least kMinBucketRows rows; a
  // side that fits one table still stays whole.  With whole tables instead:
  // merge of 1e6 x 2e8 rows 4.00 ms (3.86), count of 2e5 x 1e8 1.60 (1.54),
  // stream of 2e5 x 5e7 1.66 (1.62), but merge of 2e5 x 2e8 3.56 (3.65: the join
  // 0.15 less, the shuffle 0.25 more).  Not for the stable passes, whose cost
  // grows with the buckets (ordered output of 500K x 500K rows 0.21 ms, 0.23
  // with more).
  if (!stable_passes && n_build > target)
    target = std::min(target, std::max<uint64_t>(kMinBucketRows, n_build / (2 * (uint64_t)num_sms()) + 1));
  uint64_t need = (n_build + target - 1) / target;
  if (need < 1) need = 1;
  if (P > kMaxFanout) {
    pl.lsd = true;
    pl.S = 1;
    pl.nbuckets = P;
    pl.F1 = P;
    pl.F2 = 1;
    return pl;
  }
  if (P == 1 && need == 1 && !force_partition) {
    pl.partition = false;
    pl.S = 1;
    pl.nbuckets = 1;
    return pl;
  }
  uint64_t S = (need + P - 1) / P;
  if (S < 1) S = 1;
  if ((uint64_t)P * S <= kMaxFanout) {
    pl.S = (uint32_t)S;
    pl.F1 = P * pl.S;
    pl.F2 = 1;
    pl.nbuckets = pl.F1;
    return pl;
  }
  const uint32_t fan = stable_passes ? kStableFanout : kMergeFanout;
  const TwoPassSplit sp = two_pass_split(P, S, fan, kMaxSubBuckets, kPass2SpanMax / 2);
  pl.F2 = sp.F2;
  pl.S = sp.S1 * sp.F2;
  pl.F1 = P * sp.S1;
  pl.nbuckets = P * pl.S;
  return pl;
}

int partition_side(Workspace &ws, const mdj_table *t, int32_t key_col, const Plan &plan, Side *out) {
  if (t->cols[key_col].dtype == MDJ_I64) return partition_side_t<int64_t>(ws, t, key_col, plan, out);
  return partition_side_t<int32_t>(ws, t, key_col, plan, out);
}

namespace {
void fill_side(const mdj_table *t, int32_t key_col, const TableBufs &b, uint32_t *off, Side *out) {
  out->key = b.cols[key_col];
  out->key_dtype = t->cols[key_col].dtype;
  out->ncols = 0;
  for (int j = 0; j < t->ncols; j++) {
    if (j == key_col) continue;
    out->cols[out->ncols] = b.cols[j];
    out->widths[out->ncols] = dtype_width(t->cols[j].dtype);
    out->dtypes[out->ncols] = t->cols[j].dtype;
    out->ncols++;
  }
  out->rid = b.rid;
  out->off = off;
  out->nrows = t->nrows;
}
}  // namespace

namespace {
// The checksum term of every row (plans without the fast shuffle).
template <typename KeyT>
__global__ void k_terms(const KeyT *__restrict__ keys, const void *pay, int pw, uint32_t n, int term,
                        uint64_t *__restrict__ out) {
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint64_t r = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += stride) {
    const uint64_t pb = pay_bits(pay, pw, (uint32_t)r);
    out[r] = term == TERM_F ? term_f(key_bits(keys[r]), (uint32_t)r, pb) : term_g((uint32_t)r, pb);
  }
}

template <typename KeyT>
int partition_terms_t(Workspace &ws, const mdj_table *t, int32_t key_col, const Plan &plan, int term, Side *out) {
  cudaStream_t s = ws.stream();
  const uint32_t n = (uint32_t)t->nrows;
  mdj_col cols[2] = {t->cols[key_col], {nullptr, MDJ_U64}};
  mdj_table tt = {cols, 2, t->nrows};
  if (plan.partition && !plan.lsd && !plan.stable && fast_shuffle_enabled()) {
    uint32_t *off = (uint32_t *)ws.get((size_t)(plan.nbuckets + 1) * 4);
    if (!off) return MDJ_ERR_OOM;
    TableBufs fin, p1;
    if (plan.F2 == 1) {
      MDJ_TRY(shuffle_count_pass1_t<KeyT>(ws, t, key_col, plan, off, &fin, nullptr, term));
    } else {
      uint32_t *cur2 = nullptr;
      MDJ_TRY(shuffle_count_pass1_t<KeyT>(ws, t, key_col, plan, off, &p1, &cur2, term));
      MDJ_TRY(shuffle_pass2_t<KeyT>(ws, &tt, 0, plan, cur2, p1, &fin));
      release_table_bufs(ws, &tt, &p1);
    }
    fill_side(&tt, 0, fin, off, out);
    return MDJ_OK;
  }
  uint64_t *terms = (uint64_t *)ws.get((size_t)(n ? n : 1) * 8);
  if (!terms) return MDJ_ERR_OOM;
  const int32_t pay_col = t->ncols < 2 ? -1 : (key_col == 0 ? 1 : 0);
  if (n) {
    TraceScope tr("count_terms", s);
    k_terms<KeyT><<<std::min(tile_count(n, 256), (uint32_t)num_sms() * 8), 256, 0, s>>>(
        (const KeyT *)t->cols[key_col].data, pay_col < 0 ? nullptr : t->cols[pay_col].data,
        pay_col < 0 ? 0 : dtype_width(t->cols[pay_col].dtype), n, term, terms);
  }
  MDJ_LAUNCH_CHECK();
  cols[1].data = terms;
  return partition_side_t<KeyT>(ws, &tt, 0, plan, out);
}
}  // namespace

int partition_terms(Workspace &ws, const mdj_table *t, int32_t key_col, const Plan &plan, bool left, Side *out) {
  const int term = left ? TERM_F : TERM_G;
  return t->cols[key_col].dtype == MDJ_I64 ? partition_terms_t<int64_t>(ws, t, key_col, plan, term, out)
                                           : partition_terms_t<int32_t>(ws, t, key_col, plan, term, out);
}

bool plan_fits_one_launch(const Plan &plan) {
  return !plan.partition || (!plan.lsd && !plan.stable && plan.F2 == 1 && fast_shuffle_enabled());
}

int count_both(Workspace &ws, const mdj_table *left, int32_t lk, const mdj_table *right, int32_t rk, const Plan &plan,
               uint32_t *totL, uint32_t *totR) {
  const TotSide A = {left->cols[lk].data, totL, (uint32_t)left->nrows, 0};
  const TotSide B = {right->cols[rk].data, totR, (uint32_t)right->nrows, 0};
  const BucketSpec bs = make_spec(plan.P, plan.S, 1);
  return left->cols[lk].dtype == MDJ_I64 ? count_rows<int64_t>(ws, A, B, bs, plan.nbuckets)
                                         : count_rows<int32_t>(ws, A, B, bs, plan.nbuckets);
}

int shuffle_both(Workspace &ws, const mdj_table *left, int32_t lk, const mdj_table *right, int32_t rk,
                 const Plan &plan, uint32_t *offL, uint32_t *offR, uint32_t *curL, uint32_t *curR, Side *L, Side *R) {
  TableBufs fl, fr;
  if (plan.partition) {
    MDJ_TRY(left->cols[lk].dtype == MDJ_I64
                ? shuffle_both_t<int64_t>(ws, left, lk, right, rk, plan, curL, curR, &fl, &fr)
                : shuffle_both_t<int32_t>(ws, left, lk, right, rk, plan, curL, curR, &fl, &fr));
  } else {
    for (int j = 0; j < left->ncols; j++) fl.cols[j] = (void *)left->cols[j].data;
    for (int j = 0; j < right->ncols; j++) fr.cols[j] = (void *)right->cols[j].data;
    fl.rid = fr.rid = nullptr;
  }
  fill_side(left, lk, fl, offL, L);
  fill_side(right, rk, fr, offR, R);
  return MDJ_OK;
}

int stable_partition(Workspace &ws, const mdj_table *t, int32_t key_col, uint32_t P, void *const *out_cols,
                     uint32_t *out_rid, int64_t *out_offsets) {
  if (t->cols[key_col].dtype == MDJ_I64)
    return stable_partition_t<int64_t>(ws, t, key_col, P, out_cols, out_rid, out_offsets);
  return stable_partition_t<int32_t>(ws, t, key_col, P, out_cols, out_rid, out_offsets);
}

}  // namespace mdj

namespace mdj {
namespace {

template <typename KeyT>
int stable_partition_scratch_t(const mdj_table *t, int32_t key_col, uint32_t P, void *const *out_cols,
                               uint32_t *out_rid, int64_t *out_offsets, uint32_t *scratch, size_t scratch_words,
                               cudaStream_t s) {
  const uint32_t n = (uint32_t)t->nrows, F = P;
  if (stable_partition_scratch_words(n, P) > scratch_words) return MDJ_ERR_TOO_LARGE;
  MDJ_TRY(set_smem_attrs<KeyT>());
  if (n == 0) {
    MDJ_CUDA_TRY(cudaMemsetAsync(out_offsets, 0, (size_t)(F + 1) * 8, s));
    return MDJ_OK;
  }
  const void *src[MDJ_MAX_COLS];
  for (int j = 0; j < t->ncols; j++) src[j] = t->cols[j].data;
  const KeyT *keys = (const KeyT *)src[key_col];
  const ColMove cm = make_move(t, key_col, src, out_cols);
  const BucketSpec bs = make_spec(P, 1, 1);
  const uint32_t pw = move_pay_width(cm);
  // (tiles have at least kTile rows here, so the matrix fits the scratch words
  // counted for kTile-row tiles)
  const uint32_t tile = stable_tile_rows(sizeof(KeyT), pw, false, F);
  const uint32_t ntiles = tile_count(n, tile);
  const size_t nhist = (size_t)F * ntiles;
  uint32_t *hist = scratch, *sums = hist + nhist;
  launch_hist<KeyT>(keys, n, bs, F, tile, ntiles, hist, nullptr, 0, s);
  MDJ_LAUNCH_CHECK();
  MDJ_TRY(exclusive_scan_u32_scratch(hist, hist, nhist, sums, s));
  k_bucket_starts<int64_t><<<(F + 1 + 255) / 256, 256, 0, s>>>(hist, F, ntiles, n, out_offsets);
  MDJ_LAUNCH_CHECK();
  launch_partition<KeyT>(keys, n, bs, F, tile, ntiles, pw, hist, cm, nullptr, out_rid, s);
  MDJ_LAUNCH_CHECK();
  return MDJ_OK;
}

}  // namespace

size_t stable_partition_scratch_words(uint64_t n, uint32_t P) {
  const uint64_t nhist = (uint64_t)P * ((n + kTile - 1) / kTile);
  return (size_t)(nhist + scan_scratch_words(nhist) + P + 1);
}

int stable_partition_scratch(const mdj_table *t, int32_t key_col, uint32_t P, void *const *out_cols,
                             uint32_t *out_rid, int64_t *out_offsets, uint32_t *scratch, size_t scratch_words,
                             cudaStream_t s) {
  if (t->cols[key_col].dtype == MDJ_I64)
    return stable_partition_scratch_t<int64_t>(t, key_col, P, out_cols, out_rid, out_offsets, scratch,
                                               scratch_words, s);
  return stable_partition_scratch_t<int32_t>(t, key_col, P, out_cols, out_rid, out_offsets, scratch, scratch_words,
                                             s);
}

}  // namespace mdj

// ------------------------------------------------- segmented (batched) form
namespace mdj {
namespace {

// totals[seg_base + b] += rows of bucket b of each segment.  A block counts a
// contiguous run of tiles and adds its counters to the totals only where the
// segment changes (once per tile, one load in flight: 0.61 vs 0.42 ms for 246M rows in 512
// segments); kSegHistU keys per thread are loaded before any is counted.
constexpr int kSegHistU = 8;
template <typename KeyT>
__global__ void __launch_bounds__(kHistThreads) k_seg_hist(const KeyT *__restrict__ keys, const SegArgs sg,
                                                           uint32_t ntiles, uint32_t *__restrict__ totals) {
  extern __shared__ uint32_t cnt[];
  const uint32_t per = (ntiles + gridDim.x - 1) / gridDim.x;
  const uint32_t t0 = min(ntiles, blockIdx.x * per), t1 = min(ntiles, t0 + per);
  uint32_t seg = 0xFFFFFFFFu, NB = 0, B = 0;
  BucketSpec sp;
  for (uint32_t t = t0; t < t1; t++) {
    const SegTile td = sg.tiles[t];
    if (td.seg != seg) {  // uniform over the block
      __syncthreads();
      for (uint32_t b = threadIdx.x; b < NB; b += kHistThreads)
        if (cnt[b]) atomicAdd(&totals[B + b], cnt[b]);
      seg = td.seg;
      NB = sg.nb[seg];
      B = sg.base[seg];
      sp = make_spec_dev(sg.P[seg]);
      sp.S = sg.S[seg];
      __syncthreads();
      for (uint32_t b = threadIdx.x; b < NB; b += kHistThreads) cnt[b] = 0;
      __syncthreads();
    }
    const KeyT *k = keys + td.row0;
    for (uint32_t i0 = threadIdx.x; i0 < td.rows; i0 += kHistThreads * kSegHistU) {
      KeyT kv[kSegHistU];
#pragma unroll
      for (int u = 0; u < kSegHistU; u++) {
        const uint32_t i = i0 + u * kHistThreads;
        kv[u] = i < td.rows ? k[i] : KeyT(0);
      }
#pragma unroll
      for (int u = 0; u < kSegHistU; u++)
        if (i0 + u * kHistThreads < td.rows) atomicAdd(&cnt[sub_bucket_of(fmix64(key_bits(kv[u])), sp)], 1u);
    }
  }
  __syncthreads();
  for (uint32_t b = threadIdx.x; b < NB; b += kHistThreads)
    if (cnt[b]) atomicAdd(&totals[B + b], cnt[b]);
}

template <typename T>
T *upload(Workspace &ws, const std::vector<T> &v) {
  T *d = (T *)ws.get(v.size() * sizeof(T) + 16);
  if (!d) return nullptr;
  if (!v.empty() && cudaMemcpyAsync(d, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, ws.stream()) !=
                        cudaSuccess)
    return nullptr;
  return d;
}

template <typename KeyT>
int seg_partition_t(Workspace &ws, const mdj_table *t, int32_t key_col, const uint64_t *seg_off, uint32_t nseg,
                    const uint32_t *seg_base, const uint32_t *seg_nb, const uint32_t *seg_P, uint32_t nb,
                    Side *out) {
  cudaStream_t s = ws.stream();
  const uint32_t n = (uint32_t)t->nrows;
  const void *src[MDJ_MAX_COLS];
  for (int j = 0; j < t->ncols; j++) src[j] = t->cols[j].data;
  bool all_single = true;
  for (uint32_t i = 0; i < nseg; i++) all_single = all_single && seg_nb[i] == 1;

  const void *key = src[key_col];
  const void *const *cols = src;
  const uint32_t *rid = nullptr;
  uint32_t *off = nullptr;
  TableBufs fin;
  fin.rid = nullptr;
  if (all_single) {
    // every segment is one bucket: bucket offsets are the segment offsets
    std::vector<uint32_t> h(nseg + 1);
    for (uint32_t i = 0; i <= nseg; i++) h[i] = (uint32_t)seg_off[i];
    off = upload(ws, h);
    if (!off) return MDJ_ERR_OOM;
  } else {
    MDJ_TRY(set_shuffle_attrs<KeyT>());
    uint32_t smax = 1;
    for (uint32_t i = 0; i < nseg; i++) smax = std::max(smax, seg_nb[i]);
    const uint32_t tile = shuffle_tile_rows(sizeof(KeyT), shuffle_pay_width(t, key_col), false, smax);
    std::vector<SegTile> tiles;
    for (uint32_t i = 0; i < nseg; i++)
      for (uint64_t r = seg_off[i]; r < seg_off[i + 1]; r += tile)
        tiles.push_back(SegTile{(uint32_t)r, (uint32_t)std::min<uint64_t>(tile, seg_off[i + 1] - r), i});
    std::vector<uint32_t> hb(seg_base, seg_base + nseg), hs(seg_nb, seg_nb + nseg), hp(seg_P, seg_P + nseg),
        hS(nseg);
    for (uint32_t i = 0; i < nseg; i++) hS[i] = seg_nb[i] / seg_P[i];
    SegTile *dt = upload(ws, tiles);
    uint32_t *db = upload(ws, hb), *ds = upload(ws, hs), *dp = upload(ws, hp), *dS = upload(ws, hS);
    off = (uint32_t *)ws.get((size_t)(nb + 1) * 4);
    uint32_t *cur = (uint32_t *)ws.get((size_t)(nb + 1) * 4);
    if (!dt || !db || !ds || !dp || !dS || !off || !cur) return MDJ_ERR_OOM;
    const SegArgs sg = {dt, db, ds, dp, dS};
    const uint32_t ntiles = (uint32_t)tiles.size();
    MDJ_CUDA_TRY(cudaMemsetAsync(off, 0, (size_t)(nb + 1) * 4, s));
    if (ntiles) {
      TraceScope tr("seg_hist", s);
      const uint32_t most = (uint32_t)num_sms() * (2048 / kHistThreads);
      k_seg_hist<KeyT><<<std::min(ntiles, most), kHistThreads, smax * 4, s>>>((const KeyT *)key, sg, ntiles, off);
    }
    MDJ_LAUNCH_CHECK();
    MDJ_TRY(exclusive_scan_u32(ws, off, off, nb + 1));
    MDJ_CUDA_TRY(cudaMemcpyAsync(cur, off, (size_t)nb * 4, cudaMemcpyDeviceToDevice, s));
    MDJ_TRY(alloc_table_bufs(ws, t, &fin, true));
    ShSides sides;
    memset(&sides, 0, sizeof sides);
    sides.s[0] = shuffle_side(t, key_col, src, fin.cols, nullptr, fin.rid, cur);
    MDJ_TRY(shuffle_pass<KeyT>(ws, SH_SEG, sides, tile, shuffle_pay_width(t, key_col), ntiles, make_spec(1, 1, 1), 0, 1,
                               smax, sg));
    key = fin.cols[key_col];
    cols = fin.cols;
    rid = fin.rid;
  }
  out->key = key;
  out->key_dtype = t->cols[key_col].dtype;
  out->ncols = 0;
  for (int j = 0; j < t->ncols; j++) {
    if (j == key_col) continue;
    out->cols[out->ncols] = cols[j];
    out->widths[out->ncols] = dtype_width(t->cols[j].dtype);
    out->dtypes[out->ncols] = t->cols[j].dtype;
    out->ncols++;
  }
  out->rid = rid;
  out->off = off;
  out->nrows = n;
  return MDJ_OK;
}

}  // namespace

int partition_side_segmented(Workspace &ws, const mdj_table *t, int32_t key_col, const uint64_t *seg_off,
                             uint32_t nseg, const uint32_t *seg_base, const uint32_t *seg_nb, const uint32_t *seg_P,
                             uint32_t nbuckets, Side *out) {
  if (t->cols[key_col].dtype == MDJ_I64)
    return seg_partition_t<int64_t>(ws, t, key_col, seg_off, nseg, seg_base, seg_nb, seg_P, nbuckets, out);
  return seg_partition_t<int32_t>(ws, t, key_col, seg_off, nseg, seg_base, seg_nb, seg_P, nbuckets, out);
}

}  // namespace mdj
