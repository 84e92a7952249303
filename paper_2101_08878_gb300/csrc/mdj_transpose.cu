// The paper's second workload: the sum of an array and its transpose,
// y = x + x^T (Sec. V-B "Sum of cuPy Array and its Transpose", Fig. 7:
// 16K x 16K in 4K chunks; Sec. V-C, Fig. 9(a): 20E3 x 20E3 in 5E2 chunks).
// With the chunks spread over Dask workers, chunk (i, j) of y needs chunk
// (j, i) of x from another worker: that exchange is what the benchmark times.
// On one GPU the chunk exchange is the read of the mirrored tile.
//
// One block handles a pair of mirrored square tiles, (I, J) and (J, I) with
// I <= J: it loads both into registers, puts both in shared memory, and
// writes y(I, J) = x(I, J) + x(J, I)^T and y(J, I) = x(J, I) + x(I, J)^T, the
// direct term from registers and the mirrored one from shared memory.  Every
// element of x is read once and every element of y written once (16 bytes
// per float64 element), with coalesced rows both ways.  A block reads both
// tiles before it writes either, and no other block touches them, so y may
// be x (in place).  Integer types add with wraparound; float types with one
// IEEE addition, so the result is exact and symmetric.
#include <string.h>

#include "mdj_internal.cuh"

namespace mdj {
namespace {

template <typename V>
__device__ __forceinline__ V add(V a, V b) {
  return a + b;
}

// A thread holds E x E squares of a tile (E = 16 bytes of elements where rows
// are 16-byte aligned, else 1), row by row, so that both the direct and the
// mirrored side move as whole 16-byte words: square (g, q) needs rows qE ..
// qE + E - 1 of the mirrored tile, word g of each, transposed in registers.
// In shared memory word q of row r sits at q ^ (r / E mod 8) of its row, so 8
// threads of consecutive q, which read the same g in rows E apart, meet 8
// different 16-byte banks (E = 1: rows are padded by one element instead).
template <typename V, int TT, int E, int NT>
struct Geom {
  static constexpr int W = TT / E;                 // words (squares) per row
  static constexpr int SQ = W * W / NT;             // squares per thread
  static constexpr uint32_t kElems = E == 1 ? TT * (TT + 1) : TT * TT;
  static constexpr int ROWS = NT / W;               // rows of squares the block covers at once
  static_assert(SQ * ROWS == W && ROWS * W == NT, "whole rows of squares");
  static __device__ __forceinline__ uint32_t at(uint32_t row, uint32_t q) {
    return E == 1 ? row * (TT + 1) + q : (row * W + (q ^ ((row / E) & 7))) * E;
  }
};

template <typename V, int E>
struct alignas(sizeof(V) * E) Word {
  V v[E];
};

template <typename V, int TT, int E, int NT>
__device__ __forceinline__ void load_tile(const V *x, uint64_t n, uint64_t r0, uint64_t c0,
                                          Word<V, E> (&a)[Geom<V, TT, E, NT>::SQ][E]) {
  using G = Geom<V, TT, E, NT>;
  const uint32_t g0 = threadIdx.x / G::W, q = threadIdx.x % G::W;
  const uint64_t c = c0 + q * E;
  const V *row = x + (r0 + g0 * E) * n + c;
#pragma unroll
  for (int s = 0; s < G::SQ; s++) {
#pragma unroll
    for (int e = 0; e < E; e++) {
      if (r0 + (g0 + s * G::ROWS) * E + e < n && c < n)
        a[s][e] = *(const Word<V, E> *)(row + e * n);
      else
        a[s][e] = Word<V, E>{};
    }
    row += G::ROWS * E * n;
  }
}

template <typename V, int TT, int E, int NT>
__device__ __forceinline__ void put_tile(V *T, const Word<V, E> (&a)[Geom<V, TT, E, NT>::SQ][E]) {
  using G = Geom<V, TT, E, NT>;
  const uint32_t g0 = threadIdx.x / G::W, q = threadIdx.x % G::W;
#pragma unroll
  for (int s = 0; s < G::SQ; s++)
#pragma unroll
    for (int e = 0; e < E; e++) *(Word<V, E> *)(T + G::at((g0 + s * G::ROWS) * E + e, q)) = a[s][e];
}

// y rows r0 + .. (columns c0 + ..) = a[r][c] + M[c][r].
template <typename V, int TT, int E, int NT>
__device__ __forceinline__ void store_sum(V *y, uint64_t n, uint64_t r0, uint64_t c0,
                                          const Word<V, E> (&a)[Geom<V, TT, E, NT>::SQ][E], const V *M) {
  using G = Geom<V, TT, E, NT>;
  const uint32_t g0 = threadIdx.x / G::W, q = threadIdx.x % G::W;
  const uint64_t c = c0 + q * E;
  V *row = y + (r0 + g0 * E) * n + c;
#pragma unroll
  for (int s = 0; s < G::SQ; s++) {
    Word<V, E> m[E];
#pragma unroll
    for (int e = 0; e < E; e++) m[e] = *(const Word<V, E> *)(M + G::at(q * E + e, g0 + s * G::ROWS));
#pragma unroll
    for (int e = 0; e < E; e++) {
      Word<V, E> o;
#pragma unroll
      for (int f = 0; f < E; f++) o.v[f] = add(a[s][e].v[f], m[f].v[e]);
      if (r0 + (g0 + s * G::ROWS) * E + e < n && c < n) *(Word<V, E> *)(row + e * n) = o;
    }
    row += G::ROWS * E * n;
  }
}

template <typename V, int TT, int E, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB)
    k_transpose_add(const V *x, V *y, uint64_t n, uint32_t nt) {
  extern __shared__ __align__(16) unsigned char smem[];
  using G = Geom<V, TT, E, NT>;
  V *A = (V *)smem;        // x tile (I, J)
  V *B = A + G::kElems;    // x tile (J, I)
  // pairs (I, J), I <= J, row by row: this block takes every gridDim.x-th
  uint64_t J = blockIdx.x;
  for (uint32_t I = 0;; J += gridDim.x) {
    while (J >= nt && I < nt) J = J - nt + ++I;  // past row I's end: on into row I + 1, which starts at column I + 1
    if (I >= nt) return;
    const uint64_t rI = (uint64_t)I * TT, rJ = J * TT;
    Word<V, E> a[G::SQ][E], b[G::SQ][E];
    load_tile<V, TT, E, NT>(x, n, rI, rJ, a);
    if (I != J) load_tile<V, TT, E, NT>(x, n, rJ, rI, b);
    put_tile<V, TT, E, NT>(A, a);
    if (I != J) put_tile<V, TT, E, NT>(B, b);
    __syncthreads();
    store_sum<V, TT, E, NT>(y, n, rI, rJ, a, I != J ? B : A);
    if (I != J) store_sum<V, TT, E, NT>(y, n, rJ, rI, b, A);
    __syncthreads();
  }
}

template <typename V, int TT, int E, int NT, int MINB>
int launch_e(const void *x, void *y, uint64_t n, cudaStream_t s) {
  const uint32_t nt = (uint32_t)((n + TT - 1) / TT);
  const uint64_t npairs = (uint64_t)nt * (nt + 1) / 2;
  const size_t sm = 2 * (size_t)Geom<V, TT, E, NT>::kElems * sizeof(V);
  static PerDeviceOnce once;
  MDJ_TRY(once_per_device(once, [sm] {
    MDJ_CUDA_TRY(cudaFuncSetAttribute(k_transpose_add<V, TT, E, NT, MINB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)sm));
    return (int)MDJ_OK;
  }));
  const uint64_t most = (uint64_t)num_sms() * MINB;
  const unsigned grid = (unsigned)(npairs < most ? npairs : most);
  TraceScope tr("transpose_add", s);
  k_transpose_add<V, TT, E, NT, MINB><<<grid, NT, sm, s>>>((const V *)x, (V *)y, n, nt);
  MDJ_LAUNCH_CHECK();
  return MDJ_OK;
}

// What bounds it: DRAM.  16384^2 float64: 0.99 -> 0.672 ms (6.4 TB/s, 94% of
// a plain copy's rate); float32: 0.450 -> 0.349 ms.  The kernel it replaced
// spent its time on the FP64 pipe (few units on this GPU), finding each pair
// by a double-precision square root in every thread; the pair walk above is
// integer only.  Whole words need rows on 16-byte boundaries; tile rows are
// then 256 bytes and a block is small, so that five (4-byte types: three)
// blocks per SM overlap their load and store phases: at 16384^2 float64, 4 /
// 5 / 6 / 8 blocks 0.716 / 0.672 / 0.681 / 0.738 ms; float32, 3 / 4 / 5 / 6:
// 0.349 / 0.357 / 0.360 / 0.569 (the last spills).  Otherwise single elements,
// where 64-edge tiles and 512 threads were the fastest: 16383^2 float64 1.137
// -> 0.829 ms, float32 0.490 -> 0.474 ms.
template <typename V>
int launch(const void *x, void *y, uint64_t n, cudaStream_t s) {
  constexpr int E = 16 / sizeof(V);
  const bool words = (((uintptr_t)x | (uintptr_t)y) & 15) == 0 && n % E == 0;
  return words ? launch_e<V, 256 / sizeof(V), E, 256, sizeof(V) == 8 ? 5 : 3>(x, y, n, s)
               : launch_e<V, 64, 1, 512, 2>(x, y, n, s);
}

}  // namespace
}  // namespace mdj

extern "C" int mdj_transpose_add(const void *x, void *y, uint64_t n, int32_t dtype, void *stream) {
  using namespace mdj;
  const int w = dtype_width(dtype);
  if (w == 0) return MDJ_ERR_UNSUPPORTED_DTYPE;
  if (n == 0) return MDJ_OK;
  if (!x || !y) return MDJ_ERR_INVALID_ARG;
  if (n >= (1ull << 32)) return MDJ_ERR_TOO_LARGE;
  const uint64_t bytes = n * n * (uint64_t)w;
  const uintptr_t xa = (uintptr_t)x, ya = (uintptr_t)y;
  if (xa != ya && xa < ya + bytes && ya < xa + bytes) return MDJ_ERR_INVALID_ARG;  // partial overlap
  if (xa % w || ya % w) return MDJ_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  switch (dtype) {
    case MDJ_F32: return launch<float>(x, y, n, s);
    case MDJ_F64: return launch<double>(x, y, n, s);
    case MDJ_I32: case MDJ_U32: return launch<uint32_t>(x, y, n, s);  // wraparound add
    default: return launch<uint64_t>(x, y, n, s);
  }
}
