// Shared parts of the streaming column passes over row-major n x m blocks
// (column sums of squares, dot products, residual norms).
//
// Mapping: the threads of a CTA are laid out row after row over col_tile(m)
// consecutive columns, so a warp runs across the end of a row into the next
// one.  With a warp per 32-column tile instead, m = 71 leaves 25 of 32 lanes
// idle in the third tile of every row, and an FP64 instruction costs the same
// pipe time with 7 lanes as with 32.
//
// Second pass: the CTA partials (up to 608 per column) are summed by 32
// threads per column and a fixed tree; one thread per column is a chain of
// 608 dependent L2 loads (131 us at 71 columns, more than the bytes of a
// whole pass; 3 us now).
#pragma once
#include "kernels.cuh"

namespace lob {

constexpr int kColThreads = 256;
constexpr int kSumCols = 8;    // columns of a CTA of the second pass
constexpr int kSumLanes = 32;  // partial sums per column there

// columns of one tile: at most 128, tiles of equal width
inline int col_tile(int m) {
  return (int)ceil_div(m, ceil_div(m, 128));
}

// Sum of v over the TY = kColThreads / TX threads that share column tx;
// valid in ty == 0.  red: kColThreads doubles; barriers on both sides.
__device__ __forceinline__ double col_reduce(double v, double* red, int tx, int ty, int TX,
                                             int TY) {
  red[threadIdx.x] = v;
  __syncthreads();
  double a = 0.0;
  if (ty == 0)
    for (int t = 0; t < TY; ++t) a += red[tx + t * TX];
  __syncthreads();
  return a;
}

// Fixed-order sum over blocks of partial[(z * NV + v) * m + j]: kSumCols
// columns x kSumLanes lanes per CTA; the result is valid in lane 0.
template <int NV>
__device__ __forceinline__ void sum_partials(const double* partial, int blocks, int m,
                                             int j, double (&out)[NV]) {
  __shared__ double red[NV][kSumLanes][kSumCols];
  const int tx = threadIdx.x % kSumCols, ty = threadIdx.x / kSumCols;
  double s[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) s[v] = 0.0;
  if (j < m) {
#pragma unroll 4
    for (int z = ty; z < blocks; z += kSumLanes)
#pragma unroll
      for (int v = 0; v < NV; ++v) s[v] += partial[((int64_t)z * NV + v) * m + j];
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) red[v][ty][tx] = s[v];
  for (int o = kSumLanes / 2; o > 0; o >>= 1) {
    __syncthreads();
    if (ty < o)
#pragma unroll
      for (int v = 0; v < NV; ++v) red[v][ty][tx] += red[v][ty + o][tx];
  }
#pragma unroll
  for (int v = 0; v < NV; ++v) out[v] = red[v][0][tx];
}

// out[j] = sum over blocks of partial[z * m + j]
static __global__ void __launch_bounds__(kSumCols* kSumLanes)
    colsum_finish_kernel(const double* partial, int blocks, int m, double* out) {
  chain_wait();
  const int j = blockIdx.x * kSumCols + threadIdx.x % kSumCols;
  double s[1];
  sum_partials<1>(partial, blocks, m, j, s);
  if (threadIdx.x < kSumCols && j < m) out[j] = s[0];
}

}  // namespace lob
