// FP64 reference contractions and the fused elementwise passes of one
// iteration of Algorithm 8.
//
//   gram_f64    G = U^T V (block inner products, Sec. 5.2 / Eq. 12-14): the
//               contraction over the n rows is split into row slabs, one CTA
//               per (output tile, slab); the slab partials are summed in a
//               fixed order by a second pass, so results are deterministic.
//   update_f64  Y = beta Y0 + alpha S C (Eq. 10-11): row tiles of S are
//               staged in shared memory and multiplied by C.
//   residual    r_j = AX_j - theta_j BX_j, W = K^-1 R (Jacobi) and the column
//               norms of Eq. (9), one pass over X, AX, BX.
// These run on the FP64 units; the tensor-core versions are in ozaki.cu.
#include <algorithm>
#include <type_traits>

#include "colpass.cuh"

namespace lob {

// ---------------------------------------------------------------- Gram (FP64)
//
// The FP64 contractions are bound by the FP64 pipe (two FMAs per clock and SM),
// so what counts is that no FMA is spent on padding and that every SM has a
// share: 16 x 16 threads hold NI x NJ outputs each, tiles are NI, NJ <= 4 units
// of 16 rows or columns dealt out evenly (213 columns: 4, 4, 3, 3 units and not
// 64, 64, 64, 21 columns of a 64-wide tile), and a small contraction is split
// down to 16 rows a CTA.  With 64 x 64 tiles and 256 rows a CTA the Gram of
// 1,024 x 30 x 10 took 328 us, 14 times the useful FMAs on 4 SMs.

constexpr int kU16 = 16;       // rows or columns of a tile unit
constexpr int kTileUnits = 4;  // most units of a tile
constexpr int kGK = 16;        // contraction length of a shared-memory stage

// tile t of `tiles` covers units [first, first + count) of `units`
__host__ __device__ __forceinline__ int unit_at(int t, int units, int tiles) {
  return (int)((int64_t)t * units / tiles);
}

// calls f(NI, NJ) with the counts 1 .. 4 as compile-time constants
template <int NI, typename F>
__device__ __forceinline__ void with_nj(int nj, F&& f) {
  using I = std::integral_constant<int, NI>;
  if (nj == 1) f(I(), std::integral_constant<int, 1>());
  else if (nj == 2) f(I(), std::integral_constant<int, 2>());
  else if (nj == 3) f(I(), std::integral_constant<int, 3>());
  else f(I(), std::integral_constant<int, 4>());
}
template <typename F>
__device__ __forceinline__ void with_units(int ni, int nj, F&& f) {
  if (ni == 1) with_nj<1>(nj, f);
  else if (ni == 2) with_nj<2>(nj, f);
  else if (ni == 3) with_nj<3>(nj, f);
  else with_nj<4>(nj, f);
}

struct GramF64Plan {
  int up, uq, tp, tq;  // units and tiles of p and q
  int slabs;
  int64_t rows;  // per slab
};

// One wave of four CTAs per SM, at least 16 rows each.
static GramF64Plan gram_f64_plan(int64_t n, int p, int q) {
  GramF64Plan g;
  g.up = (int)ceil_div(p, kU16);
  g.uq = (int)ceil_div(q, kU16);
  g.tp = (int)ceil_div(g.up, kTileUnits);
  g.tq = (int)ceil_div(g.uq, kTileUnits);
  const int64_t tiles = (int64_t)g.tp * g.tq;
  int64_t s = std::max<int64_t>(1, ceil_div(4 * 152, tiles));
  s = std::min<int64_t>(s, std::max<int64_t>(1, ceil_div(n, kGK)));
  g.rows = round_up(ceil_div(n, s), kGK);
  g.slabs = (int)std::max<int64_t>(1, ceil_div(n, g.rows));
  return g;
}

int64_t gram_f64_workspace(int64_t n, int p, int q) {
  if (p <= 0 || q <= 0) return 0;
  return (int64_t)gram_f64_plan(n, p, q).slabs * p * q * (int64_t)sizeof(double);
}

__global__ void __launch_bounds__(256) gram_f64_kernel(int64_t n, const __grid_constant__ SegList U,
                                                       int p, const __grid_constant__ SegList V,
                                                       int q, GramF64Plan g,
                                                       double* __restrict__ partial) {
  __shared__ double Us[kGK][kTileUnits * kU16 + 1], Vs[kGK][kTileUnits * kU16 + 1];
  const int up0 = unit_at(blockIdx.x, g.up, g.tp), uq0 = unit_at(blockIdx.y, g.uq, g.tq);
  const int tp = up0 * kU16, tq = uq0 * kU16;
  const int64_t r0 = (int64_t)blockIdx.z * g.rows, r1 = min(n, r0 + g.rows);
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  auto tile = [&](auto NIc, auto NJc) {
    constexpr int NI = decltype(NIc)::value, NJ = decltype(NJc)::value;
    // this thread loads row ty of a stage, columns tx + 16 i
    const double *pu[NI], *pv[NJ];
    int64_t ldu[NI], ldv[NJ];
    auto column = [&](const SegList& S, int c, int cols, const double** ptr, int64_t* ld) {
      if (c >= cols) {
        *ptr = nullptr;
        *ld = 0;
        return;
      }
      int k = 0;
#pragma unroll
      for (int t = 1; t < kMaxSeg; ++t) k += (t < S.nseg && c >= S.off[t]) ? 1 : 0;
      *ld = S.ld[k];
      *ptr = S.ptr[k] + (c - S.off[k]) + (r0 + ty) * S.ld[k];
    };
#pragma unroll
    for (int i = 0; i < NI; ++i) column(U, tp + tx + 16 * i, p, &pu[i], &ldu[i]);
#pragma unroll
    for (int j = 0; j < NJ; ++j) column(V, tq + tx + 16 * j, q, &pv[j], &ldv[j]);
    double ru[NI], rv[NJ];
    auto fetch = [&](int64_t r) {  // rows r .. r + 15 of the slab
      const bool in = r + ty < r1;
#pragma unroll
      for (int i = 0; i < NI; ++i) ru[i] = in && pu[i] ? __ldg(pu[i] + (r - r0) * ldu[i]) : 0.0;
#pragma unroll
      for (int j = 0; j < NJ; ++j) rv[j] = in && pv[j] ? __ldg(pv[j] + (r - r0) * ldv[j]) : 0.0;
    };
    double acc[NI][NJ];
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j) acc[i][j] = 0.0;
    fetch(r0);
    for (int64_t r = r0; r < r1; r += kGK) {
#pragma unroll
      for (int i = 0; i < NI; ++i) Us[ty][tx + 16 * i] = ru[i];
#pragma unroll
      for (int j = 0; j < NJ; ++j) Vs[ty][tx + 16 * j] = rv[j];
      __syncthreads();
      if (r + kGK < r1) fetch(r + kGK);
#pragma unroll 4
      for (int k = 0; k < kGK; ++k) {
        double a[NI], b[NJ];
#pragma unroll
        for (int i = 0; i < NI; ++i) a[i] = Us[k][ty + 16 * i];
#pragma unroll
        for (int j = 0; j < NJ; ++j) b[j] = Vs[k][tx + 16 * j];
#pragma unroll
        for (int i = 0; i < NI; ++i)
#pragma unroll
          for (int j = 0; j < NJ; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
      }
      __syncthreads();
    }
    double* out = partial + (int64_t)blockIdx.z * p * q;
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const int gi = tp + ty + 16 * i, gj = tq + tx + 16 * j;
        if (gi < p && gj < q) out[(int64_t)gi * q + gj] = acc[i][j];
      }
  };
  with_units(unit_at(blockIdx.x + 1, g.up, g.tp) - up0, unit_at(blockIdx.y + 1, g.uq, g.tq) - uq0,
             tile);
}

// G(i, j) = fixed-order sum over the slabs, 8 lanes per output (a chain of up to
// 608 dependent loads otherwise)
__global__ void __launch_bounds__(256) slab_reduce_kernel(const double* partial, int slabs, int p,
                                                          int q, double* G, int64_t ldg) {
  chain_wait();
  __shared__ double red[8][32];
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  const int64_t e = (int64_t)blockIdx.x * 32 + tx, pq = (int64_t)p * q;
  double s = 0.0;
  if (e < pq)
#pragma unroll 4
    for (int z = ty; z < slabs; z += 8) s += partial[z * pq + e];
  red[ty][tx] = s;
  __syncthreads();
  if (ty != 0 || e >= pq) return;
  for (int t = 1; t < 8; ++t) s += red[t][tx];
  G[(int)(e / q) + (int64_t)(e % q) * ldg] = s;
}

int gram_f64(cudaStream_t st, int64_t n, const SegList& U, const SegList& V, double* G,
             int64_t ldg, void* work, int64_t work_bytes) {
  const int p = U.off[U.nseg], q = V.off[V.nseg];
  if (p <= 0 || q <= 0) return LOBPCG_OK;
  const GramF64Plan g = gram_f64_plan(std::max<int64_t>(n, 1), p, q);
  int slabs = g.slabs;
  if (work_bytes < (int64_t)slabs * p * q * (int64_t)sizeof(double)) return LOBPCG_ERR_ARG;
  double* partial = (double*)work;
  if (n > 0) {
    dim3 grid((unsigned)g.tp, (unsigned)g.tq, (unsigned)slabs);
    gram_f64_kernel<<<grid, 256, 0, st>>>(n, U, p, V, q, g, partial);
    LOB_LAUNCHED();
  } else {
    slabs = 1;
    LOB_CUDA_OK(cudaMemsetAsync(partial, 0, (size_t)p * q * sizeof(double), st));
  }
  const int64_t tot = (int64_t)p * q;
  launch_chained(slab_reduce_kernel, (unsigned)ceil_div(tot, 32), 256, 0, st, partial, slabs, p, q,
                 G, ldg);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

// -------------------------------------------------------------- update (FP64)

// Tiles of NI x 16 rows (NI a launch constant) by up to four units of 16 output
// columns; stages of 16 of the s contraction columns, the next one's loads in
// flight.
template <int NI>
__global__ void __launch_bounds__(256) update_f64_kernel(int64_t n, const __grid_constant__ SegList S, int s,
                                                         const double* __restrict__ C,
                                                         int64_t ldc, int m, double alpha,
                                                         double beta, const __grid_constant__ SegList Y0,
                                                         const __grid_constant__ OutList Y,
                                                         int units, int tiles) {
  __shared__ double Ss[NI * kU16][kGK + 1], Cs[kGK][kTileUnits * kU16 + 1];
  const int64_t r0 = (int64_t)blockIdx.x * (NI * kU16);
  const int u0 = unit_at(blockIdx.y, units, tiles), c0 = u0 * kU16;
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  auto tile = [&](auto, auto NJc) {
    constexpr int NJ = decltype(NJc)::value;
    double rs[NI], rc[NJ];
    auto fetch = [&](int k0) {  // column k0 + tx of S and row k0 + tx of C
      const bool in = k0 + tx < s;
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const int64_t row = r0 + ty + 16 * i;
        rs[i] = in && row < n ? seg_load(S, k0 + tx, row) : 0.0;
      }
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const int c = c0 + ty + 16 * j;
        rc[j] = in && c < m ? C[(k0 + tx) + (int64_t)c * ldc] : 0.0;
      }
    };
    double acc[NI][NJ];
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j) acc[i][j] = 0.0;
    fetch(0);
    for (int k0 = 0; k0 < s; k0 += kGK) {
#pragma unroll
      for (int i = 0; i < NI; ++i) Ss[ty + 16 * i][tx] = rs[i];
#pragma unroll
      for (int j = 0; j < NJ; ++j) Cs[tx][ty + 16 * j] = rc[j];
      __syncthreads();
      if (k0 + kGK < s) fetch(k0 + kGK);
      const int left = min(kGK, s - k0);
#pragma unroll 4
      for (int k = 0; k < left; ++k) {
        double a[NI], b[NJ];
#pragma unroll
        for (int i = 0; i < NI; ++i) a[i] = Ss[ty + 16 * i][k];
#pragma unroll
        for (int j = 0; j < NJ; ++j) b[j] = Cs[k][tx + 16 * j];
#pragma unroll
        for (int i = 0; i < NI; ++i)
#pragma unroll
          for (int j = 0; j < NJ; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < NI; ++i)
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const int64_t row = r0 + ty + 16 * i;
        const int c = c0 + tx + 16 * j;
        if (row < n && c < m) {
          double v = alpha * acc[i][j];
          if (beta != 0.0) v = fma(beta, seg_load(Y0, c, row), v);
          *out_addr(Y, c, row) = v;
        }
      }
  };
  with_nj<NI>(unit_at(blockIdx.y + 1, units, tiles) - u0, tile);
}

int update_f64(cudaStream_t st, int64_t n, const SegList& S, const double* C, int64_t ldc,
               int m, double alpha, double beta, const SegList& Y0, const OutList& Y) {
  const int s = S.off[S.nseg];
  if (n <= 0 || m <= 0) return LOBPCG_OK;
  const int units = (int)ceil_div(m, kU16);
  // 64-row tiles of up to four units when they give every SM four CTAs, 16-row
  // tiles of one unit when not
  int tiles = (int)ceil_div(units, kTileUnits);
  const bool small = ceil_div(n, 4 * kU16) * tiles < 4 * 152;
  if (small) tiles = units;
  const dim3 grid((unsigned)ceil_div(n, (small ? 1 : 4) * kU16), (unsigned)tiles);
  if (small)
    update_f64_kernel<1><<<grid, 256, 0, st>>>(n, S, s, C, ldc, m, alpha, beta, Y0, Y, units,
                                               tiles);
  else
    update_f64_kernel<4><<<grid, 256, 0, st>>>(n, S, s, C, ldc, m, alpha, beta, Y0, Y, units,
                                               tiles);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

// ------------------------------------------------------- residual and norms

// kinv = 1 / kdiag: the preconditioner is applied as a product, because an
// FP64 division costs ~10 FP64 instructions on a part whose FP64 rate is 1/64
// of FP32 (the residual pass was bound by it)
__global__ void reciprocal_kernel(int64_t n, const double* __restrict__ d,
                                  double* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = 1.0 / d[i];
}

int reciprocal(cudaStream_t st, int64_t n, const double* d, double* out) {
  if (n <= 0) return LOBPCG_OK;
  reciprocal_kernel<<<(unsigned)ceil_div(n, 256), 256, 0, st>>>(n, d, out);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

static int row_blocks(int64_t n) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 64), 4 * 152));
}

int64_t residual_workspace(int64_t n, int m) {
  return (int64_t)row_blocks(n) * 2 * std::max(m, 1) * (int64_t)sizeof(double);
}

// One pass over X, AX (and BX): each CTA owns a contiguous row range, threads
// over the columns of a tile and TY rows, four rows in flight per thread.  Bound
// by the four FP64 operations per element (residual, two squares, the product
// with 1 / kdiag) on a part with 1/64-rate FP64: 118 us of FP64 pipe at
// n = 262,144, m = 71, against 88 us of bytes.
template <bool kB>
__global__ void __launch_bounds__(kColThreads) residual_kernel(
    int64_t n, const double* __restrict__ X, const double* __restrict__ AX,
    const double* __restrict__ BX, int64_t ld, int m, int c0, int TX,
    const double* __restrict__ theta, const double* __restrict__ kinv, double* __restrict__ W,
    int64_t ldw, int xb, double* __restrict__ partial) {
  __shared__ double red[kColThreads];
  const int mm = m - c0, TY = kColThreads / TX;
  const int64_t per = ceil_div(n, (int64_t)gridDim.x);
  const int64_t r0 = (int64_t)blockIdx.x * per, r1 = min(n, r0 + per);
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  for (int cb = 0; cb < mm; cb += TX) {
    const int jj = cb + tx, j = c0 + jj;
    const bool live = ty < TY && jj < mm;
    double rn = 0.0, xn = 0.0;
    if (live) {
      const double th = theta[j];
      auto row = [&](int64_t r, double x, double bx, double ax, double ki) {
        const double res = fma(-th, bx, ax);
        rn = fma(res, res, rn);
        xn = fma(x, xb ? bx : x, xn);  // ||x||^2, or x^T B x for criterion (8)
        if (W) W[r * ldw + jj] = kinv ? res * ki : res;
      };
      int64_t r = r0 + ty;
      for (; r + 3 * TY < r1; r += 4 * TY) {
        double x[4], bx[4], ax[4], ki[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int64_t o = (r + i * TY) * ld + j;
          x[i] = X[o];
          ax[i] = AX[o];
          bx[i] = kB ? BX[o] : x[i];
          ki[i] = kinv ? __ldg(kinv + r + i * TY) : 1.0;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) row(r + i * TY, x[i], bx[i], ax[i], ki[i]);
      }
      for (; r < r1; r += TY) {
        const int64_t o = r * ld + j;
        const double x = X[o];
        row(r, x, kB ? BX[o] : x, AX[o], kinv ? kinv[r] : 1.0);
      }
    }
    rn = col_reduce(rn, red, tx, ty, TX, TY);
    xn = col_reduce(xn, red, tx, ty, TX, TY);
    if (live && ty == 0) {
      partial[((int64_t)blockIdx.x * 2 + 0) * mm + jj] = rn;
      partial[((int64_t)blockIdx.x * 2 + 1) * mm + jj] = xn;
    }
  }
}

__global__ void __launch_bounds__(kSumCols* kSumLanes)
    residual_finish_kernel(const double* partial, int blocks, int mm, int c0, const double* theta,
                           double normA, double normB, double* be) {
  chain_wait();
  const int j = blockIdx.x * kSumCols + threadIdx.x % kSumCols;
  double s[2];
  sum_partials<2>(partial, blocks, mm, j, s);
  if (threadIdx.x < kSumCols && j < mm)
    be[j] = sqrt(s[0]) / ((normA + fabs(theta[c0 + j]) * normB) * sqrt(s[1]));
}

int residual(cudaStream_t st, int64_t n, const double* X, const double* AX, const double* BX,
             int64_t ld, int m, int c0, const double* theta, const double* kinv, double* W,
             int64_t ldw, double normA, double normB, double* be, void* partial, int xb) {
  const int mm = m - c0;
  if (mm <= 0) return LOBPCG_OK;
  const int blocks = row_blocks(n);
  const int TX = col_tile(mm);
  if (BX)
    residual_kernel<true><<<blocks, kColThreads, 0, st>>>(n, X, AX, BX, ld, m, c0, TX, theta, kinv,
                                                          W, ldw, xb, (double*)partial);
  else
    residual_kernel<false><<<blocks, kColThreads, 0, st>>>(n, X, AX, BX, ld, m, c0, TX, theta,
                                                           kinv, W, ldw, xb, (double*)partial);
  LOB_LAUNCHED();
  launch_chained(residual_finish_kernel, (unsigned)ceil_div(mm, kSumCols), kSumCols * kSumLanes, 0,
                 st, (const double*)partial, blocks, mm, c0, theta, normA, normB, be);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

// ------------------------------------------------------- column sums of squares

int64_t colsumsq_workspace(int64_t n, int m) {
  return (int64_t)row_blocks(n) * std::max(m, 1) * (int64_t)sizeof(double);
}

__global__ void __launch_bounds__(kColThreads) colsumsq_kernel(int64_t n,
                                                               const double* __restrict__ Y,
                                                               int64_t ld, int m, int TX,
                                                               double* __restrict__ partial) {
  __shared__ double red[kColThreads];
  const int TY = kColThreads / TX;
  const int64_t per = ceil_div(n, (int64_t)gridDim.x);
  const int64_t r0 = (int64_t)blockIdx.x * per, r1 = min(n, r0 + per);
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  for (int cb = 0; cb < m; cb += TX) {
    const int j = cb + tx;
    const bool live = ty < TY && j < m;
    double s = 0.0;
    if (live) {
#pragma unroll 4
      for (int64_t r = r0 + ty; r < r1; r += TY) {
        const double y = Y[r * ld + j];
        s = fma(y, y, s);
      }
    }
    s = col_reduce(s, red, tx, ty, TX, TY);
    if (live && ty == 0) partial[(int64_t)blockIdx.x * m + j] = s;
  }
}

int colsumsq(cudaStream_t st, int64_t n, const double* Y, int64_t ld, int m, double* out,
             void* partial) {
  if (m <= 0) return LOBPCG_OK;
  const int blocks = row_blocks(n);
  colsumsq_kernel<<<blocks, kColThreads, 0, st>>>(n, Y, ld, m, col_tile(m), (double*)partial);
  LOB_LAUNCHED();
  launch_chained(colsum_finish_kernel, (unsigned)ceil_div(m, kSumCols), kSumCols * kSumLanes, 0, st,
                 (const double*)partial, blocks, m, out);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

// ------------------------------------------------------------- elementwise

__global__ void diag_scale_kernel(int64_t n, int m, const double* __restrict__ b,
                                  const double* __restrict__ X, int64_t ldx,
                                  double* __restrict__ Y, int64_t ldy) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * m) return;
  const int64_t r = e / m;
  const int c = (int)(e % m);
  Y[r * ldy + c] = b[r] * X[r * ldx + c];
}

int diag_scale(cudaStream_t st, int64_t n, int m, const double* b, const double* X,
               int64_t ldx, double* Y, int64_t ldy) {
  if (n <= 0 || m <= 0) return LOBPCG_OK;
  diag_scale_kernel<<<(unsigned)ceil_div(n * m, 256), 256, 0, st>>>(n, m, b, X, ldx, Y, ldy);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

__global__ void copy_block_kernel(int64_t n, int m, const double* __restrict__ X, int64_t ldx,
                                  double* __restrict__ Y, int64_t ldy) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n * m) return;
  const int64_t r = e / m;
  const int c = (int)(e % m);
  Y[r * ldy + c] = X[r * ldx + c];
}

int copy_block(cudaStream_t st, int64_t n, int m, const double* X, int64_t ldx, double* Y,
               int64_t ldy) {
  if (n <= 0 || m <= 0) return LOBPCG_OK;
  copy_block_kernel<<<(unsigned)ceil_div(n * m, 256), 256, 0, st>>>(n, m, X, ldx, Y, ldy);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

// One block per column: find the largest |x| (lowest row on ties), flip the sign.
__global__ void __launch_bounds__(256) sign_normalise_kernel(int64_t n, double* X, int64_t ldx) {
  __shared__ double sv[256];
  __shared__ int64_t si[256];
  const int j = blockIdx.x;
  double best = -1.0;
  int64_t bi = 0;
  for (int64_t r = threadIdx.x; r < n; r += blockDim.x) {
    const double a = fabs(X[r * ldx + j]);
    if (a > best) {
      best = a;
      bi = r;
    }
  }
  sv[threadIdx.x] = best;
  si[threadIdx.x] = bi;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      const double o = sv[threadIdx.x + s];
      const int64_t oi = si[threadIdx.x + s];
      if (o > sv[threadIdx.x] || (o == sv[threadIdx.x] && oi < si[threadIdx.x])) {
        sv[threadIdx.x] = o;
        si[threadIdx.x] = oi;
      }
    }
    __syncthreads();
  }
  // decide once: a thread that flips its rows must not change the value the
  // others read
  __shared__ int flip_s;
  if (threadIdx.x == 0) flip_s = X[si[0] * ldx + j] < 0.0 ? 1 : 0;
  __syncthreads();
  const bool flip = flip_s != 0;
  if (flip)
    for (int64_t r = threadIdx.x; r < n; r += blockDim.x) X[r * ldx + j] = -X[r * ldx + j];
}

int64_t sign_normalise_workspace(int64_t, int) { return 0; }

int sign_normalise(cudaStream_t st, int64_t n, int m, double* X, int64_t ldx, void*) {
  if (n <= 0 || m <= 0) return LOBPCG_OK;
  sign_normalise_kernel<<<m, 256, 0, st>>>(n, X, ldx);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

// ------------------------------------------------------ balance exponents
// out[k] = floor(log2(G_kk) / 2), i.e. 2^out[k] is within a factor 2 of the
// column norm sqrt(G_kk) (0 for a non-positive diagonal).  Integer ops only.
__global__ void diag_exponents_kernel(int n, const double* G, int64_t ldg, int* out) {
  chain_wait();
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const long long b = __double_as_longlong(G[k + (int64_t)k * ldg]);
  const int be = (int)((b >> 52) & 0x7FF);
  int e = 0;
  if (b > 0 && be > 0 && be < 0x7FF) {
    const int u = be - 1023;
    e = (u >= 0) ? u / 2 : -((-u + 1) / 2);
  }
  out[k] = e;
}

int diag_exponents(cudaStream_t st, int n, const double* G, int64_t ldg, int* out) {
  if (n <= 0) return LOBPCG_OK;
  launch_chained(diag_exponents_kernel, (unsigned)ceil_div(n, 128), 128, 0, st, n, G, ldg, out);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

// ------------------------------------------------------------- Philox4x32-10
// Salmon et al. (SC'11): ten rounds of two 32x32->64 multiplications with the
// constants 0xD2511F53 / 0xCD9E8D57 and a Weyl key schedule 0x9E3779B9 /
// 0xBB67AE85.

__device__ __forceinline__ uint4 philox10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
  }
  return c;
}

__device__ __forceinline__ double uniform52(uint32_t a, uint32_t b) {
  const uint64_t m = ((uint64_t)(a >> 6) << 26) | (uint64_t)(b >> 6);
  return ((double)m + 0.5) * 0x1p-52;
}

__global__ void philox_normal_kernel(int64_t total, int m, uint32_t k0, uint32_t k1,
                                     uint32_t sid, double* __restrict__ Y, int64_t ldy) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t f0 = 2 * j;
  if (f0 >= total) return;
  const uint4 o = philox10(make_uint4((uint32_t)j, (uint32_t)((uint64_t)j >> 32), sid, 0u), k0, k1);
  const double u1 = uniform52(o.x, o.y), u2 = uniform52(o.z, o.w);
  const double rad = sqrt(-2.0 * log(u1));
  double sn, cs;
  sincospi(2.0 * u2, &sn, &cs);
  Y[(f0 / m) * ldy + (f0 % m)] = rad * cs;
  if (f0 + 1 < total) Y[((f0 + 1) / m) * ldy + ((f0 + 1) % m)] = rad * sn;
}

int philox_normal(cudaStream_t st, int64_t n, int m, uint64_t seed, uint32_t stream_id,
                  double* Y, int64_t ldy) {
  const int64_t total = n * m;
  if (total <= 0) return LOBPCG_OK;
  const int64_t pairs = ceil_div(total, 2);
  philox_normal_kernel<<<(unsigned)ceil_div(pairs, 256), 256, 0, st>>>(
      total, m, (uint32_t)(seed & 0xFFFFFFFFu), (uint32_t)(seed >> 32), stream_id, Y, ldy);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

}  // namespace lob

// ------------------------------------------------------------ C ABI wrappers

static bool seg_ok(const double* p, int64_t ld, int64_t cols) { return p && ld >= cols; }

LOBPCG_EXPORT int64_t lobpcg_gram_workspace(int64_t n, int64_t p, int64_t q, int mode,
                                            int slices) {
  if (n < 0 || p < 0 || q < 0) return -1;
  if (mode == LOBPCG_GEMM_OZAKI) return lob::gram_ozaki_workspace(n, (int)p, (int)q, slices);
  if (mode == LOBPCG_GEMM_OZAKI_TC)
    return std::max(lob::gram_tc_workspace(n, (int)p, (int)q),
                    lob::gram_ozaki_workspace(n, (int)p, (int)q, slices));
  return lob::gram_f64_workspace(n, (int)p, (int)q);
}

LOBPCG_EXPORT int lobpcg_gram(int64_t n, const double* U, int64_t ldu, int64_t p,
                              const double* V, int64_t ldv, int64_t q, double* G, int64_t ldg,
                              int mode, int slices, void* work, int64_t work_bytes,
                              void* stream) {
  if (n < 0 || p < 0 || q < 0 || p > (1 << 20) || q > (1 << 20)) return LOBPCG_ERR_ARG;
  if (p == 0 || q == 0) return LOBPCG_OK;
  if (!G || ldg < p || (n > 0 && (!seg_ok(U, ldu, p) || !seg_ok(V, ldv, q))))
    return LOBPCG_ERR_ARG;
  if (mode != LOBPCG_GEMM_F64 && mode != LOBPCG_GEMM_OZAKI && mode != LOBPCG_GEMM_OZAKI_TC)
    return LOBPCG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t need = lobpcg_gram_workspace(n, p, q, mode, slices);
  void* own = nullptr;
  if (!work) {
    if (lob::scratch_alloc(&own, (size_t)need, st)) return LOBPCG_ERR_OOM;
    work = own;
    work_bytes = need;
  }
  lob::SegList Us = lob::seg1(U, ldu, (int)p), Vs = lob::seg1(V, ldv, (int)q);
  int rc = mode == LOBPCG_GEMM_OZAKI_TC
               ? lob::gram_tc(st, n, Us, Vs, G, ldg, slices, work, work_bytes)
               : mode == LOBPCG_GEMM_OZAKI
                     ? lob::gram_ozaki(st, n, Us, Vs, G, ldg, slices, work, work_bytes)
                     : lob::gram_f64(st, n, Us, Vs, G, ldg, work, work_bytes);
  lob::scratch_free(own, st);
  return rc;
}

LOBPCG_EXPORT int lobpcg_wait_selftest(int32_t polls, void* stream) {
  if (polls < 1) return LOBPCG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  int* d = nullptr;
  if (cudaMalloc(&d, sizeof(int)) != cudaSuccess) return LOBPCG_ERR_OOM;
  int h = 0;
  bool ok = cudaMemsetAsync(d, 0, sizeof(int), st) == cudaSuccess &&
            lob::wait_selftest(st, polls, d) == LOBPCG_OK &&
            cudaMemcpyAsync(&h, d, sizeof(int), cudaMemcpyDeviceToHost, st) == cudaSuccess &&
            cudaStreamSynchronize(st) == cudaSuccess;
  cudaFree(d);
  if (!ok) return LOBPCG_ERR_CUDA;
  return (h & 1) ? LOBPCG_ERR_TIMEOUT : LOBPCG_OK;
}

LOBPCG_EXPORT int lobpcg_update(int64_t n, const double* S, int64_t lds, int64_t s,
                                const double* C, int64_t ldc, int64_t m, double alpha,
                                double beta, const double* Y0, int64_t ldy0, double* Y,
                                int64_t ldy, int mode, int slices, void* stream) {
  if (n < 0 || s < 0 || m < 0 || s > (1 << 20) || m > (1 << 20)) return LOBPCG_ERR_ARG;
  if (n == 0 || m == 0) return LOBPCG_OK;
  if (!Y || ldy < m || (s > 0 && (!seg_ok(S, lds, s) || !C || ldc < s))) return LOBPCG_ERR_ARG;
  if (beta != 0.0 && !seg_ok(Y0, ldy0, m)) return LOBPCG_ERR_ARG;
  if (mode != LOBPCG_GEMM_F64 && mode != LOBPCG_GEMM_OZAKI && mode != LOBPCG_GEMM_OZAKI_TC)
    return LOBPCG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  lob::SegList Ss = s > 0 ? lob::seg1(S, lds, (int)s) : lob::seg_empty();
  lob::SegList Y0s = beta != 0.0 ? lob::seg1(Y0, ldy0, (int)m) : lob::seg_empty();
  lob::OutList out{{Y, Y}, {ldy, ldy}, (int)m};
  if (mode == LOBPCG_GEMM_OZAKI || mode == LOBPCG_GEMM_OZAKI_TC) {
    const bool tc = mode == LOBPCG_GEMM_OZAKI_TC;
    const int64_t need = tc ? lob::update_tc_workspace(n, (int)s, (int)m, slices)
                            : lob::update_ozaki_workspace(n, (int)s, (int)m, slices);
    void* own = nullptr;
    if (need > 0 && lob::scratch_alloc(&own, (size_t)need, st)) return LOBPCG_ERR_OOM;
    int rc = tc ? lob::update_tc(st, n, Ss, C, ldc, (int)m, alpha, beta, Y0s, out, slices, own,
                                 need)
                : lob::update_ozaki(st, n, Ss, C, ldc, (int)m, alpha, beta, Y0s, out, slices,
                                    own, need);
    lob::scratch_free(own, st);
    return rc;
  }
  return lob::update_f64(st, n, Ss, C, ldc, (int)m, alpha, beta, Y0s, out);
}

LOBPCG_EXPORT int lobpcg_residual(int64_t n, const double* X, const double* AX,
                                  const double* BX, int64_t ld, int64_t m, int64_t c0,
                                  const double* theta, const double* kdiag, double* W,
                                  int64_t ldw, double normA, double normB, double* be,
                                  void* stream) {
  if (n <= 0 || m < 0 || c0 < 0 || c0 > m || m > (1 << 20)) return LOBPCG_ERR_ARG;
  if (c0 == m) return LOBPCG_OK;
  if (!X || !AX || ld < m || !theta || !be || (W && ldw < m - c0)) return LOBPCG_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  void* part = nullptr;
  const size_t pb = (size_t)lob::residual_workspace(n, (int)(m - c0));
  if (lob::scratch_alloc(&part, pb + (kdiag ? (size_t)n * sizeof(double) : 0), st))
    return LOBPCG_ERR_OOM;
  double* kinv = kdiag ? (double*)((char*)part + pb) : nullptr;
  int rc = kdiag ? lob::reciprocal(st, n, kdiag, kinv) : LOBPCG_OK;
  if (!rc)
    rc = lob::residual(st, n, X, AX, BX, ld, (int)m, (int)c0, theta, kinv, W, ldw, normA, normB,
                       be, part);
  lob::scratch_free(part, st);
  return rc;
}

LOBPCG_EXPORT int lobpcg_philox_normal(int64_t n, int64_t m, uint64_t seed, uint32_t stream_id,
                                       double* Y, int64_t ldy, void* stream) {
  if (n < 0 || m < 0 || (n > 0 && m > 0 && (!Y || ldy < m))) return LOBPCG_ERR_ARG;
  return lob::philox_normal((cudaStream_t)stream, n, (int)m, seed, stream_id, Y, ldy);
}
