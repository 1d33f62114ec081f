// Device-resident small dense layer for projected pencils of order n_s <= 256:
// the eigensolver, Cholesky factorisations, triangular inverses, the Householder
// QR of the C_p construction and the small GEMMs of Algorithms 2, 4, 6 and 7,
// all in this library's kernels (no cuSOLVER, no cuBLAS).
//
// GB300's FP64 units run at 1/64 of the FP32 rate (about 2 FP64 FMA per clock
// per SM), so an O(n^3) FP64 step on one SM costs milliseconds at n = 213.
// The layer is therefore built as:
//   * O(n^3) work that must be exact to FP64 (the Ogita-Aishima refinement of
//     the eigenvectors, the products forming the projected matrix and the
//     back-transformation) runs as small FP64 GEMMs spread over the whole GPU
//     (8 x 8 output tiles);
//   * the O(n^3) work that only has to be close (the first eigendecomposition
//     and the Householder QR of C_p) runs in FP32 on one CTA, then FP64
//     refinement steps (eigenvectors) or Newton-Schulz steps (QR factor)
//     restore FP64 accuracy;
//   * the only O(n^3) FP64 factorisation left is the Cholesky factor of the
//     W-block Schur complement (order n_w <= n_x), on one CTA.
// Decisions stay on the device: refinement convergence, clustering and the
// residual check write flags that the host reads once per Rayleigh-Ritz call.
#include <algorithm>
#include <cfloat>
#include <cmath>

#include "dense.cuh"

namespace lob {

namespace {

constexpr double kEps64 = 2.220446049250313e-16;  // 2^-52
constexpr int kGT = 8;                             // GEMM output tile
constexpr int kGK = 64;                            // GEMM contraction chunk
constexpr int kRefSteps = 4;                       // Ogita-Aishima steps
constexpr int kMaxRunDev = 32;                     // cluster width of the final Jacobi

#define DLAUNCH(L)                                                    \
  do {                                                                \
    ++(L).launches;                                                   \
    ++g_launches;                                                     \
    if (cudaPeekAtLastError() != cudaSuccess) return LOBPCG_ERR_CUDA; \
  } while (0)

// ------------------------------------------------------------------ GEMM
// C = alpha op(A) op(B) + beta Cin (column-major; Cin may equal C but neither
// may alias A or B).  One 8 x 8 output tile per CTA, its 256 threads being four
// interleaved slices of the contraction x 64 outputs, summed in slice order
// (deterministic); the next chunk's operands are loaded while a chunk is
// multiplied.  The tiles are small because the products are: at order 81 a
// 16 x 16 tile leaves 36 CTAs, and splitting the contraction over CTAs costs a
// fence, a counter and a second pass through L2 (5.6 us at order 81, 31 us at
// 213; 4.8 and 21 us on average now, the symmetric products among them, in a cold
// launch list; FP64 pipe at 213: 18.6 us).
// skip != nullptr: the whole launch is a no-op when *skip is non-zero.
// sym = s > 0: s products of m x m whose results are symmetric, B and C of the
// later ones m columns on; only the upper triangles are computed (half of the
// FP64 work that bounds a product of order 213) and mirrored.
// next: the update X' = X + X E of a refinement step (C = X', Cin = X).  A skipped
// one copies X, so that the steps alternate between two buffers without a copy
// kernel, and every one sets the skip flag of the next step: when this step was
// skipped or converged, or its largest correction |E_ij| was at most 1e-10 (a
// further step would change the vectors below FP64 resolution).  Ten launches
// fewer per eigendecomposition: 32 x 32 solve 27.9 -> 26.9 ms.
__global__ void __launch_bounds__(256) gemm64_kernel(int m, int n, int k, int ta, int tb,
                                                     double alpha, const double* A,
                                                     int lda, const double* B, int ldb,
                                                     double beta, const double* Cin, int ldcin,
                                                     double* C, int ldc, const int* skip, int sym,
                                                     int* next, const unsigned long long* emax) {
  chain_wait();
  __shared__ double As[kGK][kGT + 1], Bs[kGK][kGT + 1];
  __shared__ double red[3][kGT * kGT];
  const int tiles_m = (m + kGT - 1) / kGT, tile = blockIdx.x;
  int row0 = (tile % tiles_m) * kGT, col0 = (tile / tiles_m) * kGT;
  const bool off = skip && *skip;
  if (next && tile == 0 && threadIdx.x == 0)
    *next = off || __longlong_as_double((long long)*emax) <= 1e-10 ? 1 : 0;
  if (off) {
    const int row = row0 + (threadIdx.x & 7), col = col0 + (threadIdx.x >> 3);
    if (next && threadIdx.x < kGT * kGT && row < m && col < n)
      C[row + (int64_t)col * ldc] = Cin[row + (int64_t)col * ldcin];
    return;
  }
  if (sym) {  // tile number of the upper triangle of product number `which`
    const int per = tiles_m * (tiles_m + 1) / 2, which = tile / per;
    int u = tile - which * per, tj = 0;
    while (u > tj) u -= ++tj;  // column tj holds tj + 1 tiles
    row0 = u * kGT;
    col0 = tj * kGT;
    B += (int64_t)which * m * ldb;
    C += (int64_t)which * m * ldc;
    n = m;
  }
  const int t = threadIdx.x, sl = t >> 6, i = t & 7, j = (t >> 3) & 7;
  // this thread's two elements of an operand chunk
  double ra[2], rb[2];
  auto fetch = [&](int kc) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int e = t + 256 * r;
      const int ai = ta ? e >> 6 : e & 7, ak = kc + (ta ? e & 63 : e >> 3), row = row0 + ai;
      ra[r] = (row < m && ak < k) ? (ta ? A[ak + (int64_t)row * lda] : A[row + (int64_t)ak * lda])
                                  : 0.0;
      const int bj = tb ? e & 7 : e >> 6, bk = kc + (tb ? e >> 3 : e & 63), col = col0 + bj;
      rb[r] = (col < n && bk < k) ? (tb ? B[col + (int64_t)bk * ldb] : B[bk + (int64_t)col * ldb])
                                  : 0.0;
    }
  };
  double acc0 = 0.0, acc1 = 0.0;
  fetch(0);
  for (int kc = 0; kc < k; kc += kGK) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int e = t + 256 * r;
      if (ta)
        As[e & 63][e >> 6] = ra[r];
      else
        As[e >> 3][e & 7] = ra[r];
      if (tb)
        Bs[e >> 3][e & 7] = rb[r];
      else
        Bs[e & 63][e >> 6] = rb[r];
    }
    __syncthreads();
    if (kc + kGK < k) fetch(kc + kGK);
    const int left = min(kGK, k - kc);
    for (int kk = sl; kk < left; kk += 8) {
      acc0 = fma(As[kk][i], Bs[kk][j], acc0);
      acc1 = fma(As[kk + 4][i], Bs[kk + 4][j], acc1);  // zero past k
    }
    __syncthreads();
  }
  const double acc = acc0 + acc1;
  if (sl > 0) red[sl - 1][t & 63] = acc;
  __syncthreads();
  const int row = row0 + i, col = col0 + j;
  if (sl > 0 || row >= m || col >= n || (sym && row > col)) return;
  double v = alpha * (acc + red[0][t] + red[1][t] + red[2][t]);
  if (beta != 0.0) v = fma(beta, Cin[row + (int64_t)col * ldcin], v);
  C[row + (int64_t)col * ldc] = v;
  if (sym) C[col + (int64_t)row * ldc] = v;
}

// ------------------------------------------------------- FP64 Cholesky
// A = R^T R in place (upper triangle of A becomes R; the strict lower
// triangle is zeroed), n <= kCholMax, one CTA with A staged in shared memory.
// info[0] = j + 1 for the first non-positive (or non-finite) pivot j, else 0.
constexpr int kCholMax = 160;

__global__ void __launch_bounds__(256) chol64_kernel(int n, double* A, int lda, int* info) {
  chain_wait();
  extern __shared__ double sa[];  // n x n, column-major, leading dimension n
  __shared__ int s_fail;
  __shared__ double s_r, s_inv;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nw = (int)blockDim.x >> 5;
  for (int c = warp; c < n; c += nw)
    for (int r = lane; r < n; r += 32) sa[r + c * n] = r <= c ? A[r + (int64_t)c * lda] : 0.0;
  if (t == 0) s_fail = 0;
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    if (t == 0) {
      const double piv = sa[j + j * n];
      if (!(piv > 0.0) || !isfinite(piv))
        s_fail = j + 1;
      else
        s_r = sqrt(piv);
    } else if (t == 32) {  // beside the root, not after it
      s_inv = rsqrt(sa[j + j * n]);
    }
    __syncthreads();
    if (s_fail) break;
    const double rjj = s_r, inv = s_inv;
    // row j of R: r_jk = a_jk / r_jj (k >= j)
    for (int c = j + t; c < n; c += blockDim.x) sa[j + c * n] = c == j ? rjj : sa[j + c * n] * inv;
    __syncthreads();
    // trailing update of the upper triangle: a_ic -= r_ji r_jc, j < i <= c
    // (a warp per column c, lanes over rows i)
    for (int c = j + 1 + warp; c < n; c += nw) {
      const double rjc = sa[j + c * n];
      for (int i = j + 1 + lane; i <= c; i += 32) sa[i + c * n] = fma(-sa[j + i * n], rjc, sa[i + c * n]);
    }
    __syncthreads();
  }
  __syncthreads();
  for (int c = warp; c < n; c += nw)
    for (int r = lane; r < n; r += 32) A[r + (int64_t)c * lda] = r <= c ? sa[r + c * n] : 0.0;
  if (t == 0) info[0] = s_fail;
}

// X = R^-1 for an upper triangular R (n <= kCholMax), rows from the bottom:
// X(i, i) = 1 / r_ii, X(i, j) = -(sum_{k=i+1..j} r_ik X(k, j)) / r_ii; row i
// of X replaces row i of R in shared memory once all of it is computed.
// skip: no-op when *skip != 0 (the factorisation failed).
__global__ void __launch_bounds__(256) trinv64_kernel(int n, const double* R, int ldr, double* X,
                                                      int ldx, const int* skip) {
  chain_wait();
  if (skip && *skip) return;
  extern __shared__ double sm[];  // n x n: R, rows turning into X from the bottom
  __shared__ double dinv[kCholMax];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nwp = (int)blockDim.x >> 5;
  for (int c = warp; c < n; c += nwp)
    for (int i = lane; i < n; i += 32) sm[i + c * n] = i <= c ? R[i + (int64_t)c * ldr] : 0.0;
  for (int i = t; i < n; i += blockDim.x) dinv[i] = 1.0 / R[i + (int64_t)i * ldr];
  __syncthreads();
  // eight lanes per column c share its dot product (a shuffle reduction), so
  // a row costs (n - i) / 8 dependent steps instead of n - i
  // (a warp without a column left takes no part: its shuffled sums of zeros would
  // occupy the FP64 pipe all the same; order 27: 60 -> 24 us)
  const int sub = t & 7, grp = t >> 3, ngrp = (int)blockDim.x >> 3;
  for (int i = n - 1; i >= 0; --i) {
    const double inv = dinv[i];
    double val[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int h = 0; h < 5; ++h) {
      if (i + 4 * warp + h * ngrp >= n) break;
      const int c = i + grp + h * ngrp;  // uniform within each group of 8 lanes
      double sacc = 0.0;
      if (c < n && c > i)
        for (int kk = i + 1 + sub; kk <= c; kk += 8)
          sacc = fma(sm[i + kk * n], sm[kk + c * n], sacc);
      for (int o = 4; o > 0; o >>= 1) sacc += __shfl_xor_sync(0xffffffffu, sacc, o);
      val[h] = c == i ? inv : -sacc * inv;
    }
    __syncthreads();
    if (sub == 0)
#pragma unroll
      for (int h = 0; h < 5; ++h) {
        const int c = i + grp + h * ngrp;
        if (c < n) sm[i + c * n] = val[h];
      }
    __syncthreads();
  }
  for (int c = warp; c < n; c += nwp)
    for (int i = lane; i < n; i += 32) X[i + (int64_t)c * ldx] = sm[i + c * n];
}

// ------------------------------------------- FP32 tridiagonalisation
// Householder reduction of the symmetric A (FP64) to tridiagonal T = Q^T A Q
// in FP32 (the reduction of LAPACK's sytd2, lower variant): one CTA, the lower
// triangle packed in shared memory.  Outputs d (n), e (n - 1), the reflectors
// v_k (column k of V, rows k + 1 .. n - 1, v_k[k + 1] = 1) and tau (n).  For
// orders above kTridRegMax, whose matrix does not fit the registers.
__device__ __forceinline__ int pk(int n, int i, int j) {  // (i >= j) packed lower, column-major
  return j * n - (j * (j - 1)) / 2 + (i - j);
}

__global__ void __launch_bounds__(1024, 1) tridiag32_kernel(int n, const double* A, int lda,
                                                            float* d, float* e, float* V, int ldv,
                                                            float* tau) {
  chain_wait();
  extern __shared__ float P[];  // n (n + 1) / 2
  __shared__ float v[256], p[256];
  __shared__ float wpart[32];
  __shared__ float s_tau;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int j = warp; j < n; j += 32)
    for (int i = j + lane; i < n; i += 32) P[pk(n, i, j)] = (float)A[i + (int64_t)j * lda];
  __syncthreads();
  for (int k = 0; k + 2 < n; ++k) {
    const int m = n - k - 1;  // length of the reflected column x = A(k+1 .. n-1, k)
    if (warp == 0) {
      float ss = 0.f;
      for (int i = 1 + lane; i < m; i += 32) {
        const float x = P[pk(n, k + 1 + i, k)];
        ss = fmaf(x, x, ss);
      }
      for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
      const float alpha = P[pk(n, k + 1, k)];
      float tk = 0.f, beta = alpha, scale = 0.f;
      if (ss > 0.f) {
        beta = -copysignf(sqrtf(alpha * alpha + ss), alpha);
        tk = (beta - alpha) / beta;
        scale = 1.f / (alpha - beta);
      }
      for (int i = lane; i < m; i += 32) {
        const float vi = i == 0 ? 1.f : (tk != 0.f ? P[pk(n, k + 1 + i, k)] * scale : 0.f);
        v[i] = vi;
        V[(k + 1 + i) + (int64_t)k * ldv] = vi;
      }
      if (lane == 0) {
        s_tau = tk;
        d[k] = P[pk(n, k, k)];
        e[k] = beta;
        tau[k] = tk;
      }
    }
    __syncthreads();
    const float tk = s_tau;
    if (tk == 0.f) continue;  // column already reduced; no barrier needed below
    // p = tau A22 v (warp per row) and the warp partials of p^T v
    float pv = 0.f;
    for (int i = warp; i < m; i += 32) {
      float s = 0.f;
      const int gi = k + 1 + i;
      for (int j = lane; j < m; j += 32) {
        const int gj = k + 1 + j;
        const float a = gi >= gj ? P[pk(n, gi, gj)] : P[pk(n, gj, gi)];
        s = fmaf(a, v[j], s);
      }
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      s *= tk;
      if (lane == 0) p[i] = s;
      pv = fmaf(s, v[i], pv);
    }
    if (lane == 0) wpart[warp] = pv;
    __syncthreads();
    float ptv = 0.f;
    for (int w = 0; w < 32; ++w) ptv += wpart[w];
    const float K = 0.5f * tk * ptv;
    // rank-2 update A22 -= v w^T + w v^T with w = p - K v (lower part)
    for (int j = warp; j < m; j += 32) {
      const float vj = v[j], wj = p[j] - K * v[j];
      for (int i = j + lane; i < m; i += 32) {
        const float vi = v[i], wi = p[i] - K * v[i];
        const int idx = pk(n, k + 1 + i, k + 1 + j);
        P[idx] = P[idx] - (vi * wj + wi * vj);
      }
    }
    __syncthreads();
  }
  if (t == 0) {
    if (n >= 2) {
      d[n - 2] = P[pk(n, n - 2, n - 2)];
      d[n - 1] = P[pk(n, n - 1, n - 1)];
      e[n - 2] = P[pk(n, n - 1, n - 2)];
      tau[n - 2] = 0.f;
    } else {
      d[0] = P[0];
    }
    tau[n - 1] = 0.f;
  }
}

// The same reduction with the whole symmetric matrix in registers (n <= 224):
// thread (ty, tx) of 16 warps x 32 lanes holds A(ty + 16 r, tx + 32 c), so a
// warp owns complete rows, the products A v and the rank-2 update run without
// touching memory, and a step costs two barriers: one for the column that the
// owners of its elements publish, one for p = tau A v.  Every warp forms the
// reflector and p^T v for itself (a few shuffles) instead of waiting for one
// that does.  Tiles left of or above the trailing block are skipped.  Each
// element is updated by the operations of its mirror image, in their order, so
// that the matrix stays symmetric to the last bit: the reduction does not carry an
// antisymmetric part along, and with one growing from rounding 18 % of the final
// checks in 64^3 solves failed on groups too wide (12 % so: 603 and 375 of some
// 3,260 eigenproblems).  The correction is rounded by itself: two FMAs into the
// element round twice at its size, and twice as many matrices with eigenvalues
// 1e-5 apart fail the check.  Bound by the chain of a step (two reductions of five
// shuffles, a square root, two divisions, two barriers); with the matrix in shared
// memory each element cost two loads and a store per step (811 us at n = 213; 374
// us now).
constexpr int kTridRegMax = 224;

template <int NB>
struct TridiagShared {
  // xp[k & 1][i]: x_i of step k (the column being reduced) and p_i, side by
  // side so that a row's pair is one load
  float2 xp[2][32 * NB];
};

// The steps k whose next column k + 1 lies in column tile C0: tiles left of it
// and row tiles above 2 C0 are finished, and every register index is static.
template <int NB, int C0>
__device__ __forceinline__ void tridiag_phase(int n, float (&a)[2 * NB][NB], TridiagShared<NB>& sh,
                                              float* d, float* e, float* V, int ldv, float* tau) {
  constexpr int NR = 2 * NB, R0 = 2 * C0;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int kend = min(n - 2, 32 * C0 + 31);
#pragma unroll 1
  for (int k = C0 > 0 ? 32 * C0 - 1 : 0; k < kend; ++k) {
    float2* xp = sh.xp[k & 1];
    __syncthreads();  // column k is complete; p of the step before has been read
    // reflector of x(k + 1 : n): v_{k+1} = 1, v_j = x_j scale
    float vj[NB], ss = 0.f;
#pragma unroll
    for (int c = C0; c < NB; ++c) {
      const int j = tx + 32 * c;
      vj[c] = j > k ? xp[j].x : 0.f;  // rows past n are zero
      ss = fmaf(j == k + 1 ? 0.f : vj[c], vj[c], ss);
    }
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, q);
    // (approximate quotients: tau and v are formed from the same rounded values,
    // and FP64 refines the vectors)
    const float alpha = xp[k + 1].x;
    float tk = 0.f, beta = alpha, scale = 0.f;
    if (ss > 0.f) {
      beta = -copysignf(__fsqrt_rn(fmaf(alpha, alpha, ss)), alpha);
      tk = __fdividef(beta - alpha, beta);
      scale = __fdividef(1.f, alpha - beta);
    }
#pragma unroll
    for (int c = C0; c < NB; ++c) vj[c] = tx + 32 * c == k + 1 ? 1.f : vj[c] * scale;
    if (ty == 0) {
#pragma unroll
      for (int c = C0; c < NB; ++c) {
        const int j = tx + 32 * c;
        if (j > k && j < n) V[j + (int64_t)k * ldv] = vj[c];
      }
      if (tx == 0) {
        d[k] = xp[k].x;
        e[k] = beta;
        tau[k] = tk;
      }
    }
    // p_i = tau sum_j A(i, j) v_j of this warp's rows: lane sums, reduced by
    // halving (each exchange halves the values a lane carries)
    float s[16];
#pragma unroll
    for (int r = 0; r < 16; ++r) s[r] = 0.f;
#pragma unroll
    for (int c = C0; c < NB; ++c)
#pragma unroll
      for (int r = R0; r < NR; ++r) s[r] = fmaf(a[r][c], vj[c], s[r]);
#pragma unroll
    for (int h = 8; h > 0; h >>= 1) {  // lane bit 2h keeps the upper h of 2h values
      const bool up = (tx & (2 * h)) != 0;
#pragma unroll
      for (int r = 0; r < h; ++r) {
        const float send = up ? s[r] : s[r + h], keep = up ? s[r + h] : s[r];
        s[r] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * h);
      }
    }
    s[0] += __shfl_xor_sync(0xffffffffu, s[0], 1);
    if ((tx & 1) == 0 && (tx >> 1) < NR) xp[ty + 16 * (tx >> 1)].y = tk * s[0];
    __syncthreads();
    // K = tau p^T v / 2, w = p - K v, A -= v w^T + w v^T
    float wj[NB], pv = 0.f;
#pragma unroll
    for (int c = C0; c < NB; ++c) {
      wj[c] = xp[tx + 32 * c].y;
      pv = fmaf(wj[c], vj[c], pv);
    }
#pragma unroll
    for (int q = 16; q > 0; q >>= 1) pv += __shfl_xor_sync(0xffffffffu, pv, q);
    const float K = 0.5f * tk * pv;
#pragma unroll
    for (int c = C0; c < NB; ++c) wj[c] = fmaf(-K, vj[c], wj[c]);
    const bool own = tx == ((k + 1) & 31);  // column k + 1, published for the next step
    float2* xn = sh.xp[(k + 1) & 1];
#pragma unroll
    for (int r = R0; r < NR; ++r) {
      const int i = ty + 16 * r;
      const float2 xi = xp[i];
      const float vi = i == k + 1 ? 1.f : (i > k ? xi.x * scale : 0.f);
      const float wi = fmaf(-K, vi, xi.y);
#pragma unroll
      for (int c = C0; c < NB; ++c) {  // below, above and on the diagonal tile
        if (r / 2 > c)
          a[r][c] -= fmaf(vi, wj[c], wi * vj[c]);
        else if (r / 2 < c)
          a[r][c] -= fmaf(vj[c], wi, wj[c] * vi);
        else
          a[r][c] -= __fadd_rn(__fmul_rn(vi, wj[c]), __fmul_rn(wi, vj[c]));
      }
      if (own) xn[i].x = a[r][C0];
    }
  }
  if constexpr (C0 + 1 < NB) {
    // the last step above published column 32 C0 + 31; the rows of finished
    // tiles that the next phase's x no longer reads stay as they are
    tridiag_phase<NB, C0 + 1>(n, a, sh, d, e, V, ldv, tau);
  }
}

template <int NB>
__global__ void __launch_bounds__(512, 1) tridiag32_reg_kernel(int n, const double* A,
                                                               int lda, float* d, float* e,
                                                               float* V, int ldv, float* tau) {
  chain_wait();
  constexpr int NR = 2 * NB;
  __shared__ TridiagShared<NB> sh;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  float a[NR][NB];
#pragma unroll
  for (int r = 0; r < NR; ++r)
#pragma unroll
    for (int c = 0; c < NB; ++c) {
      const int i = ty + 16 * r, j = tx + 32 * c;
      a[r][c] = (i < n && j < n) ? (float)A[j + (int64_t)i * lda] : 0.f;
    }
  if (tx == 0)
#pragma unroll
    for (int r = 0; r < NR; ++r) sh.xp[0][ty + 16 * r].x = a[r][0];
  tridiag_phase<NB, 0>(n, a, sh, d, e, V, ldv, tau);
#pragma unroll
  for (int r = 0; r < NR; ++r)
#pragma unroll
    for (int c = 0; c < NB; ++c) {
      const int i = ty + 16 * r, j = tx + 32 * c;
      if (i == j && i < n && i + 2 >= n) d[i] = a[r][c];
      if (i == n - 1 && j == n - 2) e[n - 2] = a[r][c];
    }
  if (threadIdx.x < 2 && n >= 2) tau[n - 2 + threadIdx.x] = 0.f;
}

// --------------------------- tridiagonal eigenvalues and eigenvectors
// One thread per eigenvalue index j (32 per CTA): bisection on the Sturm
// count for lambda_j (FP32), then two steps of inverse iteration with T -
// lambda_j I factored by Gaussian elimination with partial pivoting (the
// method of LAPACK's stein), from a start vector hashed from j so that
// members of a tight cluster start in different directions.  Per-thread
// work arrays live in shared memory interleaved by lane.  Y(:, j) (FP32,
// n x n column-major) receives the unit eigenvector of T; lam[j] the
// eigenvalue.
__device__ __forceinline__ float hash_unit(uint32_t a, uint32_t b) {
  uint32_t h = a * 0x9E3779B1u ^ (b + 0x7F4A7C15u) * 0x85EBCA77u;
  h ^= h >> 15;
  h *= 0x2C1B3C6Du;
  h ^= h >> 12;
  h *= 0x297A2D39u;
  h ^= h >> 15;
  return (float)(h >> 8) * (1.0f / 8388608.0f) - 1.0f;  // [-1, 1)
}

// lam[j], j = 0 .. n-1: the eigenvalues of T by multisection on the Sturm
// count (count(x) = number of eigenvalues below x, LAPACK's pivmin guard), a
// warp per eigenvalue evaluating 32 interior points of the interval at once
// (each round narrows it 33-fold: five rounds to FP32 resolution), with the
// approximate division (two ulps; the values only start an iteration that FP64
// refines).  A round is a chain of n quotients, so its count is what to save:
// four points per eigenvalue and IEEE division took 204 us at n = 213; 51 us
// now.  bounds[0], bounds[1]: ||T|| bound and pivot guard for the eigenvectors.
__global__ void __launch_bounds__(256) bisect_kernel(int n, const float* dg,
                                                     const float* eg,
                                                     float* lam,
                                                     float* bounds) {
  chain_wait();
  __shared__ float d[256], e2[257];
  __shared__ float s_gl[8], s_gu[8], s_em[8];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  float gl = FLT_MAX, gu = -FLT_MAX, emax2 = 0.f;
  if (t == 0) e2[0] = 0.f;  // e2[i]: square of the entry above d[i]
  if (t < n) {
    const float di = dg[t], el = t > 0 ? eg[t - 1] : 0.f, er = t + 1 < n ? eg[t] : 0.f;
    d[t] = di;
    e2[t + 1] = er * er;
    const float r = fabsf(el) + fabsf(er);
    gl = di - r;
    gu = di + r;
    emax2 = er * er;
  }
  for (int o = 16; o > 0; o >>= 1) {
    gl = fminf(gl, __shfl_xor_sync(0xffffffffu, gl, o));
    gu = fmaxf(gu, __shfl_xor_sync(0xffffffffu, gu, o));
    emax2 = fmaxf(emax2, __shfl_xor_sync(0xffffffffu, emax2, o));
  }
  if (lane == 0) {
    s_gl[warp] = gl;
    s_gu[warp] = gu;
    s_em[warp] = emax2;
  }
  __syncthreads();
  for (int w = 0; w < 8; ++w) {
    gl = fminf(gl, s_gl[w]);
    gu = fmaxf(gu, s_gu[w]);
    emax2 = fmaxf(emax2, s_em[w]);
  }
  const float tnorm = fmaxf(fabsf(gl), fabsf(gu));
  const float pivmin = FLT_MIN * fmaxf(1.f, emax2);
  if (blockIdx.x == 0 && t == 0) {
    bounds[0] = tnorm;
    bounds[1] = pivmin;
  }
  const int g = blockIdx.x * 8 + warp;
  if (g >= n) return;
  float lo = gl - 2.f * FLT_EPSILON * tnorm * n - pivmin;
  float hi = gu + 2.f * FLT_EPSILON * tnorm * n + pivmin;
  for (int round = 0; round < 12; ++round) {
    const float wdt = hi - lo;
    if (!(wdt > 2.f * FLT_EPSILON * fmaxf(fabsf(lo), fabsf(hi)) + pivmin)) break;
    const float step = wdt * (1.f / 33.f);
    const float x = lo + (float)(lane + 1) * step;
    int c = 0;
    float q = 1.f;
#pragma unroll 4
    for (int i = 0; i < n; ++i) {
      q = d[i] - x - __fdividef(e2[i], q);
      if (fabsf(q) < pivmin) q = -pivmin;
      c += q < 0.f;
    }
    // first of the points with count > g: the eigenvalue lies below it
    const unsigned above = __ballot_sync(0xffffffffu, c > g);
    const int first = above ? __ffs(above) - 1 : 32;
    const float x0 = lo + (float)first * step, x1 = lo + (float)(first + 1) * step;
    lo = first == 0 ? lo : x0;
    hi = first == 32 ? hi : x1;
  }
  if (lane == 0) lam[g] = 0.5f * (lo + hi);
}

// Inverse iteration (two steps) for eigenvalue lam[j] of T, one thread per j
// (32 per CTA), with T - lam_j I factored by Gaussian elimination with
// partial pivoting (the method of LAPACK's stein), from a start vector hashed
// from j so that members of a tight cluster start in different directions.
// Per-thread work arrays live in shared memory interleaved by lane.  Y(:, j)
// (FP32, n x n column-major) receives the unit eigenvector of T.
// The pivots are stored as reciprocals, so the substitutions hold no division.
__global__ void __launch_bounds__(32) tridiag_eig_kernel(int n, const float* dg,
                                                         const float* eg,
                                                         const float* lam,
                                                         const float* bounds,
                                                         float* Y, int ldy) {
  chain_wait();
  extern __shared__ float ws[];  // d, e (2 n) then 6 arrays of n x 32
  float* d = ws;
  float* e = ws + n;
  float* iu = ws + 2 * n;
  float* u1 = iu + 32 * n;
  float* u2 = u1 + 32 * n;
  float* lm = u2 + 32 * n;
  float* y = lm + 32 * n;
  float* sw = y + 32 * n;  // 1: rows i and i + 1 were swapped at step i
  const int lane = threadIdx.x;
  for (int i = lane; i < n; i += 32) {
    d[i] = dg[i];
    e[i] = i + 1 < n ? eg[i] : 0.f;
  }
  __syncwarp();
  const int j = blockIdx.x * 32 + lane;
  if (j >= n) return;
  const float L = lam[j];
  // ---- LU with partial pivoting of T - L I (rows i, i + 1 may swap):
  // U has diagonal 1 / iu, superdiagonals u1, u2; multipliers in lm, swaps in sw
  const float pert = FLT_EPSILON * bounds[0] + bounds[1];
#define AT(arr, i) arr[(i) * 32 + lane]
  auto recip = [&](float u) {
    if (fabsf(u) < pert) u = u < 0.f ? -pert : pert;
    return __fdividef(1.f, u);
  };
  float diag = d[0] - L, sup = n > 1 ? e[0] : 0.f;
  for (int i = 0; i + 1 < n; ++i) {
    const float sub = e[i], nd = d[i + 1] - L, ns = i + 2 < n ? e[i + 1] : 0.f;
    const bool keep = fabsf(diag) >= fabsf(sub);
    if (keep && diag == 0.f) diag = pert;
    const float mlt = __fdividef(keep ? sub : diag, keep ? diag : sub);
    AT(lm, i) = mlt;
    AT(sw, i) = keep ? 0.f : 1.f;
    AT(iu, i) = recip(keep ? diag : sub);
    AT(u1, i) = keep ? sup : nd;
    AT(u2, i) = keep ? 0.f : ns;
    diag = keep ? nd - mlt * sup : sup - mlt * nd;
    sup = keep ? ns : -mlt * ns;
  }
  AT(iu, n - 1) = recip(diag);
  float sc = 1.f;
  for (int step = 0; step < 2; ++step) {
    // forward: apply the row operations (to the start vector, then to the
    // scaled solution of the first step)
    float yi = step == 0 ? hash_unit((uint32_t)j, 0u) : AT(y, 0) * sc;
#pragma unroll 4
    for (int i = 0; i + 1 < n; ++i) {
      const float yn = step == 0 ? hash_unit((uint32_t)j, (uint32_t)(i + 1)) : AT(y, i + 1) * sc;
      const bool swp = AT(sw, i) != 0.f;
      const float c = AT(lm, i), top = swp ? yn : yi, bot = swp ? yi : yn;
      AT(y, i) = top;
      yi = bot - c * top;
    }
    // back substitution with U
    float y1 = 0.f, y2 = 0.f, nrm = 0.f, s = yi;
#pragma unroll 4
    for (int i = n - 1; i >= 0; --i) {
      if (i + 1 < n) s = AT(y, i) - AT(u1, i) * y1;
      if (i + 2 < n) s -= AT(u2, i) * y2;
      y2 = y1;
      y1 = s * AT(iu, i);
      AT(y, i) = y1;
      nrm = fmaxf(nrm, fabsf(y1));
    }
    sc = nrm > 0.f ? 1.f / nrm : 1.f;
  }
  float s2 = 0.f;
#pragma unroll 4
  for (int i = 0; i < n; ++i) {
    const float v = AT(y, i) * sc;
    s2 = fmaf(v, v, s2);
  }
  const float inv = s2 > 0.f ? sc * rsqrtf(s2) : 0.f;
  for (int i = 0; i < n; ++i) Y[i + (int64_t)j * ldy] = AT(y, i) * inv;
#undef AT
}

// Tight clusters of the tridiagonal spectrum (consecutive eigenvalues closer
// than 1e-5 ||T||, where inverse iteration in FP32 cannot separate the
// vectors): each cluster's vectors are orthonormalised in eigenvalue order
// by modified Gram-Schmidt (one warp per cluster, clusters found by thread
// 0).  Vectors of well separated eigenvalues are left as they are.
__global__ void __launch_bounds__(1024, 1) cluster_orth_kernel(int n, const float* lam,
                                                               float* Y, int ldy) {
  chain_wait();
  __shared__ int runs[2 * 128];
  __shared__ int nruns, near;
  __shared__ float ls[256];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  // the eigenvalues are ascending: the largest magnitude is at an end
  const float thr = 1e-5f * fmaxf(fabsf(lam[0]), fabsf(lam[n - 1]));
  if (t == 0) nruns = near = 0;
  __syncthreads();
  if (t < n) {
    ls[t] = lam[t];
    if (t > 0 && lam[t] - lam[t - 1] <= thr) near = 1;
  }
  __syncthreads();
  if (!near) return;  // no cluster: the usual case ends without the serial scan
  if (t == 0) {
    int nr = 0;
    for (int a = 0; a < n;) {
      int b = a + 1;
      while (b < n && ls[b] - ls[b - 1] <= thr) ++b;
      if (b - a >= 2 && nr < 128) {
        runs[2 * nr] = a;
        runs[2 * nr + 1] = b - a;
        ++nr;
      }
      a = b;
    }
    nruns = nr;
  }
  __syncthreads();
  for (int r = warp; r < nruns; r += 32) {
    const int a = runs[2 * r], m = runs[2 * r + 1];
    for (int c = a; c < a + m; ++c) {
      float* yc = Y + (int64_t)c * ldy;
      for (int pass = 0; pass < 2; ++pass)
        for (int b = a; b < c; ++b) {
          const float* yb = Y + (int64_t)b * ldy;
          float s = 0.f;
          for (int i = lane; i < n; i += 32) s = fmaf(yb[i], yc[i], s);
          for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          for (int i = lane; i < n; i += 32) yc[i] = fmaf(-s, yb[i], yc[i]);
          __syncwarp();
        }
      float s = 0.f;
      for (int i = lane; i < n; i += 32) s = fmaf(yc[i], yc[i], s);
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      const float inv = s > 0.f ? rsqrtf(s) : 0.f;
      for (int i = lane; i < n; i += 32) yc[i] *= inv;
      __syncwarp();
    }
  }
}

// Z = Q Y with Q = H_0 H_1 ... H_{n-3}, H_k = I - tau_k v_k v_k^T: reflectors
// applied from the last to the first, each column of Y independently: a warp
// per column, the column in registers, the reflectors staged in shared memory
// (packed, strictly lower part).  Bound by the chain of a reflector (a dot
// product's five shuffles): with half a warp per column and the column in
// shared memory a reflector took a microsecond (203 us at n = 213; 53 us
// now).  Z is written in FP64.
__device__ __forceinline__ int vpk(int n, int k) {  // start of reflector k (rows k+1 .. n-1)
  return k * (n - 1) - (k * (k - 1)) / 2;
}

template <int NB>
__global__ void __launch_bounds__(256) backtransform_kernel(int n, const float* V,
                                                            int ldv, const float* tau,
                                                            const float* Y, int ldy,
                                                            double* Z, int ldz) {
  chain_wait();
  extern __shared__ float vp[];  // n (n - 1) / 2
  __shared__ float ts[256];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int k = warp; k + 1 < n; k += 8) {
    const int base = vpk(n, k), len = n - 1 - k;
    for (int i = lane; i < len; i += 32) vp[base + i] = V[(k + 1 + i) + (int64_t)k * ldv];
  }
  for (int k = t; k < n; k += blockDim.x) ts[k] = tau[k];
  const int col = blockIdx.x * 8 + warp;
  float y[NB];
#pragma unroll
  for (int c = 0; c < NB; ++c) {
    const int i = lane + 32 * c;
    y[c] = (i < n && col < n) ? Y[i + (int64_t)col * ldy] : 0.f;
  }
  __syncthreads();
  if (col >= n) return;
  for (int k = n - 3; k >= 0; --k) {
    const float tk = ts[k];
    if (tk == 0.f) continue;
    const float* v = vp + vpk(n, k) - (k + 1);  // v[i] for i = k+1 .. n-1
    float vr[NB], s = 0.f;
#pragma unroll
    for (int c = 0; c < NB; ++c) {
      const int i = lane + 32 * c;
      vr[c] = (i > k && i < n) ? v[i] : 0.f;
      s = fmaf(vr[c], y[c], s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    s *= tk;
#pragma unroll
    for (int c = 0; c < NB; ++c) y[c] = fmaf(-s, vr[c], y[c]);
  }
#pragma unroll
  for (int c = 0; c < NB; ++c) {
    const int i = lane + 32 * c;
    if (i < n) Z[i + (int64_t)col * ldz] = (double)y[c];
  }
}

// -------------------------------------------- FP64 refinement steps
// One Ogita-Aishima step from [G, S] = X^T [X, A X] (n x 2n, column-major):
// d_i = s_ii / g_ii, R = I - G, delta = 2 (||S - diag(d) G||_F + ||A||_F ||R||_F),
// E_ij = (s_ij + d_j r_ij) / (d_j - d_i) when |d_j - d_i| > delta and that
// quotient is below 1e-2 (a first-order correction), else r_ij / 2 (the pair
// is treated as a cluster: orthogonalised only); E_ii = r_ii / 2.  Sets
// done[0] when delta <= 64 n eps ||A||_F (converged: later steps skip).
// Two kernels over the whole GPU: partial norms and d, then delta and E.
constexpr int kOaBlocks = 64;

__global__ void __launch_bounds__(256) oa_norms_kernel(int n, const double* GS,
                                                       double* part,
                                                       double* dvec, const int* done) {
  chain_wait();
  if (*done) return;
  __shared__ double red[2][8];
  const double* G = GS;
  const double* S = GS + (int64_t)n * n;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  double a = 0.0, b = 0.0;
  const int64_t nn = (int64_t)n * n;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + t; e < nn; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e % n), j = (int)(e / n);
    const double g = G[e], sv = S[e];
    if (i == j) {
      const double dd = sv / g;
      dvec[i] = dd;
      a = fma(sv - dd * g, sv - dd * g, a);
      b = fma(1.0 - g, 1.0 - g, b);
    } else {
      a = fma(sv, sv, a);
      b = fma(g, g, b);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if (lane == 0) {
    red[0][warp] = a;
    red[1][warp] = b;
  }
  __syncthreads();
  if (t == 0) {
    double sa = 0.0, sb = 0.0;
    for (int w = 0; w < 8; ++w) {
      sa += red[0][w];
      sb += red[1][w];
    }
    part[2 * blockIdx.x] = sa;
    part[2 * blockIdx.x + 1] = sb;
  }
}

__global__ void __launch_bounds__(256) oa_e_kernel(int n, const double* GS,
                                                   const double* part,
                                                   const double* dvec,
                                                   const double* scal,
                                                   double* E, int* done,
                                                   double* delta_out,
                                                   unsigned long long* emax) {
  chain_wait();
  if (*done) return;
  __shared__ double s_delta;
  __shared__ unsigned long long s_max[8];
  const double* G = GS;
  const double* S = GS + (int64_t)n * n;
  if (threadIdx.x < 32) {  // fixed-order sum of the partials (every CTA alike)
    double sa = 0.0, sb = 0.0;
    for (int q = threadIdx.x; q < kOaBlocks; q += 32) {
      sa += part[2 * q];
      sb += part[2 * q + 1];
    }
    for (int o = 16; o > 0; o >>= 1) {
      sa += __shfl_xor_sync(0xffffffffu, sa, o);
      sb += __shfl_xor_sync(0xffffffffu, sb, o);
    }
    if (threadIdx.x == 0) s_delta = 2.0 * (sqrt(sa) + scal[0] * sqrt(sb));
  }
  __syncthreads();
  const double delta = s_delta;
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long m = 0;
  if (e < (int64_t)n * n) {
    const int i = (int)(e % n), j = (int)(e / n);
    const double r = (i == j ? 1.0 : 0.0) - G[e];
    double out = 0.5 * r;
    if (i != j) {
      const double di = dvec[i], dj = dvec[j];
      const double gap = dj - di, num = S[e] + dj * r;
      if (fabs(gap) > delta && fabs(num) <= 1e-2 * fabs(gap)) out = num / gap;
    }
    E[e] = out;
    m = (unsigned long long)__double_as_longlong(fabs(out));
  }
  // largest |E_ij| of the step (non-negative doubles order as their bits)
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) s_max[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long mm = 0;
    for (int w = 0; w < 8; ++w) mm = max(mm, s_max[w]);
    atomicMax(emax, mm);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    delta_out[0] = delta;
    // converged: the update of this step and every later step are skipped
    if (!(delta > 64.0 * n * kEps64 * scal[0])) done[0] = 1;
  }
}

// Final pass on S = X^T A X, G = X^T X of the refined X: order by d_i = s_ii,
// and group the sorted positions into runs: positions k < j join one run (with
// everything between them) when |s_ij| > 8 eps ||A||_F, i.e. pairs the
// first-order steps did not decouple (clusters, and pairs whose correction the
// steps' guard refused).  Outside the runs every coupling is then below
// 8 eps ||A||_F (row norms below 8 sqrt(n) eps ||A||_F), so the run blocks' FP64
// Jacobi finishes the decomposition.  Checks ||I - G||_F at rounding level,
// finite values and runs no wider than kMaxRunDev; writes the permutation, the
// runs, the eigenvalues w (ascending) and status[0] = 0 on success, else a bit
// mask (1 orthogonality, 2 wide run, 8 non-finite) and the caller falls back.
//
// The n^2 work (norm and couplings) runs over the whole GPU, a warp per column,
// with comparisons on the bit patterns: on one CTA its FP64 instructions alone
// took 80 us at n = 213 (108 us in all; 9 us now).
__device__ __forceinline__ long long order_key(double x) {  // sorts as x does (NaN at an end)
  const long long b = __double_as_longlong(x);
  return b < 0 ? (long long)(0x8000000000000000ULL - (unsigned long long)b) : b;
}

// reach[pos(i)]: furthest sorted position coupled to column i; part[i]: column
// i's share of ||I - G||_F^2; perm and w; nonfin[0] = 1 for a non-finite d_i.
__global__ void __launch_bounds__(256) eig_scan_kernel(int n, const double* GS,
                                                       const double* scal,
                                                       int* perm,
                                                       int* reach,
                                                       double* part,
                                                       double* w, int* nonfin) {
  chain_wait();
  __shared__ long long key[256];
  __shared__ int pos[256];
  const double* G = GS;
  const double* S = GS + (int64_t)n * n;
  const int t = threadIdx.x, lane = t & 31;
  double dt = 0.0;
  if (t < n) {
    dt = S[t + (int64_t)t * n];
    key[t] = order_key(dt);
  }
  __syncthreads();
  if (t < n) {  // rank of d_t (ties by index)
    int r = 0;
    const long long kt = key[t];
    for (int j = 0; j < n; ++j) r += (key[j] < kt || (key[j] == kt && j < t)) ? 1 : 0;
    pos[t] = r;
    if (blockIdx.x == 0) {
      perm[r] = t;
      w[r] = dt;
      if ((__double_as_longlong(dt) & 0x7FF0000000000000LL) == 0x7FF0000000000000LL) nonfin[0] = 1;
    }
  }
  __syncthreads();
  const int i = blockIdx.x * 8 + (t >> 5);
  if (i >= n) return;
  const long long thr = __double_as_longlong(8.0 * kEps64 * scal[0]);  // >= 0: ordered as bits
  int rmax = pos[i];
  double b = 0.0;
  for (int j = lane; j < n; j += 32) {
    const long long m = __double_as_longlong(S[j + (int64_t)i * n]) & 0x7FFFFFFFFFFFFFFFLL;
    if (j != i && m > thr) rmax = max(rmax, pos[j]);
    const double r = (i == j ? 1.0 : 0.0) - G[j + (int64_t)i * n];
    b = fma(r, r, b);
  }
  for (int o = 16; o > 0; o >>= 1) {
    rmax = max(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if (lane == 0) {
    reach[pos[i]] = rmax;
    part[i] = b;
  }
}

__global__ void __launch_bounds__(256) eig_finalize_kernel(int n, const int* reach_g,
                                                           const double* part,
                                                           int* runs,
                                                           int* nruns_out,
                                                           int* nonfin, int* status) {
  chain_wait();
  __shared__ int reach[256];
  __shared__ double red[8];
  __shared__ int coupled;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  if (t == 0) coupled = 0;
  __syncthreads();
  double b = t < n ? part[t] : 0.0;
  if (t < n) {
    reach[t] = reach_g[t];
    if (reach[t] != t) coupled = 1;
  }
  for (int o = 16; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
  if (lane == 0) red[warp] = b;
  __syncthreads();
  if (t != 0) return;
  double sb = 0.0;
  for (int q = 0; q < 8; ++q) sb += red[q];
  int bad = nonfin[0] ? 8 : 0, nr = 0;
  nonfin[0] = 0;
  if (!(sqrt(sb) <= 64.0 * n * kEps64)) bad |= 1;
  if (coupled)
    for (int k = 0; k < n;) {
      int e2 = reach[k];
      for (int j = k; j <= e2; ++j) e2 = max(e2, reach[j]);
      const int m = e2 - k + 1;
      if (m > kMaxRunDev) bad |= 2;
      if (m >= 2) {
        runs[2 * nr] = k;
        runs[2 * nr + 1] = m;
        ++nr;
      }
      k = e2 + 1;
    }
  nruns_out[0] = nr;
  status[0] = bad;
}

// Zo(:, k) = X(:, perm[k]) (column permutation into the output).
__global__ void permute_cols_dev_kernel(int n, const double* X, int ldxx,
                                        const int* perm, double* Zo,
                                        int ldo) {
  chain_wait();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)n * n) return;
  const int r = (int)(e % n), k = (int)(e / n);
  Zo[r + (int64_t)k * ldo] = X[r + (int64_t)perm[k] * ldxx];
}

// Cyclic Jacobi (Golub & Van Loan, Sec. 8.5) on the FP64 block S(perm[a + i],
// perm[a + j]) of each run [a, a + m), one CTA per run (CTAs beyond the run
// count exit), then Zo(:, a : a + m) <- Zo(:, a : a + m) Q and w(a : a + m)
// the block's eigenvalues ascending.
__global__ void __launch_bounds__(256) run_jacobi_kernel(int n, const double* GS,
                                                         const int* perm,
                                                         const int* runs,
                                                         const int* nruns,
                                                         double* Zo, int ldo,
                                                         double* w) {
  chain_wait();
  if ((int)blockIdx.x >= nruns[0]) return;
  if (runs[2 * blockIdx.x + 1] > kMaxRunDev) return;  // flagged by the finalize pass
  const double* S = GS + (int64_t)n * n;
  __shared__ double M[kMaxRunDev][kMaxRunDev + 1], Q[kMaxRunDev][kMaxRunDev + 1];
  __shared__ double ev[kMaxRunDev];
  __shared__ int order[kMaxRunDev];
  const int a = runs[2 * blockIdx.x], m = runs[2 * blockIdx.x + 1];
  const int tid = threadIdx.x, lane = tid & 31;
  for (int e = tid; e < m * m; e += blockDim.x) {
    const int i = e % m, j = e / m;
    const double sij = S[perm[a + i] + (int64_t)perm[a + j] * n];
    const double sji = S[perm[a + j] + (int64_t)perm[a + i] * n];
    M[i][j] = 0.5 * (sij + sji);
    Q[i][j] = i == j ? 1.0 : 0.0;
  }
  __syncthreads();
  if (tid < 32) {
    for (int sweep = 0; sweep < 30; ++sweep) {
      double off = 0.0, tot = 0.0;
      for (int e = lane; e < m * m; e += 32) {
        const int i = e % m, j = e / m;
        const double v = M[i][j] * M[i][j];
        tot += v;
        if (i != j) off += v;
      }
      for (int o = 16; o > 0; o >>= 1) {
        off += __shfl_xor_sync(0xffffffffu, off, o);
        tot += __shfl_xor_sync(0xffffffffu, tot, o);
      }
      if (!(off > 1e-30 * tot)) break;
      for (int pp = 0; pp < m - 1; ++pp)
        for (int qq = pp + 1; qq < m; ++qq) {
          const double apq = M[pp][qq];
          if (apq == 0.0) continue;
          const double tau = (M[qq][qq] - M[pp][pp]) / (2.0 * apq);
          const double tt = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + hypot(1.0, tau));
          const double c = 1.0 / sqrt(1.0 + tt * tt), s = tt * c;
          __syncwarp();
          for (int kk = lane; kk < m; kk += 32) {
            const double mkp = M[kk][pp], mkq = M[kk][qq];
            M[kk][pp] = c * mkp - s * mkq;
            M[kk][qq] = s * mkp + c * mkq;
            const double qkp = Q[kk][pp], qkq = Q[kk][qq];
            Q[kk][pp] = c * qkp - s * qkq;
            Q[kk][qq] = s * qkp + c * qkq;
          }
          __syncwarp();
          for (int kk = lane; kk < m; kk += 32) {
            const double mpk = M[pp][kk], mqk = M[qq][kk];
            M[pp][kk] = c * mpk - s * mqk;
            M[qq][kk] = s * mpk + c * mqk;
          }
          __syncwarp();
        }
    }
    if (lane == 0) {
      for (int i = 0; i < m; ++i) {
        ev[i] = M[i][i];
        order[i] = i;
      }
      for (int i = 1; i < m; ++i)
        for (int j = i; j > 0 && ev[order[j]] < ev[order[j - 1]]; --j) {
          const int tmp = order[j];
          order[j] = order[j - 1];
          order[j - 1] = tmp;
        }
    }
  }
  __syncthreads();
  for (int i = tid; i < m; i += blockDim.x) w[a + i] = ev[order[i]];
  for (int r = tid; r < n; r += blockDim.x) {
    double x[kMaxRunDev];
    for (int j = 0; j < m; ++j) x[j] = Zo[r + (int64_t)(a + j) * ldo];
    for (int i = 0; i < m; ++i) {
      const int c = order[i];
      double v = 0.0;
      for (int j = 0; j < m; ++j) v = fma(x[j], Q[j][c], v);
      Zo[r + (int64_t)(a + i) * ldo] = v;
    }
  }
}

// ------------------------------------------ FP32 Householder QR (C_p)
// Thin QR of the tall M (m x c, m > c, column-major FP64): Householder QR in
// FP32 on one CTA (M in shared memory), then Q (m x c) formed by applying
// the reflectors to the first c columns of the identity, written in FP64.
// Each reflector is column-wise backward stable, so the span of a column of
// M is kept to FP32 accuracy relative to that column's own norm whatever
// the other columns' norms; the caller restores FP64 orthonormality.
__global__ void __launch_bounds__(1024, 1) qr32_kernel(int m, int c, const double* M,
                                                       int ldm, double* Q, int ldq) {
  chain_wait();
  extern __shared__ float qs[];
  float* a = qs;          // m x c
  float* q = qs + m * c;  // m x c
  __shared__ float tv[256];
  __shared__ float s_tau;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int e = t; e < m * c; e += blockDim.x) {
    const int i = e % m, j = e / m;
    a[e] = (float)M[i + (int64_t)j * ldm];
    q[e] = i == j ? 1.f : 0.f;
  }
  __syncthreads();
  for (int j = 0; j < c; ++j) {
    if (warp == 0) {
      float ss = 0.f;
      for (int i = j + 1 + lane; i < m; i += 32) ss = fmaf(a[i + j * m], a[i + j * m], ss);
      for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
      const float alpha = a[j + j * m];
      float tk = 0.f, beta = alpha, scale = 0.f;
      if (ss > 0.f) {
        beta = -copysignf(sqrtf(alpha * alpha + ss), alpha);
        tk = (beta - alpha) / beta;
        scale = 1.f / (alpha - beta);
      }
      if (lane == 0) {
        s_tau = tk;
        tv[j] = tk;
      }
      __syncwarp();
      for (int i = j + 1 + lane; i < m; i += 32) a[i + j * m] = tk != 0.f ? a[i + j * m] * scale : 0.f;
      if (lane == 0) a[j + j * m] = beta;
    }
    __syncthreads();
    const float tk = s_tau;
    if (tk != 0.f) {
      // columns j + 1 .. c - 1: x -= tau v (v^T x), v = [1; a(j+1:m, j)]
      for (int cc = j + 1 + warp; cc < c; cc += 32) {
        float s = 0.f;
        for (int i = j + lane; i < m; i += 32)
          s = fmaf(i == j ? 1.f : a[i + j * m], a[i + cc * m], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        s *= tk;
        for (int i = j + lane; i < m; i += 32)
          a[i + cc * m] = fmaf(-s, i == j ? 1.f : a[i + j * m], a[i + cc * m]);
      }
    }
    __syncthreads();
  }
  // Q = H_0 ... H_{c-1} I(:, 0:c): reflectors applied from the last
  for (int j = c - 1; j >= 0; --j) {
    const float tk = tv[j];
    if (tk != 0.f)
      for (int cc = warp; cc < c; cc += 32) {
        float s = 0.f;
        for (int i = j + lane; i < m; i += 32)
          s = fmaf(i == j ? 1.f : a[i + j * m], q[i + cc * m], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        s *= tk;
        for (int i = j + lane; i < m; i += 32)
          q[i + cc * m] = fmaf(-s, i == j ? 1.f : a[i + j * m], q[i + cc * m]);
      }
    __syncthreads();
  }
  for (int e = t; e < m * c; e += blockDim.x) {
    const int i = e % m, j = e / m;
    Q[i + (int64_t)j * ldq] = (double)q[e];
  }
}

// ------------------------------------------------- small helpers
// order 1: Z = [1], w = a, status 0
__global__ void eig1_kernel(const double* A, double* Z, double* w, int* status) {
  chain_wait();
  w[0] = A[0];
  Z[0] = 1.0;
  status[0] = 0;
}

// S = (A + A^T) / 2 (n x n), with each CTA's share of ||S||_F^2
__global__ void __launch_bounds__(256) symmetrize_copy_kernel(int n, const double* A,
                                                              int lda, double* S,
                                                              int lds, double* part) {
  chain_wait();
  __shared__ double red[8];
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double v = 0.0;
  if (e < (int64_t)n * n) {
    const int i = (int)(e % n), j = (int)(e / n);
    v = 0.5 * (A[i + (int64_t)j * lda] + A[j + (int64_t)i * lda]);
    S[i + (int64_t)j * lds] = v;
  }
  v *= v;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int q = 0; q < 8; ++q) s += red[q];
    part[blockIdx.x] = s;
  }
}

// out[0] = sqrt of the sum of m partials (m <= 256, fixed order)
__global__ void __launch_bounds__(256) norm_finish_kernel(int m, const double* part,
                                                          double* out) {
  chain_wait();
  __shared__ double red[8];
  double v = threadIdx.x < m ? part[threadIdx.x] : 0.0;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int q = 0; q < 8; ++q) s += red[q];
    out[0] = sqrt(s);
  }
}

__global__ void copy_block_cm_kernel(int rows, int cols, const double* S, int lds,
                                     double* D, int ldd, double scale) {
  chain_wait();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)rows * cols) return;
  const int i = (int)(e % rows), j = (int)(e / rows);
  D[i + (int64_t)j * ldd] = scale * S[i + (int64_t)j * lds];
}

// X(i, j) *= r[i] (row scaling), optionally adding Add(i, j) for i < add_rows first
__global__ void scale_rows_add_kernel(int rows, int cols, const double* r,
                                      double* X, int ldx, const double* Add,
                                      int ldadd, int add_rows) {
  chain_wait();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)rows * cols) return;
  const int i = (int)(e % rows), j = (int)(e / rows);
  double x = X[i + (int64_t)j * ldx];
  if (Add && i < add_rows) x += Add[i + (int64_t)j * ldadd];
  X[i + (int64_t)j * ldx] = r ? r[i] * x : x;
}

// d_i = G_ii^-1/2 (0 for a zero column); MB = D GB D, MA = D GA D (both
// symmetrised).  GA may be null (only MB).
__global__ void dscale2_kernel(int n, const double* GB, int ldb,
                               const double* GA, int lda, double* d,
                               double* MB, double* MA, int ldm) {
  chain_wait();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)n * n) return;
  const int i = (int)(e % n), j = (int)(e / n);
  const double gi = GB[i + (int64_t)i * ldb], gj = GB[j + (int64_t)j * ldb];
  const double di = gi > DBL_MIN ? 1.0 / sqrt(gi) : 0.0, dj = gj > DBL_MIN ? 1.0 / sqrt(gj) : 0.0;
  if (j == 0) d[i] = di;
  MB[i + (int64_t)j * ldm] = di * (0.5 * (GB[i + (int64_t)j * ldb] + GB[j + (int64_t)i * ldb])) * dj;
  if (GA)
    MA[i + (int64_t)j * ldm] =
        di * (0.5 * (GA[i + (int64_t)j * lda] + GA[j + (int64_t)i * lda])) * dj;
}

// The congruence T1^T M T1, T1 = blkdiag(Y11, I), of the scaled explicit
// pencil (MB, MA), completed from the blocks the GEMMs wrote: SB' has the
// identity on its leading o x o block, Fb = Y11^T MB[0:o, o:] above and its
// transpose below the diagonal, MB on the trailing block; SA' has the GEMM's
// leading block, Ka[:, o:] = Y11^T MA[0:o, o:] off the diagonal and MA on the
// trailing block.  Both come out with both triangles.
__global__ void pre_fill_kernel(int ns, int o, const double* MB,
                                const double* MA, int ldm,
                                const double* Ka, int ldk, double* SB,
                                double* SA, int lds) {
  chain_wait();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)ns * ns) return;
  const int i = (int)(e % ns), j = (int)(e / ns);
  if (i < o && j < o) {  // SA' leading block comes from its GEMM
    SB[i + (int64_t)j * lds] = i == j ? 1.0 : 0.0;
  } else if (i < o) {    // SB' upper off-diagonal block comes from its GEMM
    SA[i + (int64_t)j * lds] = Ka[i + (int64_t)j * ldk];
  } else if (j < o) {
    SB[i + (int64_t)j * lds] = SB[j + (int64_t)i * lds];
    SA[i + (int64_t)j * lds] = Ka[j + (int64_t)i * ldk];
  } else {
    SB[i + (int64_t)j * lds] = MB[i + (int64_t)j * ldm];
    SA[i + (int64_t)j * lds] = MA[i + (int64_t)j * ldm];
  }
}

// C(i, j) = d_i (i < o ? Ct(i, j) : C(i, j)): the coefficients in the basis
// S back from the congruence, C = D blkdiag(Y11, I) C'.
__global__ void pre_back_kernel(int ns, int m, int o, const double* d,
                                const double* Ct, int ldt, double* C,
                                int ldc) {
  chain_wait();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)ns * m) return;
  const int i = (int)(e % ns), j = (int)(e / ns);
  const double x = i < o ? Ct[i + (int64_t)j * ldt] : C[i + (int64_t)j * ldc];
  C[i + (int64_t)j * ldc] = d[i] * x;
}

// H (ns x ns): H[0:o, 0:o] = MA[0:o, 0:o]; H[0:o, o:] = Qm[0:o, :] and its
// transpose below; H[o:, o:] is written by a GEMM.
__global__ void assemble_h_kernel(int ns, int o, const double* MA, int ldm,
                                  const double* Qm, int ldq, double* H,
                                  int ldh) {
  chain_wait();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)ns * ns) return;
  const int i = (int)(e % ns), j = (int)(e / ns);
  if (i >= o && j >= o) return;
  double v;
  if (i < o && j < o) v = MA[i + (int64_t)j * ldm];
  else if (i < o) v = Qm[i + (int64_t)(j - o) * ldq];
  else v = Qm[j + (int64_t)(i - o) * ldq];
  H[i + (int64_t)j * ldh] = v;
}

// cond(R) of R = [[I, F], [0, Rw]] (o + nw = ns; o = 0: R = Rw) from 8 power
// iterations on M = R^T R = MB and 8 on R^-1 R^-T = MB^-1, with R^-1 =
// [[I, Yt], [0, Yw]] given by its last nw columns Y (ns x nw); FP32 in shared
// memory (the value feeds an order-of-magnitude test).  One CTA for each of the
// two, side by side: out[0] and out[1] are the largest eigenvalues of M and
// M^-1, cond(R) = sqrt(out[0] out[1]) (cond_of); inf when non-finite, or when
// *skip != 0.  A chain of barriers: 20 us at ns = 81, 38 us with one CTA for both
// (32 x 32 solve 26.9 -> 24.8 ms, 48 x 40 x 36 solve 124.6 -> 119.8 ms).
__global__ void __launch_bounds__(1024, 1) cond_struct_kernel(int ns, int o, const double* MB,
                                                              int ldm, const double* Y,
                                                              int ldy, double* out, const int* skip) {
  chain_wait();
  const int which = blockIdx.x;
  if (skip && *skip) {
    if (threadIdx.x == 0) out[which] = INFINITY;
    return;
  }
  extern __shared__ float cs[];
  const int nw = ns - o;
  float* F = cs;               // o x nw: MB[0:o, o:], or Yt
  float* Bw = F + o * nw;      // nw x nw: MB[o:, o:], or Yw
  const float *Yt = F, *Yw = Bw;
  float* x = Bw + nw * nw;     // ns
  float* y = x + ns;           // ns
  float* z = y + ns;           // ns
  __shared__ float red[3][32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  for (int e = t; e < o * nw; e += blockDim.x) {
    const int i = e % o, j = e / o;
    F[e] = (float)(which ? Y[i + (int64_t)j * ldy] : MB[i + (int64_t)(o + j) * ldm]);
  }
  for (int e = t; e < nw * nw; e += blockDim.x) {
    const int i = e % nw, j = e / nw;
    Bw[e] = (float)(which ? Y[(o + i) + (int64_t)j * ldy] : MB[(o + i) + (int64_t)(o + j) * ldm]);
  }
  __syncthreads();
  auto sum3 = [&](float a, float b, float c, float& ra, float& rb, float& rc) {
    for (int q = 16; q > 0; q >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, q);
      b += __shfl_xor_sync(0xffffffffu, b, q);
      c += __shfl_xor_sync(0xffffffffu, c, q);
    }
    if (lane == 0) {
      red[0][warp] = a;
      red[1][warp] = b;
      red[2][warp] = c;
    }
    __syncthreads();
    ra = rb = rc = 0.f;
    const int nwarps = (ns + 31) / 32;  // the others hold zeros
    for (int w = 0; w < nwarps; ++w) {
      ra += red[0][w];
      rb += red[1][w];
      rc += red[2][w];
    }
    __syncthreads();
  };
  // res(i) = sum over eight lanes of part(i, lane): with a thread per row only
  // ns of the 1024 threads worked, each on a chain of ns products (an eighth more
  // time at ns = 81)
  auto apply = [&](auto part, float* res) {
    const int sub = t & 7;
    for (int i0 = 0; i0 < ns; i0 += (int)blockDim.x >> 3) {
      const int i = i0 + (t >> 3);
      float s = i < ns ? part(i, sub) : 0.f;
      s += __shfl_xor_sync(0xffffffffu, s, 1);
      s += __shfl_xor_sync(0xffffffffu, s, 2);
      s += __shfl_xor_sync(0xffffffffu, s, 4);
      if (i < ns && sub == 0) res[i] = s;
    }
    __syncthreads();
  };
  // out = MB in:  top = in_top + F in_w;  w = F^T in_top + Bw in_w
  auto mb_apply = [&](const float* in, float* res) {
    apply([&](int i, int sub) {
      float s = 0.f;
      if (i < o) {
        s = sub == 0 ? in[i] : 0.f;
        for (int j = sub; j < nw; j += 8) s = fmaf(F[i + j * o], in[o + j], s);
      } else {
        const int iw = i - o;
        for (int j = sub; j < o; j += 8) s = fmaf(F[j + iw * o], in[j], s);
        for (int j = sub; j < nw; j += 8) s = fmaf(Bw[iw + j * nw], in[o + j], s);
      }
      return s;
    }, res);
  };
  // res = R^-T in: top = in_top; w = Yt^T in_top + Yw^T in_w
  auto rit_apply = [&](const float* in, float* res) {
    apply([&](int i, int sub) {
      if (i < o) return sub == 0 ? in[i] : 0.f;
      const int iw = i - o;
      float s = 0.f;
      for (int j = sub; j < o; j += 8) s = fmaf(Yt[j + iw * o], in[j], s);
      for (int j = sub; j < nw; j += 8) s = fmaf(Yw[j + iw * nw], in[o + j], s);
      return s;
    }, res);
  };
  // res = R^-1 in: top = in_top + Yt in_w; w = Yw in_w
  auto ri_apply = [&](const float* in, float* res) {
    apply([&](int i, int sub) {
      float s = 0.f;
      if (i < o) {
        s = sub == 0 ? in[i] : 0.f;
        for (int j = sub; j < nw; j += 8) s = fmaf(Yt[i + j * o], in[o + j], s);
      } else {
        const int iw = i - o;
        for (int j = sub; j < nw; j += 8) s = fmaf(Yw[iw + j * nw], in[o + j], s);
      }
      return s;
    }, res);
  };
  auto power = [&]() -> float {
    for (int i = t; i < ns; i += blockDim.x) x[i] = 1.0f + 0.001f * (float)(i % 7);
    __syncthreads();
    float lam = 0.f;
    for (int it = 0; it < 8; ++it) {
      float* res = y;
      if (which == 0) {
        mb_apply(x, y);
      } else {
        rit_apply(x, y);
        ri_apply(y, z);
        res = z;
      }
      float a = 0.f, b = 0.f, c = 0.f;
      for (int i = t; i < ns; i += blockDim.x) {
        a += x[i] * res[i];
        b += res[i] * res[i];
        c += x[i] * x[i];
      }
      float xy, yy, xx;
      sum3(a, b, c, xy, yy, xx);
      if (!(yy > 0.f) || !isfinite(yy)) return INFINITY;
      if (xx > 0.f) lam = fmaxf(lam, xy / xx);
      const float inv = rsqrtf(yy);
      for (int i = t; i < ns; i += blockDim.x) x[i] = res[i] * inv;
      __syncthreads();
    }
    return lam;
  };
  const float lmax = power();
  if (t == 0) out[which] = isfinite(lmax) && lmax > 0.f ? (double)lmax : INFINITY;
}

// Q2(i, j) = th[i] * Q(i, j)
__global__ void scale_rows_by_kernel(int rows, int cols, const double* th,
                                     const double* Q, int ldq, double* Q2,
                                     int ldq2) {
  chain_wait();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)rows * cols) return;
  const int i = (int)(e % rows), j = (int)(e / rows);
  Q2[i + (int64_t)j * ldq2] = th[i] * Q[i + (int64_t)j * ldq];
}

// svqb / svqbDrop transform (Algorithms 4, 6) from the eigenpairs (w ascending,
// Z) of D G D: keep J = {j : w_j > tau max|w|} (drop) or all with w clamped
// at tau max|w| (replace); T(:, t) = d .* Z(:, first + t) / sqrt(w); nkeep[0]
// is the kept count.  One CTA computes the split, all threads fill T.
__global__ void svqb_dev_kernel(int nu, const double* w, const double* d,
                                const double* Z, int ldz, int drop, double tau,
                                double* T, int ldt, int* nkeep) {
  chain_wait();
  __shared__ int s_first;
  __shared__ double s_floor;
  if (threadIdx.x == 0) {
    double mx = 0.0;
    for (int i = 0; i < nu; ++i) mx = fmax(mx, fabs(w[i]));
    int first = 0;
    double floor_ = -INFINITY;
    if (!(mx > 0.0)) {
      first = nu;
    } else if (drop) {
      while (first < nu && !(w[first] > tau * mx)) ++first;
    } else {
      floor_ = tau * mx;
    }
    s_first = first;
    s_floor = floor_;
    nkeep[0] = nu - first;
  }
  __syncthreads();
  const int first = s_first, keep = nu - first;
  for (int e = threadIdx.x; e < nu * keep; e += blockDim.x) {
    const int i = e % nu, c = e / nu;
    const double th = fmax(w[first + c], s_floor);
    T[i + (int64_t)c * ldt] = d[i] * Z[i + (int64_t)(first + c) * ldz] / sqrt(th);
  }
}

// D = diag(w[0:n]) (n x n, leading dimension ldd)
__global__ void diag_matrix_kernel(int n, const double* w, double* D,
                                   int ldd) {
  chain_wait();
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)n * n) return;
  const int i = (int)(e % n), j = (int)(e / n);
  D[i + (int64_t)j * ldd] = i == j ? w[i] : 0.0;
}

unsigned nblk(int64_t total) { return (unsigned)std::max<int64_t>(1, ceil_div(total, 256)); }

}  // namespace

// ==================================================================== host

size_t DevDense::carve(int64_t nmax_, char* base, size_t* clear_bytes) {
  const int nm = (int)std::min<int64_t>(nmax_, kDevDenseMax);
  const size_t nn = (size_t)nm * nm;
  size_t at = 0;
  auto take = [&](size_t bytes) {
    char* p = base ? base + at : nullptr;
    at += (bytes + 255) / 256 * 256;
    return (void*)p;
  };
  int* in = (int*)take((5 * (size_t)nm + 64) * sizeof(int));
  if (clear_bytes) *clear_bytes = at;
  double* m[7];
  for (double*& p : m) p = (double*)take(nn * sizeof(double));
  double* xa = (double*)take(2 * nn * sizeof(double));  // [X | A X]
  double* xb = (double*)take(2 * nn * sizeof(double));  // the same of the other steps
  double* gs = (double*)take(2 * nn * sizeof(double));  // [G | S]
  float* v32 = (float*)take(nn * sizeof(float));
  float* y32 = (float*)take(nn * sizeof(float));
  float* fv = (float*)take(4 * (size_t)nm * sizeof(float));
  double* ve = (double*)take((8 * (size_t)nm + 256) * sizeof(double));
  double* sc = (double*)take(16 * sizeof(double));
  if (base) {
    nmax = nm;
    ints = in;
    X = m[0]; E = m[1]; Zt = m[2];
    T1 = m[3]; T2 = m[4]; T3 = m[5]; T4 = m[6];
    XA = xa; XB = xb; GS = gs; V32 = v32; Y32 = y32; f32v = fv; vec = ve; scal = sc;
  }
  return at;
}

int DevDense::init(int64_t nmax_) {
  size_t clear = 0;
  const size_t bytes = carve(nmax_, nullptr, &clear);
  void* p = nullptr;
  if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    return LOBPCG_ERR_OOM;
  }
  bufs.push_back(p);
  carve(nmax_, (char*)p, nullptr);
  if (cudaMemset(p, 0, clear) != cudaSuccess) return LOBPCG_ERR_CUDA;
  if (cudaDeviceSynchronize() != cudaSuccess) return LOBPCG_ERR_CUDA;
  return LOBPCG_OK;
}

void DevDense::release() {
  for (void* p : bufs) cudaFree(p);
  bufs.clear();
  nmax = 0;
}

int dev_gemm(DenseLayer& L, bool ta, bool tb, int m, int n, int k, double alpha, const double* A,
             int lda, const double* B, int ldb, double beta, const double* Cin, int ldcin,
             double* C, int ldc, const int* skip, int sym, int* next,
             const unsigned long long* emax) {
  if (m <= 0 || n <= 0) return LOBPCG_OK;
  const int tm = (int)ceil_div(m, kGT);
  const int tiles = sym ? sym * tm * (tm + 1) / 2 : tm * (int)ceil_div(n, kGT);
  if (!Cin) {
    Cin = C;
    ldcin = ldc;
  }
  launch_chained(gemm64_kernel, (unsigned)tiles, 256, 0, L.st, m, n, k, ta ? 1 : 0, tb ? 1 : 0,
                 alpha, A, lda, B, ldb, beta, Cin, ldcin, C, ldc, skip, sym, next, emax);
  DLAUNCH(L);
  return LOBPCG_OK;
}

int dev_chol(DenseLayer& L, int n, double* A, int lda, int* info) {
  if (n > kCholMax) return LOBPCG_ERR_ARG;
  const size_t sh = (size_t)n * n * sizeof(double);
  static bool configured[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    LOB_CUDA_OK(cudaFuncSetAttribute(chol64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kCholMax * kCholMax * 8));
    LOB_CUDA_OK(cudaFuncSetAttribute(trinv64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kCholMax * kCholMax * 8));
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  launch_chained(chol64_kernel, 1, 256, sh, L.st, n, A, lda, info);
  DLAUNCH(L);
  return LOBPCG_OK;
}

int dev_trinv(DenseLayer& L, int n, const double* R, int ldr, double* X, int ldx, const int* skip) {
  if (n > kCholMax) return LOBPCG_ERR_ARG;
  launch_chained(trinv64_kernel, 1, 256, (size_t)n * n * sizeof(double), L.st, n, R, ldr, X, ldx,
                 skip);
  DLAUNCH(L);
  return LOBPCG_OK;
}

// Eigendecomposition of the symmetric n x n FP64 matrix A (column-major, not
// modified): Z (n x n, ldz) orthonormal eigenvectors, w ascending; status
// (device int) 0 on success, 1 when the refinement's check failed (the caller
// falls back).  n <= kDevDenseMax.
int dev_syev(DenseLayer& L, int n, const double* A, int lda, double* Z, int ldz, double* w,
             int* status) {
  DevDense& D = L.dev;
  if (n > D.nmax || n > kDevDenseMax) return LOBPCG_ERR_ARG;
  int dev = 0;
  cudaGetDevice(&dev);
  static bool configured[64] = {false};
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    LOB_CUDA_OK(cudaFuncSetAttribute(tridiag32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     kDevDenseMax * (kDevDenseMax + 1) / 2 * 4));
    LOB_CUDA_OK(cudaFuncSetAttribute(tridiag_eig_kernel,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (2 * kDevDenseMax + 6 * 32 * kDevDenseMax) * 4));
    constexpr int vbytes = kDevDenseMax * (kDevDenseMax - 1) / 2 * 4;
    const void* bt[8] = {(const void*)backtransform_kernel<1>, (const void*)backtransform_kernel<2>,
                         (const void*)backtransform_kernel<3>, (const void*)backtransform_kernel<4>,
                         (const void*)backtransform_kernel<5>, (const void*)backtransform_kernel<6>,
                         (const void*)backtransform_kernel<7>, (const void*)backtransform_kernel<8>};
    for (const void* f : bt)
      LOB_CUDA_OK(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, vbytes));
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  if (n == 1) {
    launch_chained(eig1_kernel, 1, 1, 0, L.st, A, Z, w, status);
    DLAUNCH(L);
    return LOBPCG_OK;
  }
  float* d32 = D.f32v;
  float* e32 = D.f32v + D.nmax;
  float* tau32 = D.f32v + 2 * D.nmax;
  float* lam32 = D.f32v + 3 * D.nmax;
  double* normA = D.scal;  // scal[0] = ||A||_F
  // the refinement multiplies by the symmetric part of A (a projected
  // matrix formed by products is symmetric only to rounding)
  // (its norm partials lie where the refinement's vectors will)
  launch_chained(symmetrize_copy_kernel, nblk((int64_t)n * n), 256, 0, L.st, n, A, lda, D.Zt, n,
                 D.vec);
  DLAUNCH(L);
  launch_chained(norm_finish_kernel, 1, 256, 0, L.st, (int)nblk((int64_t)n * n), D.vec, normA);
  DLAUNCH(L);
  A = D.Zt;
  lda = n;
  const int nb = (int)ceil_div(n, 32);
  float* bounds = reinterpret_cast<float*>(D.scal + 8);
  auto tridiag = [&](auto* kernel) {
    launch_chained(kernel, 1, 512, 0, L.st, n, A, lda, d32, e32, D.V32, n, tau32);
  };
  if (n > kTridRegMax)
    launch_chained(tridiag32_kernel, 1, 1024, (size_t)n * (n + 1) / 2 * 4, L.st, n, A, lda, d32,
                   e32, D.V32, n, tau32);
  else if (nb == 1) tridiag(tridiag32_reg_kernel<1>);
  else if (nb == 2) tridiag(tridiag32_reg_kernel<2>);
  else if (nb == 3) tridiag(tridiag32_reg_kernel<3>);
  else if (nb == 4) tridiag(tridiag32_reg_kernel<4>);
  else if (nb == 5) tridiag(tridiag32_reg_kernel<5>);
  else if (nb == 6) tridiag(tridiag32_reg_kernel<6>);
  else tridiag(tridiag32_reg_kernel<7>);
  DLAUNCH(L);
  launch_chained(bisect_kernel, (unsigned)ceil_div(n, 8), 256, 0, L.st, n, d32, e32, lam32, bounds);
  DLAUNCH(L);
  launch_chained(tridiag_eig_kernel, (unsigned)ceil_div(n, 32), 32,
                 (size_t)(2 * n + 6 * 32 * n) * 4, L.st, n, d32, e32, lam32, bounds, D.Y32, n);
  DLAUNCH(L);
  launch_chained(cluster_orth_kernel, 1, 1024, 0, L.st, n, lam32, D.Y32, n);
  DLAUNCH(L);
  // X (first n columns of XA) = Q Y
  double* X = D.XA;
  auto back = [&](auto* kernel) {
    launch_chained(kernel, (unsigned)ceil_div(n, 8), 256, (size_t)(n * (n - 1)) / 2 * 4, L.st, n,
                   D.V32, n, tau32, D.Y32, n, X, n);
  };
  switch (nb) {
    case 1: back(backtransform_kernel<1>); break;
    case 2: back(backtransform_kernel<2>); break;
    case 3: back(backtransform_kernel<3>); break;
    case 4: back(backtransform_kernel<4>); break;
    case 5: back(backtransform_kernel<5>); break;
    case 6: back(backtransform_kernel<6>); break;
    case 7: back(backtransform_kernel<7>); break;
    default: back(backtransform_kernel<8>); break;
  }
  DLAUNCH(L);
  return dev_syev_refine(L, n, Z, ldz, w, status, kRefSteps);
}

// Refinement of the current X (first block of D.XA) against the symmetric A
// kept in D.Zt: `steps` Ogita-Aishima steps, two Newton-Schulz steps, the
// final products, the finalize pass, the permutation into Z and Jacobi on
// the coupled runs.  Also the second chance after a failed check: more
// steps from where the first call stopped.
int dev_syev_refine(DenseLayer& L, int n, double* Z, int ldz, double* w, int* status, int steps) {
  DevDense& D = L.dev;
  const double* A = D.Zt;
  const int lda = n;
  double* normA = D.scal;
  double* delta = D.scal + 1;
  int* perm = D.ints + 4;
  int* runs = perm + D.nmax;
  int* nruns = runs + 2 * D.nmax;
  // skip flags of the steps (flag[s] for step s) and the largest correction
  // of each step
  if (steps > 16) return LOBPCG_ERR_ARG;
  int* flag = D.ints + 4 * D.nmax + 24;
  // (D.vec: the norm partials at 0 .. 127, d at 128 .. 128 + n, then these)
  unsigned long long* emax = reinterpret_cast<unsigned long long*>(D.vec + 136 + D.nmax);
  // X and A X side by side; each step and each product below writes the next X
  // into the other buffer (six in the first call: its X ends in D.XA, where a
  // second call starts)
  const size_t nn = (size_t)n * n;
  double *X = D.XA, *Y = D.XB;
  double* G = D.GS;
  LOB_CUDA_OK(cudaMemsetAsync(flag, 0, (steps + 1) * sizeof(int), L.st));
  LOB_CUDA_OK(cudaMemsetAsync(emax, 0, steps * sizeof(unsigned long long), L.st));
  int rc;
  for (int s = 0; s < steps; ++s) {
    int* done = flag + s;
    // [G, S] = X^T [X, A X]
    if ((rc = dev_gemm(L, false, false, n, n, n, 1.0, A, lda, X, n, 0.0, nullptr, 0, X + nn, n,
                       done)))
      return rc;
    if ((rc = dev_gemm(L, true, false, n, 2 * n, n, 1.0, X, n, X, n, 0.0, nullptr, 0, G, n, done,
                       2)))
      return rc;
    launch_chained(oa_norms_kernel, kOaBlocks, 256, 0, L.st, n, D.GS, D.vec, D.vec + 2 * kOaBlocks,
                   done);
    DLAUNCH(L);
    launch_chained(oa_e_kernel, nblk((int64_t)n * n), 256, 0, L.st, n, D.GS, D.vec,
                   D.vec + 2 * kOaBlocks, normA, D.E, done, delta, emax + s);
    DLAUNCH(L);
    // X + X E; the next step's flag
    if ((rc = dev_gemm(L, false, false, n, n, n, 1.0, X, n, D.E, n, 1.0, X, n, Y, n, done, 0,
                       flag + s + 1, emax + s)))
      return rc;
    std::swap(X, Y);
  }
  // two Newton-Schulz steps X = X (3/2 I - 1/2 X^T X), always: I + E is orthogonal
  // to first order only (S and G are mirrored, so E_ij + E_ji = r_ij), and the last
  // step that ran leaves a defect of order E^T E, up to ~1e-4 on pairs it has just
  // separated (|E_ij| <= 1e-2); each Newton-Schulz step squares it
  for (int s = 0; s < 2; ++s) {
    if ((rc = dev_gemm(L, true, false, n, n, n, 1.0, X, n, X, n, 0.0, nullptr, 0, G, n, nullptr,
                       1)))
      return rc;
    if ((rc = dev_gemm(L, false, false, n, n, n, -0.5, X, n, G, n, 1.5, X, n, Y, n, nullptr)))
      return rc;
    std::swap(X, Y);
  }
  // final [G, S] = X^T [X, A X]
  if ((rc = dev_gemm(L, false, false, n, n, n, 1.0, A, lda, X, n, 0.0, nullptr, 0, X + nn, n,
                     nullptr)))
    return rc;
  if ((rc = dev_gemm(L, true, false, n, 2 * n, n, 1.0, X, n, X, n, 0.0, nullptr, 0, G, n, nullptr,
                     2)))
    return rc;
  int* nonfin = D.ints + 4 * D.nmax + 60;
  int* reach = D.ints + 4 * D.nmax + 64;
  launch_chained(eig_scan_kernel, (unsigned)ceil_div(n, 8), 256, 0, L.st, n, D.GS, normA, perm,
                 reach, D.vec, w, nonfin);
  DLAUNCH(L);
  launch_chained(eig_finalize_kernel, 1, 256, 0, L.st, n, reach, D.vec, runs, nruns, nonfin,
                 status);
  DLAUNCH(L);
  launch_chained(permute_cols_dev_kernel, nblk((int64_t)n * n), 256, 0, L.st, n, X, n, perm, Z,
                 ldz);
  DLAUNCH(L);
  launch_chained(run_jacobi_kernel, (unsigned)std::max(1, n / 2), 256, 0, L.st, n, D.GS, perm, runs,
                 nruns, Z, ldz, w);
  DLAUNCH(L);
  return LOBPCG_OK;
}

// Thin orthonormal basis of the span of the tall M (m x c, m > c) into Q
// (m x c, ldq): FP32 Householder QR, then two FP64 Newton-Schulz steps.
int dev_orth_basis(DenseLayer& L, int m, int c, const double* M, int ldm, double* Q, int ldq) {
  DevDense& D = L.dev;
  static bool configured[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    LOB_CUDA_OK(cudaFuncSetAttribute(qr32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     200 * 1024));
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  const size_t sh = 2 * (size_t)m * c * sizeof(float);
  if (sh > 200 * 1024 || c > 256) return LOBPCG_ERR_ARG;
  launch_chained(qr32_kernel, 1, 1024, sh, L.st, m, c, M, ldm, Q, ldq);
  DLAUNCH(L);
  int rc;
  for (int s = 0; s < 2; ++s) {
    if ((rc = dev_gemm(L, true, false, c, c, m, 1.0, Q, ldq, Q, ldq, 0.0, nullptr, 0, D.T4, c,
                       nullptr)))
      return rc;
    if ((rc = dev_gemm(L, false, false, m, c, c, -0.5, Q, ldq, D.T4, c, 1.5, Q, ldq, D.T3, m,
                       nullptr)))
      return rc;
    launch_chained(copy_block_cm_kernel, nblk((int64_t)m * c), 256, 0, L.st, m, c, D.T3, m, Q, ldq,
                   1.0);
    DLAUNCH(L);
  }
  return LOBPCG_OK;
}

// --------------------------------------------- Rayleigh-Ritz, device path

// The device path takes a projected pencil when every piece fits its
// one-CTA kernels: order <= 256 (eigensolver), Cholesky factors of order
// <= 160, the cond(R) estimate's FP32 copies and the C_p QR in shared memory.
// (The cond(R) bound counts the matrices of both estimates, which one CTA once
// held: pencils of n_s = 2 n_x, n_x > 112, stay on cuSOLVER, not measured here.)
bool dev_rr_fits(const DenseLayer& L, int ns, int nx, int nw) {
  if (L.eig_mode != 0 || ns > L.dev.nmax || ns > kDevDenseMax) return false;
  if (nw > kCholMax || nx > kCholMax) return false;
  const int o = ns - nw;
  const size_t cond_sh = (size_t)(2 * o * nw + 2 * nw * nw + 3 * ns) * 4;
  const size_t qr_sh = 2 * (size_t)(ns - nx) * nx * 4;
  return cond_sh <= 200 * 1024 && qr_sh <= 200 * 1024;
}

int syevd_fallback(DenseLayer& L, int n, double* A, int lda) {
  ++L.dev_fallbacks;
  if (cusolverDnDsyevd(L.sol, CUSOLVER_EIG_MODE_VECTOR, CUBLAS_FILL_MODE_LOWER, n, A, lda, L.ev,
                       L.work, L.lwork, L.info) != CUSOLVER_STATUS_SUCCESS)
    return LOBPCG_ERR_CUDA;
  return LOBPCG_OK;
}

namespace {

int configure_cond(DenseLayer& L) {
  static bool configured[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    LOB_CUDA_OK(cudaFuncSetAttribute(cond_struct_kernel,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  (void)L;
  return LOBPCG_OK;
}

// read n_ints device ints (from ints) and n_dbl device doubles (from dbl) in
// one host wait
int read_flags(DenseLayer& L, const int* ints, int n_ints, const double* dbl, int n_dbl,
               int* ih, double* dh) {
  if (n_ints) LOB_CUDA_OK(cudaMemcpyAsync(L.host, ints, n_ints * sizeof(int), cudaMemcpyDeviceToHost, L.st));
  if (n_dbl)
    LOB_CUDA_OK(cudaMemcpyAsync(L.host + 8, dbl, n_dbl * sizeof(double), cudaMemcpyDeviceToHost, L.st));
  LOB_CUDA_OK(cudaStreamSynchronize(L.st));
  ++L.syncs;
  if (n_ints) memcpy(ih, L.host, n_ints * sizeof(int));
  if (n_dbl) memcpy(dh, L.host + 8, n_dbl * sizeof(double));
  return LOBPCG_OK;
}

// cond(R) from the two results of cond_struct_kernel
double cond_of(const double* cr) {
  return std::isfinite(cr[0]) && std::isfinite(cr[1]) ? std::sqrt(cr[0] * cr[1]) : INFINITY;
}

// count the reasons of a failed check of the device eigensolver
void note_check(DenseLayer& L, int mask) {
  if (mask & 1) ++L.check_fail[0];
  if (mask & 2) ++L.check_fail[1];
  if (mask & 8) ++L.check_fail[2];
}

// Eigenvectors Z of H (order n) with eigenvalues in L.ev: device eigensolver,
// its status read back with the other flags by the caller.
int eig_into(DenseLayer& L, int n, const double* H, double* Z, int* status) {
  ++L.dev_calls;
  return dev_syev(L, n, H, n, Z, n, L.ev, status);
}

// After a failed check: when only the coupled groups were too wide, three
// more refinement steps from where the first call stopped (one more host
// read); otherwise, or when that fails too, cuSOLVER on a copy of H.
int eig_recover(DenseLayer& L, int n, const double* H, double* Z, int mask) {
  int rc;
  if (mask == 2) {
    int* est = L.dev.ints + 2;
    if ((rc = dev_syev_refine(L, n, Z, n, L.ev, est, 3))) return rc;
    int fl = 0;
    LOB_CUDA_OK(cudaMemcpyAsync(L.host, est, sizeof(int), cudaMemcpyDeviceToHost, L.st));
    LOB_CUDA_OK(cudaStreamSynchronize(L.st));
    ++L.syncs;
    memcpy(&fl, L.host, sizeof(int));
    if (fl == 0) return LOBPCG_OK;
    note_check(L, fl);
  }
  launch_chained(copy_block_cm_kernel, nblk((int64_t)n * n), 256, 0, L.st, n, n, H, n, Z, n, 1.0);
  DLAUNCH(L);
  return syevd_fallback(L, n, Z, n);
}


// C = [C_x, C_p] and the next P^T A P from T Z (ns x ns), Z and the
// eigenvalues L.ev (Algorithm 7, the LQ-based C_p of Sec. 4.2 restricted to
// the unlocked columns; an orthonormal basis of the span of
// M = Z_1perp^T Z_1(:, nc:nx) replaces the Householder Q of its LQ).
int rr_tail(DenseLayer& L, const double* TZ, const double* Z, int ns, int nx, int nc, double* C,
            int* npn_out, double* theta, double* PAP) {
  DevDense& D = L.dev;
  const int mrow = ns - nx, mcol = nx - nc;
  const int npn = std::min(mrow, mcol);
  int rc;
  launch_chained(copy_block_cm_kernel, nblk((int64_t)ns * nx), 256, 0, L.st, ns, nx, TZ, ns, C, ns,
                 1.0);
  DLAUNCH(L);
  if (npn > 0) {
    if (mcol >= mrow) {  // M spans the whole (ns - nx)-dimensional space: Q = I
      launch_chained(copy_block_cm_kernel, nblk((int64_t)ns * mrow), 256, 0, L.st, ns, mrow,
                     TZ + (int64_t)nx * ns, ns, C + (int64_t)nx * ns, ns, 1.0);
      DLAUNCH(L);
      launch_chained(diag_matrix_kernel, nblk((int64_t)npn * npn), 256, 0, L.st, npn, L.ev + nx,
                     PAP, npn);
      DLAUNCH(L);
    } else {
      double* M = D.Zt;
      double* Q = D.E;
      double* Q2 = D.X;
      if ((rc = dev_gemm(L, true, false, mrow, mcol, nx, 1.0, Z + (int64_t)nx * ns, ns,
                         Z + (int64_t)nc * ns, ns, 0.0, nullptr, 0, M, mrow, nullptr)))
        return rc;
      if ((rc = dev_orth_basis(L, mrow, mcol, M, mrow, Q, mrow))) return rc;
      if ((rc = dev_gemm(L, false, false, ns, mcol, mrow, 1.0, TZ + (int64_t)nx * ns, ns, Q, mrow,
                         0.0, nullptr, 0, C + (int64_t)nx * ns, ns, nullptr)))
        return rc;
      launch_chained(scale_rows_by_kernel, nblk((int64_t)mrow * mcol), 256, 0, L.st, mrow, mcol,
                     L.ev + nx, Q, mrow, Q2, mrow);
      DLAUNCH(L);
      if ((rc = dev_gemm(L, true, false, mcol, mcol, mrow, 1.0, Q, mrow, Q2, mrow, 0.0, nullptr, 0,
                         PAP, npn, nullptr)))
        return rc;
    }
  }
  LOB_CUDA_OK(cudaMemcpyAsync(theta, L.ev, nx * sizeof(double), cudaMemcpyDeviceToDevice, L.st));
  *npn_out = npn;
  return LOBPCG_OK;
}

}  // namespace

// Algorithm 2 on the Gram pair (GA, GB), device path.
int rr_initial_dev(DenseLayer& L, const double* GA, const double* GB, int nx, double* C,
                   double* theta, bool* breakdown) {
  DevDense& D = L.dev;
  *breakdown = false;
  double* MB = L.A[0];
  double* MA = L.A[1];
  double* H = L.A[2];
  double* Z = L.A[3];
  double* Rf = D.T1;
  double* Ri = L.A[5];
  double* T = D.T2;
  int* info = D.ints + 1;
  int* est = D.ints + 2;
  double* cr = D.scal + 2;
  int rc;
  if ((rc = configure_cond(L))) return rc;
  LOB_CUDA_OK(cudaMemsetAsync(info, 0, 2 * sizeof(int), L.st));
  launch_chained(dscale2_kernel, nblk((int64_t)nx * nx), 256, 0, L.st, nx, GB, nx, GA, nx, L.d, MB,
                 MA, nx);
  DLAUNCH(L);
  launch_chained(copy_block_cm_kernel, nblk((int64_t)nx * nx), 256, 0, L.st, nx, nx, MB, nx, Rf, nx,
                 1.0);
  DLAUNCH(L);
  if ((rc = dev_chol(L, nx, Rf, nx, info))) return rc;
  if ((rc = dev_trinv(L, nx, Rf, nx, Ri, nx, info))) return rc;
  launch_chained(cond_struct_kernel, 2, 1024, (size_t)(nx * nx + 3 * nx) * 4, L.st, nx, 0, MB,
                 nx, Ri, nx, cr, info);
  DLAUNCH(L);
  // H = Ri^T MA Ri
  if ((rc = dev_gemm(L, false, false, nx, nx, nx, 1.0, MA, nx, Ri, nx, 0.0, nullptr, 0, T, nx, info)))
    return rc;
  if ((rc = dev_gemm(L, true, false, nx, nx, nx, 1.0, Ri, nx, T, nx, 0.0, nullptr, 0, H, nx, info)))
    return rc;
  if ((rc = eig_into(L, nx, H, Z, est))) return rc;
  int fl[2];
  double crh[2];
  if ((rc = read_flags(L, info, 2, cr, 2, fl, crh))) return rc;
  const double condR = cond_of(crh);
  // breakdown: Cholesky failed or D X0^T B X0 D = R^T R is numerically
  // singular, cond(R)^2 >= 1 / (n_x eps)
  if (fl[0] != 0 || !(condR * condR < 1.0 / (nx * kEps64))) {
    *breakdown = true;
    return LOBPCG_OK;
  }
  note_check(L, fl[1]);
  if (fl[1] != 0 && (rc = eig_recover(L, nx, H, Z, fl[1]))) return rc;
  // C = D Ri Z
  if ((rc = dev_gemm(L, false, false, nx, nx, nx, 1.0, Ri, nx, Z, nx, 0.0, nullptr, 0, C, nx,
                     nullptr)))
    return rc;
  launch_chained(scale_rows_add_kernel, nblk((int64_t)nx * nx), 256, 0, L.st, nx, nx, L.d, C, nx,
                 nullptr, 0, 0);
  DLAUNCH(L);
  LOB_CUDA_OK(cudaMemcpyAsync(theta, L.ev, nx * sizeof(double), cudaMemcpyDeviceToDevice, L.st));
  return LOBPCG_OK;
}

// Algorithm 7, device path.  With S = [X, P, W] and the identities (12)-(13),
// D S^T B S D = [[I, F], [F^T, Bw]] (F the o x n_w block of the X and P rows,
// o = n_x + n_p), so its Cholesky factor is R = [[I, F], [0, Rw]] with
// Rw^T Rw = Bw - F^T F, and R^-1 = [[I, Y_t], [0, Y_w]], Y_w = Rw^-1,
// Y_t = -F Y_w.  With MA = D S^T A S D and Y = R^-1(:, o:), the projected
// matrix H = R^-T MA R^-1 is MA on the first o rows and columns, Q = MA Y on
// the off-diagonal blocks and Y^T Q on the W block; T Z = D R^-1 Z =
// D ([Z_top; 0] + Y Z(o:, :)).
int rr_modified_dev(DenseLayer& L, const double* SAS, const double* SBS, int ns, int nx, int np,
                    int nc, bool use_ortho, double tau_skip, bool* flip, double* condR, double* C,
                    int* npn_out, double* theta, double* PAP) {
  DevDense& D = L.dev;
  *flip = false;
  *condR = 1.0;
  const int o = nx + np, nw = ns - o;
  double* MB = L.A[0];
  double* MA = L.A[1];
  double* H = L.A[2];
  double* Z = L.A[3];
  double* TZ = L.A[4];
  double* Y = L.A[5];  // ns x nw, leading dimension ns
  double* Sw = D.T1;   // nw x nw
  double* Qm = D.T2;   // ns x nw
  int* info = D.ints + 1;
  int* est = D.ints + 2;
  double* cr = D.scal + 2;
  int rc;
  if ((rc = configure_cond(L))) return rc;
  LOB_CUDA_OK(cudaMemsetAsync(info, 0, 2 * sizeof(int), L.st));
  if (use_ortho) {
    if ((rc = eig_into(L, ns, SAS, Z, est))) return rc;
    int fl[1];
    if ((rc = read_flags(L, est, 1, nullptr, 0, fl, nullptr))) return rc;
    note_check(L, fl[0]);
    if (fl[0] != 0 && (rc = eig_recover(L, ns, SAS, Z, fl[0]))) return rc;
    return rr_tail(L, Z, Z, ns, nx, nc, C, npn_out, theta, PAP);
  }
  launch_chained(dscale2_kernel, nblk((int64_t)ns * ns), 256, 0, L.st, ns, SBS, ns, SAS, ns, L.d,
                 MB, MA, ns);
  DLAUNCH(L);
  const double* Hsrc = MA;
  if (nw > 0) {
    const double* F = MB + (int64_t)o * ns;  // rows 0..o-1 of the W columns
    // Sw = Bw - F^T F
    if ((rc = dev_gemm(L, true, false, nw, nw, o, -1.0, F, ns, F, ns, 1.0,
                       MB + o + (int64_t)o * ns, ns, Sw, nw, nullptr)))
      return rc;
    if ((rc = dev_chol(L, nw, Sw, nw, info))) return rc;
    if ((rc = dev_trinv(L, nw, Sw, nw, Y + o, ns, info))) return rc;
    if ((rc = dev_gemm(L, false, false, o, nw, nw, -1.0, F, ns, Y + o, ns, 0.0, nullptr, 0, Y, ns,
                       info)))
      return rc;
    launch_chained(cond_struct_kernel, 2, 1024, (size_t)(o * nw + nw * nw + 3 * ns) * 4,
                   L.st, ns, o, MB, ns, Y, ns, cr, info);
    DLAUNCH(L);
    if ((rc = dev_gemm(L, false, false, ns, nw, ns, 1.0, MA, ns, Y, ns, 0.0, nullptr, 0, Qm, ns,
                       info)))
      return rc;
    launch_chained(assemble_h_kernel, nblk((int64_t)ns * ns), 256, 0, L.st, ns, o, MA, ns, Qm, ns,
                   H, ns);
    DLAUNCH(L);
    if ((rc = dev_gemm(L, true, false, nw, nw, ns, 1.0, Y, ns, Qm, ns, 0.0, nullptr, 0,
                       H + o + (int64_t)o * ns, ns, info)))
      return rc;
    Hsrc = H;
  } else {
    LOB_CUDA_OK(cudaMemsetAsync(cr, 0, 2 * sizeof(double), L.st));  // cond(I) = 1, set below
  }
  if ((rc = eig_into(L, ns, Hsrc, Z, est))) return rc;
  int fl[2];
  double crh[2];
  if ((rc = read_flags(L, info, 2, cr, 2, fl, crh))) return rc;
  const double c = nw == 0 ? 1.0 : cond_of(crh);
  if (fl[0] != 0) {
    *flip = true;
    *condR = INFINITY;
    return LOBPCG_OK;
  }
  *condR = c;
  if (!(pow(c, -3.0) >= tau_skip)) {
    *flip = true;
    return LOBPCG_OK;
  }
  note_check(L, fl[1]);
  if (fl[1] != 0 && (rc = eig_recover(L, ns, Hsrc, Z, fl[1]))) return rc;
  // T Z = D ([Z_top; 0] + Y Z(o:, :))
  if (nw > 0) {
    if ((rc = dev_gemm(L, false, false, ns, ns, nw, 1.0, Y, ns, Z + o, ns, 0.0, nullptr, 0, TZ, ns,
                       nullptr)))
      return rc;
    launch_chained(scale_rows_add_kernel, nblk((int64_t)ns * ns), 256, 0, L.st, ns, ns, L.d, TZ, ns,
                   Z, ns, o);
  } else {
    launch_chained(copy_block_cm_kernel, nblk((int64_t)ns * ns), 256, 0, L.st, ns, ns, Z, ns, TZ,
                   ns, 1.0);
    DLAUNCH(L);
    launch_chained(scale_rows_add_kernel, nblk((int64_t)ns * ns), 256, 0, L.st, ns, ns, L.d, TZ, ns,
                   nullptr, 0, 0);
  }
  DLAUNCH(L);
  return rr_tail(L, TZ, Z, ns, nx, nc, C, npn_out, theta, PAP);
}

// The explicit Rayleigh-Ritz (every block of S^T A S and S^T B S computed,
// nothing taken from the identities (12)-(14)), device path.  With the
// scaling D = diag(S^T B S)^-1/2, MB = D S^T B S D and MA likewise, the
// leading o x o block (the X and P columns, o = n_x + n_p) is factored on its
// own, MB11 = R11^T R11, Y11 = R11^-1; the congruence T1 = blkdiag(Y11, I)
// turns the pencil into one whose B-block is [[I, Fb], [Fb^T, MB22]], which
// the structured path above factors (Cholesky of the Schur complement only).
// Together the two steps are the Cholesky factor of MB, R = [[R11, R11 Fb],
// [0, Rw]], so this is Algorithm 7 on the explicit pencil; the coefficients
// come back as C = D T1 C'.  The cond(R) estimate that drives the switch to
// orthogonalisation is that of the second factor: R11 is the factor of the
// Gram matrix of the previous iteration's B-orthonormal X and P, within
// rounding of the identity.  A failed R11 factorisation is a Cholesky
// failure (*flip, cond = inf), as in Algorithm 7.
bool dev_explicit_fits(const DenseLayer& L, int ns, int nx, int np) {
  const int o = nx + np;
  return o <= kCholMax && dev_rr_fits(L, ns, nx, ns - o);
}

int rr_explicit_dev(DenseLayer& L, const double* SAS, const double* SBS, int ns, int nx, int np,
                    int nc, double tau_skip, bool* flip, double* condR, double* C, int* npn_out,
                    double* theta, double* PAP) {
  DevDense& D = L.dev;
  *flip = false;
  *condR = 1.0;
  const int o = nx + np, nw = ns - o;
  // L.R[] hold the FP32-refinement blocks of dense_eig 1, unused on this path
  double* SB = L.R[0];   // ns x ns, T1^T MB T1
  double* SA = L.R[1];   // ns x ns, T1^T MA T1
  double* R11 = L.R[2];  // o x o, then kept as Y11 in Y
  double* Y = L.R[3];    // o x o, Y11
  double* d0 = L.R[4];   // ns
  double* Ka = L.R[5];   // o x ns, Y11^T MA[0:o, :]; then Y11 C'[0:o, :]
  double* MB = L.A[0];
  double* MA = L.A[1];
  int* info = D.ints + 4 * D.nmax + 16;
  int rc;
  launch_chained(dscale2_kernel, nblk((int64_t)ns * ns), 256, 0, L.st, ns, SBS, ns, SAS, ns, d0, MB,
                 MA, ns);
  DLAUNCH(L);
  launch_chained(copy_block_cm_kernel, nblk((int64_t)o * o), 256, 0, L.st, o, o, MB, ns, R11, o,
                 1.0);
  DLAUNCH(L);
  LOB_CUDA_OK(cudaMemsetAsync(info, 0, sizeof(int), L.st));
  if ((rc = dev_chol(L, o, R11, o, info))) return rc;
  int fl = 0;
  LOB_CUDA_OK(cudaMemcpyAsync(L.host, info, sizeof(int), cudaMemcpyDeviceToHost, L.st));
  LOB_CUDA_OK(cudaStreamSynchronize(L.st));
  ++L.syncs;
  memcpy(&fl, L.host, sizeof(int));
  if (fl != 0) {
    *flip = true;
    *condR = INFINITY;
    return LOBPCG_OK;
  }
  if ((rc = dev_trinv(L, o, R11, o, Y, o, nullptr))) return rc;
  // Ka = Y11^T MA[0:o, :], SA'11 = Ka[:, 0:o] Y11, SB'12 = Y11^T MB[0:o, o:]
  if ((rc = dev_gemm(L, true, false, o, ns, o, 1.0, Y, o, MA, ns, 0.0, nullptr, 0, Ka, o,
                     nullptr)))
    return rc;
  if ((rc = dev_gemm(L, false, false, o, o, o, 1.0, Ka, o, Y, o, 0.0, nullptr, 0, SA, ns,
                     nullptr)))
    return rc;
  if (nw > 0 && (rc = dev_gemm(L, true, false, o, nw, o, 1.0, Y, o, MB + (int64_t)o * ns, ns, 0.0,
                               nullptr, 0, SB + (int64_t)o * ns, ns, nullptr)))
    return rc;
  launch_chained(pre_fill_kernel, nblk((int64_t)ns * ns), 256, 0, L.st, ns, o, MB, MA, ns, Ka, o,
                 SB, SA, ns);
  DLAUNCH(L);
  int npn = 0;
  if ((rc = rr_modified_dev(L, SA, SB, ns, nx, np, nc, false, tau_skip, flip, condR, C, &npn,
                            theta, PAP)))
    return rc;
  if (*flip) return LOBPCG_OK;
  const int m = nx + npn;
  if ((rc = dev_gemm(L, false, false, o, m, o, 1.0, Y, o, C, ns, 0.0, nullptr, 0, Ka, o, nullptr)))
    return rc;
  launch_chained(pre_back_kernel, nblk((int64_t)ns * m), 256, 0, L.st, ns, m, o, d0, Ka, o, C, ns);
  DLAUNCH(L);
  *npn_out = npn;
  return LOBPCG_OK;
}

// svqb (Algorithm 4) / svqbDrop (Algorithm 6) transform, device path.
int svqb_transform_dev(DenseLayer& L, const double* G, int nu, bool drop, double tau, double* T,
                       int* nkeep) {
  DevDense& D = L.dev;
  double* MB = L.A[0];
  double* Z = L.A[3];
  int* est = D.ints + 2;
  int* keep = D.ints + 3;
  int rc;
  launch_chained(dscale2_kernel, nblk((int64_t)nu * nu), 256, 0, L.st, nu, G, nu, nullptr, 0, L.d,
                 MB, nullptr, nu);
  DLAUNCH(L);
  if ((rc = eig_into(L, nu, MB, Z, est))) return rc;
  launch_chained(svqb_dev_kernel, 1, 256, 0, L.st, nu, L.ev, L.d, Z, nu, drop ? 1 : 0, tau, T, nu,
                 keep);
  DLAUNCH(L);
  int fl[2];
  if ((rc = read_flags(L, est, 2, nullptr, 0, fl, nullptr))) return rc;
  note_check(L, fl[0]);
  if (fl[0] != 0) {
    if ((rc = eig_recover(L, nu, MB, Z, fl[0]))) return rc;
    launch_chained(svqb_dev_kernel, 1, 256, 0, L.st, nu, L.ev, L.d, Z, nu, drop ? 1 : 0, tau, T, nu,
                   keep);
    DLAUNCH(L);
    if ((rc = read_flags(L, keep, 1, nullptr, 0, fl + 1, nullptr))) return rc;
  }
  *nkeep = fl[1];
  return LOBPCG_OK;
}

}  // namespace lob
