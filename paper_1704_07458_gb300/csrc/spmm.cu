// Block CSR sparse product Y = A X (the A W, B W products of Algorithm 8 and
// Sec. 5.2), with the diagonal-B product BY = diag(b) X fused into the same
// pass over X, and the Chebyshev step that follows a product fused into its
// epilogue (see precond.cu).
//
// Layout: X and Y are row-major n x m blocks, so the m values of one row are
// contiguous.  The (row, column pair) items of the block are numbered row after
// row and dealt to the threads in that order: every nonzero a_ij reads one
// 16-byte piece of row j of X per thread, coalesced along the row, and stencil
// neighbours of consecutive rows overlap, so neighbour rows are served from L2
// and X streams from HBM about once.
//
// Bound by the FP64 pipe: 2 FMAs per clock and SM, 64 cycles per warp
// instruction and scheduler whether 32 lanes take part or 4.  So the items must
// fill the warps: with a warp per row (m = 71: 36 pairs, 64 lanes issued) the
// 64^3 7-point product with diagonal B took 453 us against 237 us of FP64 pipe
// and 69 us of bytes; numbered through it takes 293 us.
#include <algorithm>

#include "kernels.cuh"

namespace lob {

int64_t g_launches = 0;

namespace {

constexpr int kSpmmThreads = 256;
constexpr int kSpmmCtas = 5;  // per SM: 40 warps hide the three dependent loads of a row
constexpr int kBatch = 4;     // nonzeros in flight per thread (8 of them leave room for 24 warps)

// One column pair of a row, or one column when rows are not 16-byte aligned.
template <bool kPair>
struct Cols;
template <>
struct Cols<true> {
  double2 v;
  // ro: memory that nothing writes while the kernel runs.  two: the second
  // column exists; if not, it is not read (the caller's block may end there).
  __device__ __forceinline__ void load_ro(const double* p, bool two) {
    v = two ? __ldg(reinterpret_cast<const double2*>(p)) : make_double2(__ldg(p), 0.0);
  }
  __device__ __forceinline__ void load(const double* p, bool two) {
    v = two ? *reinterpret_cast<const double2*>(p) : make_double2(*p, 0.0);
  }
  __device__ __forceinline__ void zero() { v = make_double2(0.0, 0.0); }
  __device__ __forceinline__ void fma_(double a, const Cols& x) {
    v.x = fma(a, x.v.x, v.x);
    v.y = fma(a, x.v.y, v.y);
  }
  __device__ __forceinline__ void scale(double a) {
    v.x *= a;
    v.y *= a;
  }
  __device__ __forceinline__ void add(const Cols& x) {
    v.x += x.v.x;
    v.y += x.v.y;
  }
  __device__ __forceinline__ void sub(const Cols& x) {
    v.x -= x.v.x;
    v.y -= x.v.y;
  }
  // both columns when the second exists
  __device__ __forceinline__ void store(double* p, bool two) const {
    if (two && (reinterpret_cast<uintptr_t>(p) & 15) == 0) {
      *reinterpret_cast<double2*>(p) = v;
    } else {
      p[0] = v.x;
      if (two) p[1] = v.y;
    }
  }
};
template <>
struct Cols<false> {
  double v;
  __device__ __forceinline__ void load_ro(const double* p, bool) { v = __ldg(p); }
  __device__ __forceinline__ void load(const double* p, bool) { v = *p; }
  __device__ __forceinline__ void zero() { v = 0.0; }
  __device__ __forceinline__ void fma_(double a, const Cols& x) { v = fma(a, x.v, v); }
  __device__ __forceinline__ void scale(double a) { v *= a; }
  __device__ __forceinline__ void add(const Cols& x) { v += x.v; }
  __device__ __forceinline__ void sub(const Cols& x) { v -= x.v; }
  __device__ __forceinline__ void store(double* p, bool) const { *p = v; }
};

// acc += A(row, :) X(:, c) for this thread's columns; kBatch nonzeros of
// the row are in flight (their column indices and values, then their X pieces).
// The loop ends at the longest row of the warp by a branch: an FMA predicated
// off for all lanes occupies the FP64 pipe like any other (three of eight of
// them doubled the time of 5-point rows).  Lanes whose row is shorter add 0 * 0.
// Every lane of the warp calls it; live: this lane has an item.
template <bool kPair>
__device__ __forceinline__ void row_product(const int32_t* __restrict__ rowptr,
                                            const int32_t* __restrict__ col,
                                            const double* __restrict__ val,
                                            const double* __restrict__ X, int64_t ldx, int64_t row,
                                            int c, bool live, bool two, Cols<kPair>& acc) {
  const int lo = live ? __ldg(rowptr + row) : 0, hi = live ? __ldg(rowptr + row + 1) : 0;
  const int longest = __reduce_max_sync(0xffffffffu, hi - lo);
  for (int p = 0; p < longest; p += kBatch) {
    int ci[kBatch];
    double a[kBatch];
    Cols<kPair> x[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const bool on = lo + p + j < hi;
      ci[j] = on ? __ldg(col + lo + p + j) : -1;
      a[j] = on ? __ldg(val + lo + p + j) : 0.0;
    }
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      x[j].zero();
      if (ci[j] >= 0) x[j].load_ro(X + (int64_t)ci[j] * ldx + c, two);
    }
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      if (p + j >= longest) break;
      acc.fma_(a[j], x[j]);
    }
  }
}

// This thread's item of its column tile (blockIdx.y): rows of `width` items.
struct Item {
  int64_t row;
  int q;
};
__device__ __forceinline__ Item item_of(int width) {
  const int64_t first = (int64_t)blockIdx.x * kSpmmThreads;
  const int64_t row0 = first / width;
  const unsigned t = (unsigned)(first - row0 * width) + threadIdx.x, dr = t / (unsigned)width;
  return {row0 + dr, (int)(t - dr * (unsigned)width) + (int)blockIdx.y * width};
}

template <bool kPair>
__global__ void __launch_bounds__(kSpmmThreads, kSpmmCtas) spmm_csr_kernel(
    int64_t n, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
    const double* __restrict__ val, const double* __restrict__ X, int64_t ldx, int m, int width,
    double* __restrict__ Y, int64_t ldy, const double* __restrict__ b, double* __restrict__ BY,
    int64_t ldby) {
  const Item it = item_of(width);
  const int c = kPair ? 2 * it.q : it.q;
  const bool live = it.row < n && c < m, two = c + 1 < m;
  Cols<kPair> acc;
  acc.zero();
  row_product<kPair>(rowptr, col, val, X, ldx, it.row, c, live, two, acc);
  if (!live) return;
  acc.store(Y + it.row * ldy + c, two);
  if (b) {
    Cols<kPair> x;
    x.load_ro(X + it.row * ldx + c, two);
    x.scale(__ldg(b + it.row));
    x.store(BY + it.row * ldby + c, two);
  }
}

// One Chebyshev step on the fly (see precond.cu): with z = D^-1 (r - A w),
// d <- a d + bz z and w' = w + d.  The last step writes w' only.  A w is summed
// by itself and z rounded before bz multiplies it, as in separate passes: terms
// of A w taken from r one by one would cost r the bits that they cancel among
// themselves.  d and, where W is R, r are written by the thread that has read
// them: ordinary loads, not the read-only path, which is for memory that stays as
// it is while the kernel runs.
template <bool kPair>
__global__ void __launch_bounds__(kSpmmThreads, kSpmmCtas) cheb_step_kernel(
    int64_t n, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
    const double* __restrict__ val, const double* __restrict__ w, int64_t ld, int m, int width,
    const double* R, int64_t ldr, const double* __restrict__ dinv, double a, double bz, double* d,
    double* wnew, int64_t ldw, bool last) {
  const Item it = item_of(width);
  const int c = kPair ? 2 * it.q : it.q;
  const bool live = it.row < n && c < m, two = c + 1 < m;
  Cols<kPair> acc, z, dn, wn;
  acc.zero();
  if (live) {
    z.load(R + it.row * ldr + c, two);
    dn.load(d + it.row * ld + c, two);
    wn.load_ro(w + it.row * ld + c, two);
  }
  row_product<kPair>(rowptr, col, val, w, ld, it.row, c, live, two, acc);
  if (!live) return;
  z.sub(acc);
  z.scale(__ldg(dinv + it.row));
  z.scale(bz);
  z.fma_(a, dn);  // a d + bz z
  dn = z;
  wn.add(dn);
  if (!last) dn.store(d + it.row * ld + c, two);
  wn.store(wnew + it.row * ldw + c, two);
}

// Column tiles of at most 40 items: a CTA then covers six rows or more, whose
// neighbours along x it shares in L1, and the planes that the neighbours along z
// lie in stay in L2 at any block width (m = 282 in one tile: 11.6 ms at 128^3).
struct Tiles {
  int width, count;
};
Tiles tiles_of(int items) {
  const int count = (int)ceil_div(items, 40);
  return {(int)ceil_div(items, count), count};
}
dim3 grid_of(int64_t n, Tiles t) {
  return dim3((unsigned)ceil_div(n * t.width, kSpmmThreads), (unsigned)t.count);
}

// pairs: rows 16-byte aligned (base and leading dimension even)
bool pairs_ok(const double* X, int64_t ldx) {
  return ((uintptr_t)X % 16 == 0) && (ldx % 2 == 0);
}

}  // namespace

int spmm(cudaStream_t st, int64_t n, const int32_t* rowptr, const int32_t* col,
         const double* val, const double* X, int64_t ldx, int m, double* Y, int64_t ldy,
         const double* b, double* BY, int64_t ldby) {
  if (n <= 0 || m <= 0) return LOBPCG_OK;
  const double* bb = BY ? b : nullptr;
  if (pairs_ok(X, ldx)) {
    const Tiles t = tiles_of((m + 1) / 2);
    spmm_csr_kernel<true><<<grid_of(n, t), kSpmmThreads, 0, st>>>(
        n, rowptr, col, val, X, ldx, m, t.width, Y, ldy, bb, BY, ldby);
  } else {
    const Tiles t = tiles_of(m);
    spmm_csr_kernel<false><<<grid_of(n, t), kSpmmThreads, 0, st>>>(
        n, rowptr, col, val, X, ldx, m, t.width, Y, ldy, bb, BY, ldby);
  }
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

int cheb_step(cudaStream_t st, int64_t n, const int32_t* rowptr, const int32_t* col,
              const double* val, const double* w, int64_t ld, int m, const double* R, int64_t ldr,
              const double* dinv, double a, double bz, double* d, double* wnew, int64_t ldw,
              bool last) {
  if (n <= 0 || m <= 0) return LOBPCG_OK;
  if (pairs_ok(w, ld) && pairs_ok(d, ld) && pairs_ok(R, ldr)) {
    const Tiles t = tiles_of((m + 1) / 2);
    cheb_step_kernel<true><<<grid_of(n, t), kSpmmThreads, 0, st>>>(
        n, rowptr, col, val, w, ld, m, t.width, R, ldr, dinv, a, bz, d, wnew, ldw, last);
  } else {
    const Tiles t = tiles_of(m);
    cheb_step_kernel<false><<<grid_of(n, t), kSpmmThreads, 0, st>>>(
        n, rowptr, col, val, w, ld, m, t.width, R, ldr, dinv, a, bz, d, wnew, ldw, last);
  }
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

}  // namespace lob

LOBPCG_EXPORT int lobpcg_spmm(int64_t n, const int32_t* rowptr, const int32_t* col,
                              const double* val, const double* X, int64_t ldx, int64_t m,
                              double* Y, int64_t ldy, const double* b, double* BY,
                              int64_t ldby, void* stream) {
  if (n < 0 || m < 0 || m > (1 << 20)) return LOBPCG_ERR_ARG;
  if (n > 0 && m > 0 && (!rowptr || !col || !val || !X || !Y || ldx < m || ldy < m))
    return LOBPCG_ERR_ARG;
  if (b && (!BY || ldby < m)) return LOBPCG_ERR_ARG;
  if (BY && !b) return LOBPCG_ERR_ARG;
  return lob::spmm((cudaStream_t)stream, n, rowptr, col, val, X, ldx, (int)m, Y, ldy, b, BY,
                   ldby);
}
