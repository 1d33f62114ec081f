// Block CSR sparse product Y = A X (the A W, B W products of Algorithm 8 and
// Sec. 5.2), with the diagonal-B product BY = diag(b) X fused into the same
// pass over X, and the Chebyshev step that follows a product fused into its
// epilogue (see precond.cu).
//
// Layout: X and Y are row-major n x m blocks, so the m values of one row are
// contiguous.  The items of the block (a row with a pair of columns, or with one
// or two single columns where rows are not 16-byte aligned) are numbered row
// after row and dealt to the threads in that order: every nonzero a_ij reads one
// piece of row j of X per item, coalesced along the row, and stencil neighbours
// of consecutive rows overlap, so neighbour rows are served from L2 and X streams
// from HBM about once.
//
// Bound by the FP64 pipe: 2 FMAs per clock and SM, 64 cycles per warp
// instruction and scheduler whether 32 lanes take part or 4, or none: an FMA
// predicated off for all of them occupies the pipe like any other.  So the items
// must fill the warps: with a warp per row (m = 71: 36 pairs, 64 lanes issued) the
// 64^3 7-point product with diagonal B took 453 us against 237 us of FP64 pipe
// and 69 us of bytes.
#include <algorithm>

#include "kernels.cuh"

namespace lob {

int64_t g_launches = 0;

namespace {

constexpr int kSpmmThreads = 256;
constexpr int kSpmmCtas = 6;  // per SM: 48 warps hide the three dependent loads of a row
constexpr int kBatch = 3;     // nonzeros in flight per thread; more leave room for fewer warps

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

// acc[k] += A(row, :) X(:, c[k]) for this thread's G items of a row; kBatch
// nonzeros of the row are in flight (their column indices and values, then their X
// pieces).  A batch that the warp's longest row does not fill is summed by code of
// its own for each count, so that the sum ends by a branch: in a batch cut short by
// conditions the compiler predicates the last FMA, which then costs what it would
// have added (four at a time took eight FMAs for 7 points: the 64^3 product of 32
// columns 119 us, of 71 columns with diagonal B 293 us; 101 and 256 so).  Lanes
// whose row is shorter than the longest add 0 * 0.  Every lane of the warp calls
// it; on[k]: this lane has item k.
template <bool kPair, int G>
__device__ __forceinline__ void row_product(const int32_t* __restrict__ rowptr,
                                            const int32_t* __restrict__ col,
                                            const double* __restrict__ val,
                                            const double* __restrict__ X, int64_t ldx, int64_t row,
                                            const int (&c)[G], const bool (&on)[G], bool two,
                                            Cols<kPair> (&acc)[G]) {
  static_assert(kBatch == 3, "the counts below");
  const int lo = on[0] ? __ldg(rowptr + row) : 0, hi = on[0] ? __ldg(rowptr + row + 1) : 0;
  const int longest = __reduce_max_sync(0xffffffffu, hi - lo);
  for (int p = 0; p < longest; p += kBatch) {
    int ci[kBatch];
    double a[kBatch];
    Cols<kPair> x[kBatch][G];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const bool in = lo + p + j < hi;
      ci[j] = in ? __ldg(col + lo + p + j) : -1;
      a[j] = in ? __ldg(val + lo + p + j) : 0.0;
    }
#pragma unroll
    for (int j = 0; j < kBatch; ++j)
#pragma unroll
      for (int k = 0; k < G; ++k) {
        x[j][k].zero();
        if (ci[j] >= 0 && on[k]) x[j][k].load_ro(X + (int64_t)ci[j] * ldx + c[k], two);
      }
    auto add = [&](int j) {
#pragma unroll
      for (int k = 0; k < G; ++k) acc[k].fma_(a[j], x[j][k]);
    };
    const int left = longest - p;
    if (left >= kBatch) {
      add(0);
      add(1);
      add(2);
    } else if (left == 1) {
      add(0);
    } else if (left == 2) {  // not a plain else, which the compiler folds into one predicated sum
      add(0);
      add(1);
    }
  }
}

// Column tiles: tile blockIdx.y has `width` items a row and thread, G of them
// `width` apart.  The quotients by the width are multiplications: exact for
// first < 2^48 and t < 320, width <= 40 (a 64-bit and a 32-bit division cost 4 to
// 8 % of a narrow product).
struct Tiles {
  int width, count;
  uint64_t by_row;   // floor(2^64 / width) + 1
  uint32_t by_item;  // floor(2^16 / width) + 1
};
constexpr int kMaxWidth = 40;

// This thread's row and its first item.
struct Item {
  int64_t row;
  int q;
};
__device__ __forceinline__ Item item_of(const Tiles& tl, int G) {
  const uint64_t first = (uint64_t)blockIdx.x * kSpmmThreads;
  const uint64_t row0 = tl.width == 1 ? first : __umul64hi(first, tl.by_row);
  const uint32_t t = (uint32_t)(first - row0 * tl.width) + threadIdx.x;
  const uint32_t dr = (t * tl.by_item) >> 16;
  return {(int64_t)(row0 + dr),
          (int)(t - dr * (uint32_t)tl.width) + (int)blockIdx.y * tl.width * G};
}

template <bool kPair, int G, int kCtas>
__global__ void __launch_bounds__(kSpmmThreads, kCtas) spmm_csr_kernel(
    int64_t n, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
    const double* __restrict__ val, const double* __restrict__ X, int64_t ldx, int m,
    const Tiles tl, double* __restrict__ Y, int64_t ldy, const double* __restrict__ b,
    double* __restrict__ BY, int64_t ldby) {
  const Item it = item_of(tl, G);
  int c[G];
  bool on[G];
#pragma unroll
  for (int k = 0; k < G; ++k) {
    c[k] = (kPair ? 2 : 1) * (it.q + k * tl.width);
    on[k] = it.row < n && c[k] < m;
  }
  const bool two = c[0] + 1 < m;
  Cols<kPair> acc[G];
#pragma unroll
  for (int k = 0; k < G; ++k) acc[k].zero();
  row_product<kPair, G>(rowptr, col, val, X, ldx, it.row, c, on, two, acc);
#pragma unroll
  for (int k = 0; k < G; ++k) {
    if (!on[k]) continue;
    acc[k].store(Y + it.row * ldy + c[k], two);
    if (b) {
      Cols<kPair> x;
      x.load_ro(X + it.row * ldx + c[k], two);
      x.scale(__ldg(b + it.row));
      x.store(BY + it.row * ldby + c[k], two);
    }
  }
}

// One Chebyshev step on the fly (see precond.cu): with z = D^-1 (r - A w),
// d <- a d + bz z and w' = w + d.  The last step writes w' only.  A w is summed
// by itself and z rounded before bz multiplies it, as in separate passes: terms
// of A w taken from r one by one would cost r the bits that they cancel among
// themselves.  d and, where W is R, r are written by the thread that has read
// them: ordinary loads, not the read-only path, which is for memory that stays as
// it is while the kernel runs.
__global__ void __launch_bounds__(kSpmmThreads, kSpmmCtas) cheb_step_kernel(
    int64_t n, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
    const double* __restrict__ val, const double* __restrict__ w, int64_t ld, int m,
    const Tiles tl, const double* R, int64_t ldr, bool r_pairs, const double* __restrict__ dinv,
    double a, double bz, double* d, double* wnew, int64_t ldw, bool last) {
  const Item it = item_of(tl, 1);
  const int c[1] = {2 * it.q};
  const bool on[1] = {it.row < n && c[0] < m}, two = c[0] + 1 < m;
  Cols<true> acc[1], z, dn, wn;
  acc[0].zero();
  row_product<true, 1>(rowptr, col, val, w, ld, it.row, c, on, two, acc);
  if (!on[0]) return;
  const double* r = R + it.row * ldr + c[0];
  if (r_pairs)
    z.load(r, two);
  else
    z.v = make_double2(r[0], two ? r[1] : 0.0);
  dn.load(d + it.row * ld + c[0], two);
  wn.load_ro(w + it.row * ld + c[0], two);
  z.sub(acc[0]);
  z.scale(__ldg(dinv + it.row));
  z.scale(bz);
  z.fma_(a, dn);  // a d + bz z
  dn = z;
  wn.add(dn);
  if (!last) dn.store(d + it.row * ld + c[0], two);
  wn.store(wnew + it.row * ldw + c[0], two);
}

// Column tiles of at most 40 pairs: a CTA then covers six rows or more, whose
// neighbours along x it shares in L1, and the planes that the neighbours along z
// lie in stay in L2 at any block width (m = 282 in one tile: 11.6 ms at 128^3).
Tiles tiles_of(int items, int G, int most) {
  const int count = (int)ceil_div(items, (int64_t)G * most);
  const int width = (int)ceil_div(items, (int64_t)G * count);
  return {width, count, ~0ull / (unsigned)width + 1, 65536u / (unsigned)width + 1};
}
dim3 grid_of(int64_t n, const Tiles& t) {
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
  auto run = [&](auto* kernel, const Tiles& t) {
    kernel<<<grid_of(n, t), kSpmmThreads, 0, st>>>(n, rowptr, col, val, X, ldx, m, t, Y, ldy, bb,
                                                   BY, ldby);
  };
  // Two columns a thread where few lanes are then idle: aligned rows in pairs up to
  // one in ten (512^2, 7 columns: 22.8 us, 20.7 singly; diagonal B, 9 columns: 35.2
  // and 37.3), if these make four CTAs an SM (30 x 26 x 28: 6.0 us in pairs at 4
  // columns, 5.3 singly, with diagonal B at 8 columns 8.4 and 7.1); others in two
  // single columns up to one in fourteen, twice the work behind each row's chain of
  // loads (64^3, 64 columns: 248 us with one, 203 with two), if four waves of CTAs
  // remain (200 x 90, 31 columns, 1.2 waves: 8.6 and 10.1 us).  One column a thread
  // takes 64 warps an SM, with a few values spilled, for blocks that do not stay in
  // L2 (100^3, 7 columns: 95 us, 105 with 48 warps; 64^3, 6 columns: 25.0 and 23.4);
  // a row of A is taken as seven nonzeros.
  const bool even = m % 2 == 0;
  const Tiles pairs = tiles_of((m + 1) / 2, 1, kMaxWidth), two = tiles_of(m, 2, 32);
  auto ctas = [&](const Tiles& t) { return ceil_div(n * t.width, kSpmmThreads) * t.count; };
  if ((even || m > 8) && pairs_ok(X, ldx) && ctas(pairs) >= 4 * 152)
    run(spmm_csr_kernel<true, 1, kSpmmCtas>, pairs);
  else if ((even || m > 12) && m > 4 && ctas(two) >= 4 * kSpmmCtas * 152)
    run(spmm_csr_kernel<false, 2, kSpmmCtas>, two);
  else if (n * (8 * (ldx + ldy) + 84) <= (96 << 20))
    run(spmm_csr_kernel<false, 1, kSpmmCtas>, tiles_of(m, 1, 32));
  else
    run(spmm_csr_kernel<false, 1, 8>, tiles_of(m, 1, 32));
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

int cheb_step(cudaStream_t st, int64_t n, const int32_t* rowptr, const int32_t* col,
              const double* val, const double* w, int64_t ld, int m, const double* R, int64_t ldr,
              const double* dinv, double a, double bz, double* d, double* wnew, int64_t ldw,
              bool last) {
  if (n <= 0 || m <= 0) return LOBPCG_OK;
  if (!pairs_ok(w, ld) || !pairs_ok(d, ld)) return LOBPCG_ERR_ARG;
  const Tiles t = tiles_of((m + 1) / 2, 1, kMaxWidth);
  cheb_step_kernel<<<grid_of(n, t), kSpmmThreads, 0, st>>>(
      n, rowptr, col, val, w, ld, m, t, R, ldr, pairs_ok(R, ldr), dinv, a, bz, d, wnew, ldw, last);
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
