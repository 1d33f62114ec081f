// Tensor-core (tcgen05 / TMEM) FP64 emulation of the two n-scaled
// contractions of an LOBPCG iteration (Sec. 5.2, Eqs. (10)-(14)): the Gram
// G = U^T V and the basis update Y = beta Y0 + alpha S C.
//
// Arithmetic (the contract of ozaki.cu): each FP64 operand is cut, relative to
// an exponent shared by a block of values, into S signed 8-bit digits (exact
// in BF16); digit products are exact; every level of digit pairs but the last
// is summed exactly in an FP32 TMEM accumulator; accumulators are converted
// exactly into int64 registers and the FP64 result is assembled with integer
// operations only.  No FP64 instruction runs on the hot path.
//
// GB300 mapping:
//  * one CTA per SM owns a 128 x NT output tile (512 compute threads and a
//    helper warpgroup), NT <= 96 a multiple of 16: tcgen05.mma kind::f16,
//    M = 128, N = NT, K = 16, A in TMEM, B in shared memory;
//  * the contraction runs in chunks of 16 (rows of U and V for the Gram,
//    columns of S for the update), grouped in blocks of at most 256 (the Gram's
//    share one exponent per operand column; the update has one per row).  With
//    |digit| <= 128 (129 in the last of up to six) the sums of levels 0, 1, 2 (and 3 for S = 7) stay below 2^24
//    in their units over a block, so they are exact in FP32; the deeper levels
//    (below 2^-24 resp. 2^-32 of level 0) share one inexact accumulator.  4 or 5
//    accumulators x NT columns and two to four digit stages of A fit the 512
//    TMEM columns, and the accumulators are read once per block;
//  * compute warps cut FP64 values from global memory straight into digit
//    planes; their loads for the chunk after next are in flight meanwhile.  The
//    digits of the small matrix C of the update are cut once per call and
//    arrive by cp.async.bulk four chunks ahead;
//  * the shared exponents come from a streaming pre-pass at full occupancy;
//  * every mbarrier wait is bounded: a wait that runs out marks the result NaN
//    (and, for the update, sets a status bit that the solver reads with its
//    per-iteration scalars) and the CTA returns instead of hanging.
#include <algorithm>
#include <type_traits>

#include "kernels.cuh"
#include "ozaki_common.cuh"

namespace lob {
namespace {

constexpr int TCM = 128;            // MMA M
constexpr int TCK = 16;             // contraction length of a chunk (one MMA K)
constexpr int KG = TCK / 8;         // core-matrix groups along K in a chunk
constexpr int kChunksPerBlock = 16; // 256 rows / columns share one exponent
constexpr int kBlock = TCK * kChunksPerBlock;
constexpr int NTMAX = 96;           // max MMA N (output columns of a tile)
constexpr int kFrac = 30;           // fraction bits of the int64 accumulators
constexpr int kEZero = -4000;       // exponent of an all-zero block
constexpr uint32_t kTmemCols = 512;
constexpr int kSpin = 1 << 22;      // bound of every mbarrier wait
constexpr int kMaxUpdateK = 6144;   // columns of S an update takes (3 n_x <= 6144)

template <int S>
__host__ __device__ constexpr int nacc() { return S >= 7 ? 5 : (S < 4 ? S : 4); }
// accumulator of digit level l = s + t (0-based digit indices)
template <int S>
__host__ __device__ constexpr int acc_of(int l) { return l < nacc<S>() - 1 ? l : nacc<S>() - 1; }
__host__ __device__ inline size_t planeB_bytes(int NT) { return (size_t)KG * (NT / 8) * 128; }

// 0x80 in each of the S-1 low bytes: adding it turns the fixed-point value
// into bytes that are the balanced digits plus 128.
template <int S>
__host__ __device__ constexpr long long digit_bias() {
  long long b = 0;
  for (int i = 0; i < S - 1; ++i) b |= 0x80LL << (8 * i);
  return b;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Digits of x relative to the exponent bound E (|x| < 2^E): the fixed-point
// integer F = round(x 2^(8S-1-E)) (|F| <= 2^(8S-1)) written in balanced base
// 256, F = sum_s d_s 256^(S-1-s), |d_s| <= 128; returns the pre-weighted
// values d_s 2^(-8s), each exact in BF16.  Integer operations only.
template <int S>
__device__ __forceinline__ void digits(double x, int E, float (&d)[S]) {
  const long long bits = __double_as_longlong(x);
  const int be = (int)((bits >> 52) & 0x7FF);
  const long long mant = (bits & 0x000FFFFFFFFFFFFFLL) | ((long long)(be != 0) << 52);
  // F = round(mant 2^sh), sh = max(be, 1) - 1076 + 8S - E <= 2 whenever
  // |x| < 2^E (a zero x gives F = 0 for any sh).  Branch-free: with
  // v = mant 2^3 < 2^56 and t = 2 - sh clamped to [0, 63],
  // F = ((v >> t) + 1) >> 1 (round half up in magnitude).
  const int t = min(max(2 - (max(be, 1) - 1076 + 8 * S - E), 0), 63);
  const long long F = (((mant << 3) >> t) + 1) >> 1;
  const long long G = digit_bias<S>() + (bits < 0 ? -F : F);
  const uint32_t lo = (uint32_t)G, hi = (uint32_t)((unsigned long long)G >> 32);
#pragma unroll
  for (int s = 1; s < S; ++s) {
    const int b = S - 1 - s;  // byte of digit s
    const uint32_t w = b < 4 ? lo : hi;
    // 0x4B0000xx is 2^23 + xx; minus (2^23 + 128), scaled by 2^-8s (exact)
    const float f = __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7540u | (uint32_t)(b & 3)));
    const float sc = __uint_as_float((uint32_t)(127 - 8 * s) << 23);
    d[s] = fmaf(f, sc, -8388736.0f * sc);
  }
  d[0] = (float)(int)(G >> (8 * (S - 1)));
}

// The splits of the compute warps: eight consecutive K values of one row or
// column, first in a form that frees the registers of the values (load), then
// plane by plane (plane): four packed BF16 pairs each.  The exponent bounds come
// as thr = split_thr(E), which is additive in E modulo 2^32; it serves
// kFastEMin < E < kFastEMax, `load_any` serves every E.
//
// S <= 6, on the FP32 pipe.  The integer pipe takes an instruction every two
// cycles, so a split by shifts and byte permutes (25 integer instructions per
// value) bounded the kernels at 1,400 to 2,200 cycles a chunk against 1,300 of
// MMAs.  Here x 2^(7-E) is a sum of two floats: a takes the top 24 bits of the
// mantissa with the exponent field moved by one multiply-add (values below
// 2^-87 of the bound are raised to it: all their digits are zero), b the other
// 29 bits.  Digit s is what the sum rounds to at a multiple of 2^-8s: adding and
// subtracting 1.5 * 2^(23-8s) leaves it, exact, pre-weighted and balanced
// (|d_s| <= 129, the 129 in the last digit only).
//
// The digits sum to F of `digits`, every bit of it: F is one rounding of x, and
// 29 bits do not fit a float, so b and all that follows it round down and b
// carries the half unit of the last digit, 2^(7-8S), with it.  Then the last
// digit is a floor, and a floor is not changed by floors at finer multiples
// before it.  (Rounded to the nearest at each step, x was rounded twice for
// S = 6: largest error 0.73 units of the last digit and not 0.5, 17 % of the
// values in the top binade with another F.)  A negative x takes the one's
// complement of its low bits, which breaks its ties away from zero as F does.  b
// joins a after the fourth digit (a + b is exact enough before that only to
// choose a digit).  Ten integer instructions per value remain.
constexpr int kFastEMin = -900, kFastEMax = 1100;

__host__ __device__ constexpr uint32_t split_thr(int E) { return (uint32_t)(E + 889) << 20; }

__host__ __device__ constexpr float pow2f(int e) {
  return e >= 0 ? (float)(1ull << e) : 1.0f / (float)(1ull << -e);
}

// F = round(x 2^(8S-1-E)), the fixed-point integer of `digits`
template <int S>
__device__ __noinline__ long long fixed_any(double x, int E) {
  const long long bits = __double_as_longlong(x);
  const int be = (int)((bits >> 52) & 0x7FF);
  const long long mant = (bits & 0x000FFFFFFFFFFFFFLL) | ((long long)(be != 0) << 52);
  const int t = min(max(2 - (max(be, 1) - 1076 + 8 * S - E), 0), 63);
  const long long F = (((mant << 3) >> t) + 1) >> 1;
  return bits < 0 ? -F : F;
}

template <int S>
struct Split {
  float a[8], b[8];

  __device__ __forceinline__ void load(int i, double x, uint32_t thr) {
    const uint32_t xh = (uint32_t)__double2hiint(x), xl = (uint32_t)__double2loint(x);
    const uint32_t m = (uint32_t)max((int)(xh & 0x7FFFFFFFu), (int)(thr + (40u << 20)));
    // exponent field be - E - 889 = (be - 1023) + (7 - E) + 127
    const uint32_t w = __funnelshift_l(xl, m, 3) - thr * 8u;
    a[i] = __uint_as_float((xh & 0x80000000u) | w);
    const int low = (int)((xl & 0x1FFFFFFFu) ^ (uint32_t)((int)xh >> 31));
    b[i] = __fmaf_rd(__int2float_rd(low) * pow2f(-52), __uint_as_float(w & 0x7F800000u),
                     pow2f(7 - 8 * S));
  }
  // a + b is F itself: no bits below the last digit, so no half unit
  __device__ __forceinline__ void load_any(int i, double x, int E) {
    constexpr int sh = 8 * S - 24;
    const long long F = fixed_any<S>(x, E);
    a[i] = (float)(int)(F >> sh) * pow2f(-16);
    b[i] = (float)(int)(F & ((1LL << sh) - 1)) * pow2f(8 - 8 * S);
  }
  template <int s>
  __device__ __forceinline__ void plane(uint32_t (&w)[4]) {
    constexpr float M = 1.5f * pow2f(23 - 8 * s);
    constexpr int kJoin = S > 4 ? 3 : S - 1;  // where b joins a
    float d[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (s == S - 1) {
        if (s == kJoin) a[i] = __fadd_rd(a[i], b[i]);
        d[i] = __fadd_rd(a[i], M) - M;
      } else {
        d[i] = ((s >= 2 && s <= kJoin ? a[i] + b[i] : a[i]) + M) - M;
        a[i] -= d[i];
        if (s == kJoin) a[i] = __fadd_rd(a[i], b[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
      w[i] = __byte_perm(__float_as_uint(d[2 * i]), __float_as_uint(d[2 * i + 1]), 0x7632);
  }
};

// S = 7: 55 bits do not fit two floats; the fixed-point integer by 32-bit shifts,
// its digits as bytes with 128 added.
template <>
struct Split<7> {
  uint2 g[8];

  static __device__ __forceinline__ uint2 bias(uint32_t Fl, uint32_t Fh) {
    uint2 r;  // 0x80 in each of the six low bytes balances the digits
    asm("add.cc.u32 %0, %2, 0x80808080;\n\taddc.u32 %1, %3, 0x00008080;\n"
        : "=r"(r.x), "=r"(r.y)
        : "r"(Fl), "r"(Fh));
    return r;
  }
  __device__ __forceinline__ void load(int i, double x, uint32_t thr) {
    const uint32_t xh = (uint32_t)__double2hiint(x), xl = (uint32_t)__double2loint(x);
    // with M the 53-bit mantissa at the top of 64 bits, 2 F = M >> q
    const uint32_t q = ((thr - (889u << 20) + (1030u << 20)) - (xh & 0x7FF00000u)) >> 20;
    const uint32_t mh = (xh & 0x000FFFFFu) | 0x00100000u;
    const uint32_t Mh = __funnelshift_l(xl, mh, 11), Ml = xl << 11;
    uint32_t Fl, Fh;  // 64-bit shift by any q: the shifts clamp at 32 instead of wrapping
    asm("shr.u32 %0, %1, %2;\n" : "=r"(Fh) : "r"(Mh), "r"(q));
    asm("shr.u32 %0, %1, %2;\n"
        : "=r"(Fl)
        : "r"(__funnelshift_rc(Ml, Mh, q)), "r"((uint32_t)max((int)q - 32, 0)));
    asm("add.cc.u32 %0, %0, 1;\n\taddc.u32 %1, %1, 0;\n" : "+r"(Fl), "+r"(Fh));
    Fl = __funnelshift_r(Fl, Fh, 1);
    Fh >>= 1;
    const uint32_t sg = (uint32_t)((int)xh >> 31);
    Fl ^= sg;
    Fh ^= sg;
    asm("sub.cc.u32 %0, %0, %2;\n\tsubc.u32 %1, %1, %2;\n" : "+r"(Fl), "+r"(Fh) : "r"(sg));
    g[i] = bias(Fl, Fh);
  }
  __device__ __forceinline__ void load_any(int i, double x, int E) {
    const long long F = fixed_any<7>(x, E);
    g[i] = bias((uint32_t)F, (uint32_t)(F >> 32));
  }
  template <int s>
  __device__ __forceinline__ float digit(uint2 v) const {
    constexpr int b = 6 - s;
    // the leading digit has nine bits (it reaches +128)
    constexpr uint32_t sel = s == 0 ? 0x7432u : (0x7540u | (uint32_t)(b & 3));
    const uint32_t t = __byte_perm(b < 4 ? v.x : v.y, 0x4B000000u, sel);
    // 0x4B000000 + u is 2^23 + u; minus its bias, scaled by 2^-8s (exact)
    const float off = s == 0 ? -8388608.0f : -8388736.0f;
    return fmaf(__uint_as_float(t), pow2f(-8 * s), off * pow2f(-8 * s));
  }
  template <int s>
  __device__ __forceinline__ void plane(uint32_t (&w)[4]) {
    if (s == 0) {  // the leading digit carries no bias: signed 16 bits
#pragma unroll
      for (int i = 0; i < 4; ++i)
        w[i] = __byte_perm(__float_as_uint((float)((int)g[2 * i].y >> 16)),
                           __float_as_uint((float)((int)g[2 * i + 1].y >> 16)), 0x7632);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        w[i] = __byte_perm(__float_as_uint(digit<s>(g[2 * i])),
                           __float_as_uint(digit<s>(g[2 * i + 1])), 0x7632);
    }
  }
};

// UMMA shared-memory descriptor: K-major, no swizzle.  lbo: byte distance of
// K-adjacent core matrices, sbo: byte distance of M/N-adjacent core matrices.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version for the sm_100 family
  return d;                // base offset 0, layout type 0 (no swizzle)
}

// Instruction descriptor, kind::f16: BF16 A and B (K-major), FP32 accumulator.
__host__ __device__ constexpr uint32_t instr_desc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float v[4]) {
  uint32_t r[4];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = __uint_as_float(r[i]);
}

// One lane of the (converged) warp.  An elected lane, unlike a test of the
// thread index, is known to be the only one, so MMA operands stay in uniform
// registers instead of being moved there lane by lane.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.b32 %0, 1, 0, P;\n\t}\n"
      : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ void mbar_init(uint32_t a, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(a), "r"(count));
}

// Bounded wait for the completion of the mbarrier phase with the given parity
// (at most `limit` polls); false when it ran out.
__device__ __forceinline__ bool mbar_wait(uint32_t a, uint32_t parity, int limit = kSpin) {
  uint32_t done = 0;
  for (int spin = 0; spin < limit && !done; ++spin)
    asm volatile(
        "{\n\t.reg .pred P;\n\tmbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, P;\n\t}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
  return done != 0;
}

__device__ __forceinline__ void mma_commit(uint32_t mbar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(mbar)
      : "memory");
}

__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                   dst_smem),
               "r"(kTmemCols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t tmem) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
               "r"(kTmemCols));
}

// v * 2^e in FP64 for the usual case |v| < 2^51 and a normal result: the
// integer is added to the bits of 1.5 * 2^52, one FP64 subtraction (exact)
// normalises it, and the exponent field takes e.  One FP64 instruction per
// output is pipe time that nothing else uses and replaces a 64-bit leading
// zero count, two variable shifts and a rounding.
__device__ __forceinline__ double i64_scaled(long long v, int e) {
  const int hi = (int)(v >> 32);
  if ((unsigned)(hi + 0x00080000) < 0x00100000u) {
    const double d = __hiloint2double(hi + 0x43380000, (int)v) - 6755399441055744.0;
    const int dh = __double2hiint(d);
    if ((unsigned)(((dh >> 20) & 0x7FF) + e - 1) < 2046u && v != 0)
      return __hiloint2double(dh + (int)((unsigned)e << 20), __double2loint(d));
  }
  return int_to_double(v, e);
}

// v * 2^e + y0, aligned in 62 bits and rounded once; integer operations only.
__device__ __noinline__ double i64_scaled_sum(long long v, int e, double y0) {
  long long my;
  int ey;
  double_parts(y0, my, ey);
  if (my == 0) return int_to_double(v, e);
  const int base = max(e + bitlen(v), ey + bitlen(my)) - 61;
  auto shifted = [&](long long m, int k) {
    return k >= 0 ? m << k : (k < -62 ? 0LL : m >> -k);
  };
  return int_to_double(shifted(v, e - base) + shifted(my, ey - base), base);
}

// v * 2^e + y0 with one rounding: below 2^53 the integer is a double as it stands
// (always so over one block of 256 columns: levels below 2^52 + 2^45), above it
// would be rounded before Y0 joins.
__device__ __forceinline__ double i64_scaled_plus(long long v, int e, double y0) {
  if ((unsigned long long)(v + (1LL << 53)) <= (1ULL << 54)) return i64_scaled(v, e) + y0;
  return i64_scaled_sum(v, e, y0);
}

// float -> int without the conversion unit (which takes 16 values per clock
// and SM): f + kMagic for |f| <= 2^22 holds the integer nearest f in its low
// mantissa bits, as_int(f + kMagic) - kMagicInt.
constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23
constexpr int kMagicInt = 0x4B400000;

// Exact int64 value (units 2^-kFrac of the level-0 unit) of the accumulators
// of one output: levels 0..2 (and 3 for S = 7) are exact FP32 integers in
// their units (< 2^24), the last accumulator is rounded at 2^-kFrac.  Four conversions per output would bound the drain of TMEM
// (32 cycles per warp and output on the conversion unit), during which the
// tensor core waits, so levels 0 and 1 go through the FP32 adder: level 0 is an
// integer of at most 2^22, level 1 of at most 2^23 in units of 2^-8, split into
// 2 h + l.  The integer offsets of the magic constant leave by one constant.
template <int S, int kF = kFrac>
__device__ __forceinline__ long long acc_sum(const float (&v)[5]) {
  constexpr int NA = nacc<S>();
  static_assert(NA >= 3, "levels 0 and 1 have accumulators of their own");
  const float hm = fmaf(v[1], 128.0f, kMagic), h = hm - kMagic;
  const float lm = fmaf(v[1], 256.0f, -2.0f * h) + kMagic;
  const int i0 = __float_as_int(v[0] + kMagic);
  const int i1 = 2 * __float_as_int(hm) + __float_as_int(lm);  // modulo 2^32, offset below
  long long T = 0;
#pragma unroll
  for (int a = NA - 1; a >= 2; --a) {
    const bool last = (a == NA - 1) && (S >= 4);
    const int sc = last ? kF : 8 * a;
    const int i = __float2int_rn(v[a] * __uint_as_float((uint32_t)(127 + sc) << 23));
    asm("mad.wide.s32 %0, %1, %2, %0;\n" : "+l"(T) : "r"(i), "r"(last ? 1 : 1 << (kF - 8 * a)));
  }
  const int w1 = i1 - (int)(3u * (unsigned)kMagicInt);
  asm("mad.wide.s32 %0, %1, %2, %0;\n" : "+l"(T) : "r"(w1), "r"(1 << (kF - 8)));
  const int w0 = i0 - kMagicInt;
  if (kF >= 32)
    T += (long long)(w0 * (1 << (kF >= 32 ? kF - 32 : 0))) << 32;
  else
    asm("mad.wide.s32 %0, %1, %2, %0;\n" : "+l"(T) : "r"(w0), "r"(1 << (kF < 32 ? kF : 0)));
  return T;
}

__device__ __forceinline__ void seg_col_ptr(const SegList& s, int c, const double** p,
                                            long long* ld) {
  int i = 0;
#pragma unroll
  for (int t = 1; t < kMaxSeg; ++t) i += (t < s.nseg && c >= s.off[t]) ? 1 : 0;
  *p = s.ptr[i] + (c - s.off[i]);
  *ld = s.ld[i];
}

// ------------------------------------------- shared by Gram and update kernels
constexpr int kUWarps = 16;             // compute warps
constexpr int kUThr = kUWarps * 32;
constexpr int kUThrAll = kUThr + 128;   // + a warpgroup for the MMA and the C copy warp
// Registers per thread: the launch gives every warp kURegs; the helper
// warpgroup gives most of its share to the compute warps (setmaxnreg), whose
// pending loads would otherwise be spilled, i.e. waited for.  The shares must
// add up to the launch's total.
constexpr int kURegs = 96, kURegsCompute = 104, kURegsHelper = 64;
static_assert(kUThr * kURegsCompute + (kUThrAll - kUThr) * kURegsHelper == kUThrAll * kURegs,
              "register shares must add up to the launch's registers");
constexpr int kUStagesA = 4;            // most digit stages of A in TMEM
constexpr int kUSlots = 4;              // chunks in flight; stages of C's digits in shared memory
static_assert(kUStagesA <= kUSlots, "a slot's barrier outlives its digit stage");
constexpr int kUPitch = NTMAX / 4 + 1;  // int64 slots per row and warp (odd: no bank conflicts)

// widest output tile: the accumulators leave TMEM room for two digit stages of A
template <int S>
__host__ __device__ constexpr int upd_ntmax() { return S >= 7 ? 80 : 96; }
// digit stages of A that fit beside the accumulators (8 columns per plane)
template <int S>
__host__ __device__ inline int upd_stages(int NT) {
  const int fit = ((int)kTmemCols - nacc<S>() * NT) / (8 * S);
  return fit < kUStagesA ? fit : kUStagesA;
}

__device__ __forceinline__ void tmem_st4(uint32_t taddr, uint32_t a, uint32_t b, uint32_t c,
                                         uint32_t d) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(taddr),
               "r"(a), "r"(b), "r"(c), "r"(d)
               : "memory");
}

// A from TMEM (lane = row, a 32-bit column = two consecutive K), B from shared memory
__device__ __forceinline__ void mma_bf16_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t b,
                                            uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "r"(tmem_a), "l"(b), "r"(idesc), "r"(accumulate));
}

// digit planes s .. S - 1 of 8 K values of this lane's row into TMEM
template <int S, int s>
__device__ __forceinline__ void store_planes(Split<S>& sp, uint32_t dst) {
  uint32_t w[4];
  sp.template plane<s>(w);
  tmem_st4(dst + s * 8, w[0], w[1], w[2], w[3]);
  if constexpr (s + 1 < S) store_planes<S, s + 1>(sp, dst);
}

// the same into K-major core-matrix rows in shared memory, planes pstride apart
template <int S, int s>
__device__ __forceinline__ void store_planes_shared(Split<S>& sp, uint32_t dst, uint32_t pstride) {
  uint32_t w[4];
  sp.template plane<s>(w);
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};\n" ::"r"(dst + s * pstride), "r"(w[0]),
               "r"(w[1]), "r"(w[2]), "r"(w[3])
               : "memory");
  if constexpr (s + 1 < S) store_planes_shared<S, s + 1>(sp, dst, pstride);
}

__device__ __forceinline__ void mbar_arrive(uint32_t a) {
  asm volatile("{\n\t.reg .b64 t;\n\tmbarrier.arrive.shared::cta.b64 t, [%0];\n\t}\n" ::"r"(a)
               : "memory");
}

// One poll of an mbarrier phase.
__device__ __forceinline__ bool mbar_try(uint32_t a, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred P;\n\tmbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, P;\n\t}\n"
      : "=r"(done)
      : "r"(a), "r"(parity)
      : "memory");
  return done != 0;
}

// Bounded wait that also ends when another warp of the CTA has given up;
// running out raises the CTA's failure flag.
__device__ __forceinline__ bool wait_or_fail(uint32_t bar, uint32_t parity, int* fail) {
  if (mbar_try(bar, parity)) return true;
  for (int spin = 0; spin < kSpin; spin += 64) {
    if (mbar_wait(bar, parity, 64)) return true;
    if (*reinterpret_cast<volatile int*>(fail)) return false;
  }
  *reinterpret_cast<volatile int*>(fail) = 1;
  return false;
}

// ------------------------------------------------------------------- Gram
// Rows that share one exponent per column: 256 (the bound of the exact levels),
// 64 when 256 would leave CTAs without a block.
struct GramPlan {
  int ntq, NT;        // column tiles of V and their width
  int cpb;            // chunks per exponent block
  int64_t nblk, per;  // blocks in all, blocks per slab
  int slabs;
};

// Fraction bits of the int64 sums of a Gram: with seven slices the rounding of
// each block at 2^-30 would show (the last accumulator, below 2^-7 there, leaves
// room for more); 64 blocks of at most 2^22 stay below 2^63.
template <int S>
__host__ __device__ constexpr int gram_frac() { return S >= 7 ? 34 : kFrac; }

struct GramShared {
  unsigned long long full[kUStagesA], mdone[kUStagesA];  // digits written / multiplied
  unsigned long long accfull, accempty;                  // accumulators of a block
  uint32_t tmem_base;
  int fail;
  int RB[NTMAX];  // reference exponents of the V columns over the slab
};

template <int S>
size_t gram_smem_bytes(int NT) {
  return (size_t)upd_stages<S>(NT) * S * planeB_bytes(NT) + (size_t)kUThr * kUPitch * 8 +
         sizeof(GramShared) + 1024 + 64;
}

// E[b][c] = exponent bound of column c over the rows of block b: the biased
// exponent maximum (at least 1) minus 1022.  One CTA per (block, 32 columns),
// lanes over columns, the block's 8 R rows dealt to its eight warps and all in
// flight at once (with a warp per block a 32-column Gram of 262,144 rows had
// 1,024 warps in all: 33 us a launch, two of them; 21 us for both now); the columns
// of U, then those of V; high words only.  __grid_constant__: indexed by segment, a
// plain parameter is copied to the stack by every thread (Gram 262,144 x 213 x 142
// 709 -> 666 us).
template <int R>
__global__ void __launch_bounds__(256) block_col_exp_kernel(int64_t n,
                                                            const __grid_constant__ SegList U, int p,
                                                            const __grid_constant__ SegList V, int q,
                                                            int* __restrict__ EU,
                                                            int* __restrict__ EV) {
  __shared__ int red[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int ub = (p + 31) / 32;
  const int64_t b = blockIdx.x;
  const bool isv = (int)blockIdx.y >= ub;
  const int c = (isv ? (int)blockIdx.y - ub : (int)blockIdx.y) * 32 + lane, nc = isv ? q : p;
  int e = 1;
  if (c < nc) {
    const double* ptr;
    long long ld;
    seg_col_ptr(isv ? V : U, c, &ptr, &ld);
    const int64_t r0 = b * 8 * R, r1 = min(n, r0 + 8 * R);
    const int* src = reinterpret_cast<const int*>(ptr + (r0 + warp) * ld) + 1;
    int hw[R];
    if (r0 + 8 * R <= n) {
#pragma unroll
      for (int i = 0; i < R; ++i) hw[i] = __ldg(src + 16 * i * ld);
    } else {
#pragma unroll
      for (int i = 0; i < R; ++i)
        hw[i] = r0 + warp + 8 * i < r1 ? __ldg(src + 16 * i * ld) : 0;
    }
#pragma unroll
    for (int i = 0; i < R; ++i) e = max(e, (hw[i] >> 20) & 0x7FF);
  }
  red[warp][lane] = e;
  __syncthreads();
  if (warp == 0 && c < nc) {
    for (int w = 1; w < 8; ++w) e = max(e, red[w][lane]);
    (isv ? EV : EU)[b * nc + c] = e - 1022;
  }
}

// One CTA per (128 columns of U, NT columns of V, row slab), built like the
// update kernel: 16 compute warps, an elected MMA thread, mbarriers and no
// CTA-wide barrier in the loop.  In a chunk of 16 rows some of the compute warps
// cut the U columns (a thread owns one column, its TMEM lane, and 8 rows) into
// digit planes in TMEM and others the V columns into planes in shared memory;
// a warp needs about 2,000 cycles for 32 x 8 values, so the work of a chunk is
// dealt over all of them in turn, and each warp's loads for its next turn are in
// flight meanwhile.  The columns' reference
// exponents over the slab are known beforehand (block_col_exp_kernel), so a
// block's sums only shift and add.  The form before this one (all digits in
// shared memory, 8 warps, one CTA barrier per chunk) took 896 us at
// n = 262,144, p = 213, q = 142; 552 us now.
template <int S>
__global__ void __launch_bounds__(kUThrAll, 1)
    ozaki_gram_tc_kernel(int64_t n, const __grid_constant__ SegList U, int p,
                         const __grid_constant__ SegList V, int q, int NT, int cpb, int64_t nblk,
                         int64_t per, const int* __restrict__ EU, const int* __restrict__ EV,
                         int4* __restrict__ partial) {
  constexpr int NA = nacc<S>();
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  const uint32_t pb = (uint32_t)planeB_bytes(NT);
  const int NSA = upd_stages<S>(NT);
  const uint32_t bS0 = smem_u32(base);
  unsigned char* after = base + (size_t)NSA * S * pb;
  long long* all_slots = reinterpret_cast<long long*>(after);
  GramShared& sh = *reinterpret_cast<GramShared*>(after + (size_t)kUThr * kUPitch * 8);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tp = blockIdx.x * TCM, tq = blockIdx.y * NT;
  const int np_ = min(TCM, p - tp), nq_ = min(NT, q - tq);
  const int64_t b0 = (int64_t)blockIdx.z * per, b1 = min(nblk, b0 + per);
  const int64_t r0 = b0 * cpb * TCK, r1 = min(n, b1 * cpb * TCK);
  const int nchunks = (int)((r1 - r0 + TCK - 1) / TCK), nb = (int)(b1 - b0);
  const int bunits = NT / 16;  // warps that cut the V columns of a chunk
  // lane quarters with U columns: the others are neither cut nor read (their
  // rows of the products hold whatever TMEM held)
  const int quarters = (np_ + 31) / 32;

  if (warp == 0) tmem_alloc(smem_u32(&sh.tmem_base));
  if (tid == 0) {
    for (int i = 0; i < kUStagesA; ++i) {
      mbar_init(smem_u32(&sh.full[i]), 2 * quarters + bunits);
      mbar_init(smem_u32(&sh.mdone[i]), 1);
    }
    mbar_init(smem_u32(&sh.accfull), 1);
    mbar_init(smem_u32(&sh.accempty), 4 * quarters);
    sh.fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n");
  }
  // columns past the tile's end repeat its last one; their sums are not stored
  if (tid < NT) {
    int R = kEZero;
    const int* e = EV + b0 * q + tq + min(tid, nq_ - 1);
#pragma unroll 8
    for (int b = 0; b < nb; ++b) R = max(R, __ldg(e + (int64_t)b * q));
    sh.RB[tid] = R;
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n");
  const uint32_t tmem = sh.tmem_base;
  const uint32_t tmemA = tmem + (uint32_t)(NA * NT);

  if (warp < kUWarps) {
    // ------------------------------------------------------ compute warps
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(kURegsCompute));
    const int qd = warp & 3, grp = warp >> 2, half = grp & 1, par = grp >> 1;
    const uint32_t lane_off = (uint32_t)(32 * qd) << 16;
    const int W = NT / 4;  // output columns of a warp
    long long* slots = all_slots + (size_t)warp * 32 * kUPitch;
    // The U columns of a quarter are cut by its four warps, each in every second
    // chunk.  The V columns are `bunits` items of 32 (column, row half) pairs; an
    // item belongs to vper warps in turn, those without U columns when they are
    // enough, so that no warp has more than it can do in the time of the MMAs.
    const bool cuts_u = qd < quarters;
    const int idle = 4 * (4 - quarters);
    const bool by_idle = idle >= bunits;
    // (not more than NSA warps: one that sat out longer could be two phases ahead
    // of the barrier it waits on, where the parity no longer tells them apart)
    const int vper = min((by_idle ? idle : kUWarps) / bunits, NSA);
    const int vidx = by_idle ? (qd - quarters) * 4 + grp : warp;  // place among these warps
    const bool cuts_v = vidx >= 0 && vidx < vper * bunits;
    const int vturn = cuts_v ? vidx / bunits : 0;  // cuts its item in chunks vturn mod vper
    const int item = (cuts_v ? vidx % bunits : 0) * 32 + lane;
    const int ca = min(32 * qd + lane, np_ - 1);
    const int vj = item % NT, vh = item / NT, cb = min(vj, nq_ - 1);
    const int* ea = EU + b0 * p + tp + ca;
    const int* eb = EV + b0 * q + tq + cb;
    const double *pa, *pv;
    long long lda, ldv;
    seg_col_ptr(U, tp + ca, &pa, &lda);
    seg_col_ptr(V, tq + cb, &pv, &ldv);
    // this lane's addresses in its first chunks (U: par, par + 2, ..)
    pa += (r0 + (int64_t)par * TCK + 8 * half) * lda;
    pv += (r0 + (int64_t)vturn * TCK + 8 * vh) * ldv;
    const uint32_t vdst = (uint32_t)((vh * (NT / 8) + (vj >> 3)) * 128 + (vj & 7) * 16);
    int RA = kEZero;  // reference exponent of the U column over the slab
#pragma unroll 8
    for (int b = 0; b < nb; ++b) RA = max(RA, __ldg(ea + (int64_t)b * p));
    for (int u = 0; u < W; ++u) slots[lane * kUPitch + u] = 0;

    // 8 rows of a column from row r on (zero past the slab's end)
    auto load8 = [&](const double* ptr, long long ld, int64_t r, double (&x)[8]) {
      if (r + 8 <= r1) {
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = __ldg(ptr + e * ld);
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = r + e < r1 ? __ldg(ptr + e * ld) : 0.0;
      }
    };
    auto split = [&](const double (&x)[8], int E, Split<S>& sp) {
      if (__all_sync(0xffffffffu, E > kFastEMin && E < kFastEMax)) {
        const uint32_t thr = split_thr(E);
#pragma unroll
        for (int e = 0; e < 8; ++e) sp.load(e, x[e], thr);
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e) sp.load_any(e, x[e], E);
      }
    };
    // accumulators of block b -> the warp's int64 sums
    uint32_t fphase = 0;
    auto flush = [&](int b) -> bool {
      if (!cuts_u) return true;
      // the block's distances from the references, read before the wait: lane j
      // holds that of the warp's column j
      const int si = RA - __ldg(ea + (int64_t)b * p);  // >= 0
      const int jl = W * grp + min(lane, W - 1);
      const int sl = sh.RB[jl] - __ldg(EV + (b0 + b) * q + tq + min(jl, nq_ - 1));
      if (!__all_sync(0xffffffffu, wait_or_fail(smem_u32(&sh.accfull), fphase, &sh.fail)))
        return false;
      fphase ^= 1;
      asm volatile("tcgen05.fence::after_thread_sync;\n");
#pragma unroll 1
      for (int j = 0; j < W; j += 4) {
        float v[5][4];
#pragma unroll
        for (int a = 0; a < NA; ++a) tmem_ld4(tmem + lane_off + a * NT + W * grp + j, v[a]);
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float w[5] = {v[0][e], v[1][e], v[2][e], v[3][e], v[4][e]};
          long long* slot = slots + lane * kUPitch + j + e;
          const int k = si + __shfl_sync(0xffffffffu, sl, j + e);
          long long T = acc_sum<S, gram_frac<S>()>(w);
          if (k > 0) T = k < 62 ? (T + (1LL << (k - 1))) >> k : 0;  // round to nearest
          *slot += T;
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sh.accempty));
      return true;
    };

    double xa[8], xv[8];
    if (cuts_u && par < nchunks) load8(pa, lda, r0 + (int64_t)par * TCK + 8 * half, xa);
    if (cuts_v && vturn < nchunks) load8(pv, ldv, r0 + (int64_t)vturn * TCK + 8 * vh, xv);
    // E of the block of the chunk at hand: read when a block is entered
    int Ea = __ldg(ea), Ev = __ldg(eb);
    int blk = 0, inblk = 0;    // block of chunk c and its chunk in it
    int fl = 0, fend = min(cpb, nchunks) - 1;  // next block to flush, its last chunk
    int st = 0;
    uint32_t phase = 1;
    int vnext = vturn;
    bool ok = true;
    for (int c = 0;; ++c) {
      while (ok && fl < nb && (c >= nchunks || c > fend + NSA - 1)) {
        ok = flush(fl);
        ++fl;
        fend = min(fend + cpb, nchunks - 1);
      }
      if (!ok || c >= nchunks) break;
      const bool do_u = cuts_u && (c & 1) == par, do_v = cuts_v && c == vnext;
      auto stage_free = [&]() {
        if (c >= NSA && !wait_or_fail(smem_u32(&sh.mdone[st]), phase, &sh.fail)) ok = false;
        ok = __all_sync(0xffffffffu, ok);
        return ok;
      };
      const int64_t r = r0 + (int64_t)c * TCK;
      if (do_u) {
        Split<S> sp;
        split(xa, Ea, sp);
        pa += 2 * TCK * lda;
        if (c + 2 < nchunks) load8(pa, lda, r + 2 * TCK + 8 * half, xa);
        if (!stage_free()) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        store_planes<S, 0>(sp, tmemA + lane_off + (uint32_t)(st * 8 * S + half * 4));
        asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n");
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sh.full[st]));
      }
      if (do_v) {
        Split<S> sp;
        split(xv, Ev, sp);
        vnext += vper;
        pv += (int64_t)vper * TCK * ldv;
        if (vnext < nchunks) load8(pv, ldv, r + vper * TCK + 8 * vh, xv);
        if (!stage_free()) break;
        store_planes_shared<S, 0>(sp, bS0 + (uint32_t)st * S * pb + vdst, pb);
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sh.full[st]));
      }
      if (++st == NSA) {
        st = 0;
        phase ^= 1;
      }
      if (++inblk == cpb) {
        inblk = 0;
        ++blk;
        if (blk < nb) {
          Ea = __ldg(ea + (int64_t)blk * p);
          Ev = __ldg(eb + (int64_t)blk * q);
        }
      }
    }
    // ---- slab partial: (value, exponent) = sum * 2^(R_i + R_j - 14 - kFrac), lanes
    // along the columns of V
    __syncwarp();
    const unsigned inv = 65536u / (unsigned)W + 1u;  // idx / W for idx < 768
    for (int u = 0; u < W; ++u) {
      const unsigned idx = 32u * u + lane;
      const int r = (int)((idx * inv) >> 16), j = (int)idx - r * W, jj = W * grp + j;
      const int Ri = __shfl_sync(0xffffffffu, RA, r);
      const int i = 32 * qd + r;
      if (i < np_ && jj < nq_) {
        const long long v = ok ? slots[r * kUPitch + j] : 0;
        int4 w;
        w.x = (int)(unsigned)(unsigned long long)v;
        w.y = (int)(v >> 32);
        w.z = Ri + sh.RB[jj] - 14 - gram_frac<S>();
        w.w = ok ? 0 : 1;
        partial[((int64_t)blockIdx.z * p + tp + i) * q + tq + jj] = w;
      }
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kURegsHelper));
    if (warp == kUWarps && elect_one()) {
      // -------------------------------------------------------- MMA issue
      const uint64_t pb16 = pb >> 4;
      const uint32_t idesc = instr_desc(TCM, NT);
      const uint64_t db_first = smem_desc(bS0, (uint32_t)(NT / 8) * 128, 128);
      const uint32_t full0 = smem_u32(&sh.full[0]), mdone0 = smem_u32(&sh.mdone[0]);
      int gc = 0, left = 0, st = 0;
      uint32_t blk = 0, ph = 0;
      for (; gc < nchunks; ++gc) {
        uint32_t seen = 0xFFu;
        if (left == 0) {  // a block starts: its accumulators must have been read
          seen = 0u;
          left = min(cpb, nchunks - gc);
          if (blk > 0 && !wait_or_fail(smem_u32(&sh.accempty), (blk - 1) & 1u, &sh.fail)) break;
        }
        if (!wait_or_fail(full0 + 8 * st, ph, &sh.fail)) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        const uint64_t db0 = db_first + (uint64_t)st * S * pb16;
        const uint32_t a0 = tmemA + (uint32_t)(st * 8 * S);
#pragma unroll
        for (int sl = 0; sl < S; ++sl)
#pragma unroll
          for (int tl = 0; tl + sl < S; ++tl) {
            const int a = acc_of<S>(sl + tl);
            mma_bf16_ts(tmem + (uint32_t)(a * NT), a0 + sl * 8, db0 + tl * pb16, idesc,
                        (seen >> a) & 1u);
            seen |= 1u << a;
          }
        mma_commit(mdone0 + 8 * st);
        if (--left == 0) {
          mma_commit(smem_u32(&sh.accfull));
          ++blk;
        }
        if (++st == NSA) {
          st = 0;
          ph ^= 1;
        }
      }
      // every committed MMA (and its arrival) ends before the CTA
      if (gc > 0)
        mbar_wait(smem_u32(&sh.mdone[(gc - 1) % NSA]), (uint32_t)((gc - 1) / NSA) & 1u);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    tmem_dealloc(tmem);
  }
}

// G(i, j) = sum over slabs of the int64 partials, aligned and summed in 128-bit
// integers (associative: any order gives the same bits), rounded once to FP64.
// A warp's 32 lanes are 8 slab lanes x 4 outputs: with one thread per output
// the two passes over up to 152 slabs are chains of dependent L2 loads on a few
// warps (p = q = 32: 52 us; 9 us now).
__global__ void __launch_bounds__(256) gram_tc_reduce_kernel(const int4* partial, int slabs, int p,
                                                             int q, double* G, int64_t ldg) {
  chain_wait();
  const int sl = (threadIdx.x & 31) >> 2;
  const int64_t idx =
      ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 4 + (threadIdx.x & 3);
  const bool live = idx < (int64_t)p * q;
  const int i = live ? (int)(idx / q) : 0, j = live ? (int)(idx % q) : 0;
  const int4* src = partial + (int64_t)i * q + j;
  const int64_t step = (int64_t)p * q;
  int emax = -2000000000;
  int bad = 0;
#pragma unroll 4
  for (int s = sl; s < slabs; s += 8) {
    const int4 w = src[s * step];
    bad |= w.w;
    if (w.x != 0 || w.y != 0) emax = max(emax, w.z);
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
  }
  __int128 sum = 0;
#pragma unroll 4
  for (int s = sl; s < slabs; s += 8) {
    const int4 w = src[s * step];
    const long long v = ((long long)w.y << 32) | (long long)(unsigned)w.x;
    const int k = emax - w.z;  // >= 0 wherever v != 0
    if (v != 0 && k < 100) sum += (((__int128)v) << 56) >> k;
  }
#pragma unroll
  for (int o = 4; o < 32; o <<= 1) {
    const unsigned long long lo = (unsigned long long)sum, hi = (unsigned long long)(sum >> 64);
    const unsigned long long ol = __shfl_xor_sync(0xffffffffu, lo, o),
                             oh = __shfl_xor_sync(0xffffffffu, hi, o);
    sum += (__int128)(((unsigned __int128)oh << 64) | ol);
  }
  if (sl != 0 || !live) return;
  double out = 0.0;
  if (bad) {
    out = __longlong_as_double(0x7FF8000000000000LL);
  } else if (sum != 0) {
    const bool neg = sum < 0;
    const unsigned __int128 a = neg ? (unsigned __int128)(-sum) : (unsigned __int128)sum;
    const unsigned long long hi = (unsigned long long)(a >> 64), lo = (unsigned long long)a;
    const int top = hi ? 127 - __clzll((long long)hi) : 63 - __clzll((long long)lo);
    const int sh = top > 62 ? top - 62 : 0;
    unsigned long long m = (unsigned long long)(a >> sh);
    if (sh > 0 && (a & ((((unsigned __int128)1) << sh) - 1)) != 0) m |= 1;  // sticky
    out = int_to_double(neg ? -(long long)m : (long long)m, emax - 56 + sh);
  }
  G[i + (int64_t)j * ldg] = out;
}

GramPlan gram_plan(int64_t n, int p, int q, int slices) {
  GramPlan g;
  const int ntmax = slices >= 7 ? upd_ntmax<7>() : upd_ntmax<6>();
  g.ntq = (int)ceil_div(q, ntmax);
  g.NT = (int)round_up(ceil_div(q, g.ntq), 16);
  const int64_t tiles = ceil_div(p, TCM) * g.ntq;
  g.cpb = tiles * ceil_div(n, kBlock) < 152 ? kChunksPerBlock / 4 : kChunksPerBlock;
  g.nblk = std::max<int64_t>(1, ceil_div(n, (int64_t)g.cpb * TCK));
  // one wave of CTAs; at most 64 blocks per slab keeps the int64 sums < 2^61
  int64_t s = std::max<int64_t>(ceil_div(152, tiles), ceil_div(g.nblk, 64));
  s = std::min(s, g.nblk);
  g.per = ceil_div(g.nblk, s);
  g.slabs = (int)ceil_div(g.nblk, g.per);
  return g;
}

template <int S>
int gram_tc_launch(cudaStream_t st, int64_t n, const SegList& U, int p, const SegList& V, int q,
                   const GramPlan& g, const int* EU, const int* EV, int4* partial) {
  static bool configured[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    size_t sh = 0;  // the stage count falls as the tile widens
    for (int NT = 16; NT <= upd_ntmax<S>(); NT += 16) sh = std::max(sh, gram_smem_bytes<S>(NT));
    LOB_CUDA_OK(cudaFuncSetAttribute(ozaki_gram_tc_kernel<S>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh));
    cudaFuncAttributes at;  // a launch with other registers would wait for its shares forever
    LOB_CUDA_OK(cudaFuncGetAttributes(&at, ozaki_gram_tc_kernel<S>));
    if (at.numRegs != kURegs) return LOBPCG_ERR_CUDA;
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  dim3 grid((unsigned)ceil_div(p, TCM), (unsigned)g.ntq, (unsigned)g.slabs);
  ozaki_gram_tc_kernel<S><<<grid, kUThrAll, gram_smem_bytes<S>(g.NT), st>>>(
      n, U, p, V, q, g.NT, g.cpb, g.nblk, g.per, EU, EV, partial);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

// ----------------------------------------------------------------- update
// Y = beta Y0 + alpha S C.  A = S (M = 128 rows, K = s columns; one exponent
// per row over all columns of the balanced S(i, k) 2^-colexp[k]), B = alpha C
// with rows scaled by 2^colexp[k] (one exponent per column over all k), cut
// once per call by split_c_tc_kernel into the shared-memory plane layout
// [chunk][tile][S][KG][NT/8][8][8].  Persistent CTAs walk the (row block,
// column tile) pairs; the row exponents come from a pass of their own
// (row_exp_kernel).

template <int S>
__global__ void split_c_tc_kernel(const double* __restrict__ C, int64_t ldc, int s, int m,
                                  int ntiles, int NT, double alpha, const int* __restrict__ colexp,
                                  uint16_t* __restrict__ Cs, int* __restrict__ Ce) {
  // one warp per padded column; lanes over k
  const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  const int ncols = ntiles * NT;
  if (w >= ncols) return;
  const int tile = w / NT, j = w % NT;
  const int nch = (int)ceil_div(s, TCK);
  auto val = [&](int k) -> double {
    if (w >= m || k >= s) return 0.0;
    return ldexp(alpha * C[k + (int64_t)w * ldc], colexp ? colexp[k] : 0);
  };
  int e = 0;  // biased exponent maximum; 0 = all zero
  for (int k = lane; k < s; k += 32) {
    const double x = val(k);
    if (x != 0.0) e = max(e, max((int)((__double_as_longlong(x) >> 52) & 0x7FF), 1));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, o));
  const int E = e ? e - 1022 : kEZero;
  if (lane == 0) Ce[w] = E;
  const size_t blk = (size_t)S * KG * (NT / 8) * 64;  // bf16 per (chunk, tile)
  for (int k = lane; k < nch * TCK; k += 32) {
    float d[S];
    digits<S>(val(k), E, d);
    const int ch = k / TCK, kk = k % TCK;
    uint16_t* dst = Cs + (size_t)(ch * ntiles + tile) * blk;
#pragma unroll
    for (int sl = 0; sl < S; ++sl)
      dst[(((size_t)sl * KG + (kk >> 3)) * (NT / 8) + (j >> 3)) * 64 + (j & 7) * 8 + (kk & 7)] =
          (uint16_t)(__float_as_uint(d[sl]) >> 16);
  }
}

// What is rarely needed of the finished tile whose int64 sums lie in a warp's
// slots (the rest is in registers, where more would push the pending loads out):
// its first row, and its corner in Y0 (null without Y0, or with several segments).
struct UpdOut {
  const double* y0base;
  int64_t y0ld;
  int64_t row0;
};

struct UpdShared {
  UpdOut out[kUWarps];
  // chunk g uses slot g % kUSlots: its digits of S are written and those of C
  // have arrived (full), its MMAs are done (mdone)
  unsigned long long full[kUSlots], mdone[kUSlots];
  unsigned long long accfull, accempty;  // accumulators of a K block
  uint32_t tmem_base;
  int fail;
  int cxmin, cxmax;  // range of the column exponents
};

// ER[i] = exponent bound of row i of the balanced S(i, k) 2^-colexp[k] over all
// k (kEZero for a zero row).  A warp takes kErRows rows at a time, lanes over the
// columns of each segment in turn (plain pointer arithmetic within a segment),
// the rows' loads all in flight: with one row per warp a pass over 262,144 x 32
// took 31 us against 10 us of bytes (18 us now, cold).
constexpr int kErRows = 4;
__global__ void __launch_bounds__(256) row_exp_kernel(int64_t n,
                                                      const __grid_constant__ SegList Sg, int s,
                                                      const int* __restrict__ colexp,
                                                      int* __restrict__ ER) {
  const int lane = threadIdx.x & 31;
  const int64_t row = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kErRows;
  if (row >= n) return;
  int e[kErRows];
#pragma unroll
  for (int i = 0; i < kErRows; ++i) e[i] = -1000000;
#pragma unroll
  for (int g = 0; g < kMaxSeg; ++g) {
    if (g >= Sg.nseg) break;
    const int c0 = Sg.off[g], w = Sg.off[g + 1] - c0;
    const int64_t ld = Sg.ld[g];
    const double* base = Sg.ptr[g] + row * ld;
    for (int c = lane; c < w; c += 64) {  // two columns of every row in flight
      const bool two = c + 32 < w;
      long long b0[kErRows], b1[kErRows];
#pragma unroll
      for (int i = 0; i < kErRows; ++i) {
        const bool in = row + i < n;
        b0[i] = in ? __double_as_longlong(__ldg(base + i * ld + c)) : 0LL;
        b1[i] = in && two ? __double_as_longlong(__ldg(base + i * ld + c + 32)) : 0LL;
      }
      const int x0 = colexp ? __ldg(colexp + c0 + c) : 0;
      const int x1 = (colexp && two) ? __ldg(colexp + c0 + c + 32) : 0;
#pragma unroll
      for (int i = 0; i < kErRows; ++i) {
        if ((b0[i] << 1) != 0) e[i] = max(e[i], max((int)((b0[i] >> 52) & 0x7FF), 1) - x0);
        if ((b1[i] << 1) != 0) e[i] = max(e[i], max((int)((b1[i] >> 52) & 0x7FF), 1) - x1);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < kErRows; ++i) {
    const int m = __reduce_max_sync(0xffffffffu, e[i]);
    if (lane == 0 && row + i < n) ER[row + i] = m > -1000000 ? m - 1022 : kEZero;
  }
}

template <int S>
size_t upd_smem_bytes(int NT, int s) {
  return (size_t)kUSlots * S * planeB_bytes(NT) + sizeof(UpdShared) +
         (size_t)ceil_div(std::max(s, 1), TCK) * TCK * 4 +
         (size_t)kUThr * kUPitch * 8 + 1024 + 64;
}

// One CTA per SM walks (row block, column tile) pairs; its warps hand chunks
// of 16 columns of S to one another through mbarriers, with no CTA-wide
// barrier in the loop:
//  * 16 compute warps: a thread owns one row (its TMEM lane) and cuts 8 of a
//    chunk's 16 columns, every other chunk, from global memory straight into
//    digit planes in TMEM, the A operand of tcgen05.mma; the loads of its next
//    chunk are in flight meanwhile.  At the end of a block of 256 columns it
//    moves the accumulators into int64 sums in shared memory, after having cut
//    the first chunks of the next block, and forms the outputs a few at a time
//    between the chunks that follow, so that the tensor core waits for the
//    drain of TMEM only;
//  * warp 16: an elected thread issues the S (S + 1) / 2 MMAs of a chunk (a
//    thread found by its index instead makes every operand pass through a
//    lane-by-lane move to uniform registers: 1,430 cycles a chunk, 870 so);
//  * warp 17: one thread fetches C's digits, kUSlots chunks ahead.
// The floor is the tensor pipe's 61 cycles for an M = 128, K = 16 MMA up to
// N = 80 (64 at 96), 21 of them per chunk; what bounds it is the instruction
// issue of the compute warps (about 30 per value cut, at the half rate of the
// integer pipe, 45 per output).  The form before this one (digits in shared
// memory, one CTA barrier per chunk, 64-bit shifts, the tensor core idle during
// the outputs) took 1,010 us at n = 262,144, s = 213, m = 142 and 79.0 ms at
// n = 2,097,152, s = 846, m = 564; this one 455 us and 34 ms.
// kOneBlock: s <= 256, a single block of columns; otherwise the int64 sums are
// kept in shared memory across the blocks, one slot per thread and output.
// kY0: Y0 is added (an instantiation of its own: without it the loads and
// addresses would cost the common case registers).
template <int S, bool kOneBlock, bool kY0>
__global__ void __launch_bounds__(kUThrAll, 1)
    ozaki_update_tc_kernel(int64_t n, const __grid_constant__ SegList Sg, int s,
                           const int* __restrict__ colexp, const uint16_t* __restrict__ Cs,
                           const int* __restrict__ Ce, const int* __restrict__ ER, int m,
                           int ntiles, int NT, int ntile_total,
                           const __grid_constant__ SegList Y0, const __grid_constant__ OutList Y,
                           int* status) {
  constexpr int NA = nacc<S>();
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = smem_raw + ((1024 - (smem_u32(smem_raw) & 1023)) & 1023);
  const uint32_t pb = (uint32_t)planeB_bytes(NT);
  const uint32_t bS0 = smem_u32(base);
  unsigned char* after = base + (size_t)kUSlots * S * pb;
  UpdShared& sh = *reinterpret_cast<UpdShared*>(after);
  const int nch = (s + TCK - 1) / TCK;
  int* cx = reinterpret_cast<int*>(after + ((sizeof(UpdShared) + 15) / 16) * 16);
  long long* carry = reinterpret_cast<long long*>(cx + nch * TCK);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int NSA = upd_stages<S>(NT);
  const uint32_t cs_blk = (uint32_t)S * KG * (NT / 8) * 64;  // bf16 per (chunk, tile)

  if (warp == 0) tmem_alloc(smem_u32(&sh.tmem_base));
  if (tid == 0) {
    for (int i = 0; i < kUSlots; ++i) {
      mbar_init(smem_u32(&sh.full[i]), kUWarps / 2 + 1);
      mbar_init(smem_u32(&sh.mdone[i]), 1);
    }
    mbar_init(smem_u32(&sh.accfull), 1);
    mbar_init(smem_u32(&sh.accempty), kUWarps);
    sh.fail = 0;
    sh.cxmin = sh.cxmax = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n");
  }
  __syncthreads();
  for (int k = tid; k < nch * TCK; k += kUThrAll) {
    const int v = (colexp && k < s) ? colexp[k] : 0;
    cx[k] = (int)((unsigned)v << 20);  // as the fast digits add it
    if (v < 0) atomicMin(&sh.cxmin, v);
    if (v > 0) atomicMax(&sh.cxmax, v);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n");
  const uint32_t tmem = sh.tmem_base;
  const uint32_t tmemA = tmem + (uint32_t)(NA * NT);
  const int t0 = blockIdx.x, tstep = gridDim.x;
  const int my_chunks = ((ntile_total - t0 + tstep - 1) / tstep) * nch;

  if (warp < kUWarps) {
    // ------------------------------------------------------ compute warps
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(kURegsCompute));
    const int q = warp & 3, grp = warp >> 2, half = grp & 1;
    const int rl = 32 * q + lane;
    const uint32_t lane_off = (uint32_t)(32 * q) << 16;
    const int W = NT / 4;  // output columns of a warp: W grp .. W grp + W - 1
    long long* slots = carry + (size_t)warp * 32 * kUPitch;
    // Position of this warp's next chunk: counted over the CTA's chunks (g),
    // tile t, first column k0 of its 8; the row (rows past n repeat the last
    // one), the segment holding k0 (its end, this row's address of k0, whether
    // every row's address takes 16-byte loads), and the row's exponent bound,
    // in the form of the fast digits when they can be used.
    int g = grp >> 1, t = t0, k0 = g * TCK + half * 8, segend = 0;
    const double* p = nullptr;
    bool wide = false, fast = false;
    int64_t row = 0;
    int er = 0;
    auto locate = [&]() {
      int i = 0;
#pragma unroll
      for (int u = 1; u < kMaxSeg; ++u) i += (u < Sg.nseg && k0 >= Sg.off[u]) ? 1 : 0;
      const int64_t ld = Sg.ld[i];
      p = Sg.ptr[i] + (k0 - Sg.off[i]);
      wide = ((reinterpret_cast<uintptr_t>(p) | (uintptr_t)(ld * 8)) & 15) == 0;
      p += row * ld;
      segend = Sg.off[i + 1];
    };
    auto enter_tile = [&]() {
      row = min((int64_t)(t / ntiles) * TCM + rl, n - 1);
      er = __ldg(ER + row);
      const int ef = er == kEZero ? 0 : er;  // a zero row's digits are zero for any bound
      fast = __all_sync(0xffffffffu, ef + sh.cxmin > kFastEMin && ef + sh.cxmax < kFastEMax);
      if (fast) er = (int)split_thr(ef);
      locate();
    };
    auto load8 = [&](double (&x)[8]) {
      if (k0 + 8 <= segend) {
        if (wide) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const double2 v = __ldg(reinterpret_cast<const double2*>(p) + e);
            x[2 * e] = v.x;
            x[2 * e + 1] = v.y;
          }
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) x[e] = __ldg(p + e);
        }
      } else {  // across segments, or past s
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = k0 + e < s ? seg_load(Sg, k0 + e, row) : 0.0;
      }
    };
    auto wrap = [&]() {  // k0 past the tile's chunks
      do {
        k0 -= nch * TCK;
        t += tstep;
      } while (k0 >= nch * TCK);
      if (g < my_chunks) enter_tile();
    };
    int st = g;  // digit stage of chunk g
    while (st >= NSA) st -= NSA;
    // next block of accumulators to move: tile pt, block pblk of it, ending at
    // chunk pend; parity of its barrier phases
    int pt = t0, pblk = 0, pend = min(kChunksPerBlock, nch) - 1;
    uint32_t pphase = 0;
    // output steps of the finished tile: the next one (W or more: none left),
    // rows, first column, row exponents, and its corner in Y when the warp's
    // columns go to one destination (else null)
    UpdOut& fin = sh.out[warp];
    int ou = W, onrow = 0, ocol = 0, oerow = 0, oyld = 0;
    double* ybase = nullptr;
    bool ok = true;
    double x[8];
    if (k0 >= nch * TCK) {
      wrap();
    } else if (g < my_chunks) {
      enter_tile();
    }
    if (g < my_chunks) load8(x);

    // Y = T 2^(E_row + E_col - 14 - kFrac) + beta Y0 for 32 U of the warp's 32 x W
    // outputs, lanes along the columns: a store covers two or three row
    // segments (one thread per row would touch 32 rows with every store)
    const unsigned inv = 65536u / (unsigned)W + 1u;  // idx / W for idx < 768
    auto out_steps = [&](auto U) {
      constexpr int kU = decltype(U)::value;
      long long T[kU];
      int e[kU], r[kU], j[kU];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const unsigned idx = 32u * (ou + u) + lane;
        r[u] = (int)((idx * inv) >> 16);
        j[u] = (int)idx - r[u] * W;
        e[u] = __shfl_sync(0xffffffffu, oerow, r[u] & 31);
        if (r[u] < onrow && ocol + j[u] < m) {
          T[u] = slots[r[u] * kUPitch + j[u]];
          e[u] += __ldg(Ce + ocol + j[u]);
        } else {
          r[u] = -1;
        }
      }
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        if (r[u] < 0) continue;
        double out;
        if (kY0) {
          const double* yb = fin.y0base;
          const double y0 = yb ? yb[r[u] * fin.y0ld + j[u]]
                               : seg_load(Y0, ocol + j[u], fin.row0 + r[u]);
          out = kOneBlock ? i64_scaled(T[u], e[u]) + y0 : i64_scaled_plus(T[u], e[u], y0);
        } else {
          out = i64_scaled(T[u], e[u]);
        }
        if (ybase)
          ybase[(int64_t)r[u] * oyld + j[u]] = out;
        else
          *out_addr(Y, ocol + j[u], fin.row0 + r[u]) = out;
      }
      ou += kU;
    };
    auto drain_outputs = [&]() {
      while (ou < W) out_steps(std::integral_constant<int, 2>());
    };
    // outputs are formed a few steps after each chunk, spread over the chunks of
    // the next tile, so that the tensor core never waits for them
    const int own = max(1, min(nch, kChunksPerBlock) / 2);
    const bool spread3 = W <= 3 * own;  // three steps a chunk are enough
    // With Y0 (s <= 256) a tile's outputs are formed at once, eight a thread with
    // their Y0 in flight together, the first eight since before the wait for the
    // MMAs: steps of two or three waited for Y0 each time (n = 262,144: 204 ->
    // 153 us at 32 x 32, 268 -> 235 at 96 x 32, 933 -> 744 at 213 x 142).
    constexpr int kNow = 8;
    constexpr bool kNowY0 = kOneBlock && kY0;
    double y0[kNow];
    auto load_y0 = [&](int b) {
      const int64_t row0 = (int64_t)(pt / ntiles) * TCM + 32 * q;
      const int col = (pt % ntiles) * NT + W * grp;
      const double* yb = Y0.ptr[0] + row0 * Y0.ld[0] + col;
#pragma unroll
      for (int u = 0; u < kNow; ++u) {
        const unsigned idx = 32u * (b + u) + lane;
        const int r = (int)((idx * inv) >> 16), j = (int)idx - r * W;
        y0[u] = r < 32 && row0 + r < n && col + j < m ? yb[r * Y0.ld[0] + j] : 0.0;
      }
    };
    // accumulators -> int64 sums in this warp's slots; the tensor core has TMEM
    // back before the outputs are formed
    auto flush = [&]() -> bool {
      drain_outputs();  // the previous tile's outputs leave the slots
      __syncwarp();
      const bool now = kNowY0 && Y0.nseg == 1;
      if (now) load_y0(0);
      if (!__all_sync(0xffffffffu, wait_or_fail(smem_u32(&sh.accfull), pphase, &sh.fail)))
        return false;
      asm volatile("tcgen05.fence::after_thread_sync;\n");
#pragma unroll 1
      for (int j = 0; j < W; j += 4) {
        float v[5][4];
#pragma unroll
        for (int a = 0; a < NA; ++a) tmem_ld4(tmem + lane_off + a * NT + W * grp + j, v[a]);
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float w[5] = {v[0][e], v[1][e], v[2][e], v[3][e], v[4][e]};
          long long* slot = slots + lane * kUPitch + j + e;
          long long T = acc_sum<S>(w);
          if (!kOneBlock && pblk > 0) T += *slot;
          *slot = T;
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sh.accempty));
      pphase ^= 1;
      if (++pblk * kChunksPerBlock >= nch) {  // the tile is complete
        ou = 0;
        ocol = (pt % ntiles) * NT + W * grp;
        const int64_t row0 = (int64_t)(pt / ntiles) * TCM + 32 * q;
        onrow = (int)max((int64_t)0, min((int64_t)32, n - row0));
        oerow = lane < onrow ? __ldg(ER + row0 + lane) - 14 - kFrac : 0;
        const int dst = ocol >= Y.split ? 1 : 0;
        const int64_t ld = Y.ld[dst];
        const bool plain = (dst || ocol + W <= Y.split || m <= Y.split) && ld < (1LL << 31);
        ybase = plain ? Y.ptr[dst] + row0 * ld + (ocol - dst * Y.split) : nullptr;
        oyld = (int)ld;
        if (lane == 0) {
          if (kY0) {
            fin.y0base = Y0.nseg == 1 ? Y0.ptr[0] + row0 * Y0.ld[0] + ocol : nullptr;
            fin.y0ld = Y0.ld[0];
          }
          fin.row0 = row0;
        }
        __syncwarp();
        if (now) {
          for (int b = 0; b < W; b += kNow) {
            if (b > 0) load_y0(b);
#pragma unroll
            for (int u = 0; u < kNow; ++u) {
              const unsigned idx = 32u * (b + u) + lane;
              const int r = (int)((idx * inv) >> 16), j = (int)idx - r * W;
              const int er = __shfl_sync(0xffffffffu, oerow, r & 31);
              if (r < onrow && ocol + j < m) {
                const double v =
                    i64_scaled(slots[r * kUPitch + j], er + __ldg(Ce + ocol + j)) + y0[u];
                if (ybase)
                  ybase[(int64_t)r * oyld + j] = v;
                else
                  *out_addr(Y, ocol + j, fin.row0 + r) = v;
              }
            }
          }
          ou = W;
        }
        pblk = 0;
        pt += tstep;
      }
      pend += min(kChunksPerBlock, nch - pblk * kChunksPerBlock);
      return true;
    };

    for (;;) {
      const bool more = g < my_chunks;
      // a block is moved once the digit stages that do not wait for its last
      // MMAs are filled with chunks of the next one
      while (ok && pt < ntile_total && (!more || g > pend + NSA - 1)) ok = flush();
      if (!ok || !more) break;
      // chunk g in fixed point; its registers then take the loads of chunk g + 2
      Split<S> sp;
      {
        const int4* ce = reinterpret_cast<const int4*>(cx + k0);
        const int4 c0 = ce[0], c1 = ce[1];
        const int cv[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
        if (fast) {
#pragma unroll
          for (int e = 0; e < 8; ++e) sp.load(e, x[e], (uint32_t)(er + cv[e]));
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) sp.load_any(e, x[e], er + (cv[e] >> 20));
        }
      }
      const int gc = g, sc = st;
      g += 2;
      k0 += 2 * TCK;
      p += 2 * TCK;
      st += 2;
      while (st >= NSA) st -= NSA;
      if (k0 >= nch * TCK)
        wrap();
      else if (k0 >= segend && k0 < s)
        locate();
      if (g < my_chunks) load8(x);
      // the stage is free when the MMAs of chunk gc - NSA are done
      const unsigned go = (unsigned)(gc - NSA);
      if (gc >= NSA && !wait_or_fail(smem_u32(&sh.mdone[go % kUSlots]), (go / kUSlots) & 1u, &sh.fail))
        ok = false;
      if (!(ok = __all_sync(0xffffffffu, ok))) break;
      asm volatile("tcgen05.fence::after_thread_sync;\n");
      store_planes<S, 0>(sp, tmemA + lane_off + (uint32_t)(sc * 8 * S + half * 4));
      asm volatile("tcgen05.wait::st.sync.aligned;\n" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;\n");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sh.full[(unsigned)gc % kUSlots]));
      if (ou < W) {
        if (spread3)
          out_steps(std::integral_constant<int, 3>());
        else
          drain_outputs();
      }
    }
    drain_outputs();
    if (!ok) {  // a wait ran out: the tiles not finished are marked
      for (; pt < ntile_total; pt += tstep) {
        const int tn = (pt % ntiles) * NT, nq = min(NT, m - tn);
        const int64_t row = (int64_t)(pt / ntiles) * TCM + rl;
        if (row < n)
          for (int j = grp; j < nq; j += kUWarps / 4)
            *out_addr(Y, tn + j, row) = __longlong_as_double(0x7FF8000000000000LL);
      }
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(kURegsHelper));
    if (warp == kUWarps) {
      if (elect_one()) {
        // ---------------------------------------------------------- MMA issue
        const uint64_t pb16 = pb >> 4;
        const uint32_t idesc = instr_desc(TCM, NT);
        const uint64_t db_first = smem_desc(bS0, (uint32_t)(NT / 8) * 128, 128);
        const uint32_t full0 = smem_u32(&sh.full[0]), mdone0 = smem_u32(&sh.mdone[0]);
        int gc = 0, left = 0, c = 0;  // chunks to the end of the block; chunk of the tile
        uint32_t blk = 0;
        int st = 0;
        for (; gc < my_chunks; ++gc) {
          const uint32_t slot = (uint32_t)gc % kUSlots;
          uint32_t seen = 0xFFu;
          if (left == 0) {  // a block starts: its accumulators must have been read
            seen = 0u;
            left = min(kChunksPerBlock, nch - c);
            if (blk > 0 && !wait_or_fail(smem_u32(&sh.accempty), (blk - 1) & 1u, &sh.fail)) break;
          }
          if (!wait_or_fail(full0 + 8 * slot, ((uint32_t)gc / kUSlots) & 1u, &sh.fail)) break;
          asm volatile("tcgen05.fence::after_thread_sync;\n");
          const uint64_t db0 = db_first + (uint64_t)slot * S * pb16;
          const uint32_t a0 = tmemA + (uint32_t)(st * 8 * S);
#pragma unroll
          for (int sl = 0; sl < S; ++sl)
#pragma unroll
            for (int tl = 0; tl + sl < S; ++tl) {
              const int a = acc_of<S>(sl + tl);
              mma_bf16_ts(tmem + (uint32_t)(a * NT), a0 + sl * 8, db0 + tl * pb16, idesc,
                          (seen >> a) & 1u);
              seen |= 1u << a;
            }
          mma_commit(mdone0 + 8 * slot);
          if (--left == 0) {
            mma_commit(smem_u32(&sh.accfull));
            ++blk;
          }
          if (++c == nch) c = 0;
          if (++st == NSA) st = 0;
        }
        // every committed MMA (and its arrival) ends before the CTA
        if (gc > 0)
          mbar_wait(mdone0 + 8 * ((gc - 1) % kUSlots), (uint32_t)((gc - 1) / kUSlots) & 1u);
      }
    } else if (tid == kUThr + 32) {
      // ------------------------------------------------- copies of C's digits
      const uint32_t bbytes = cs_blk * 2;
      bool ok = true;
      unsigned gc = 0;
      for (int t = t0; t < ntile_total && ok; t += tstep) {
        const int tile = t % ntiles;
        for (int c = 0; c < nch; ++c) {
          const uint32_t slot = gc % kUSlots, use = gc / kUSlots;
          if (use > 0 && !(ok = wait_or_fail(smem_u32(&sh.mdone[slot]), (use - 1) & 1u, &sh.fail)))
            break;
          const uint16_t* src = Cs + ((size_t)c * ntiles + (size_t)tile) * cs_blk;
          uint64_t state;
          asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 %0, [%1], %2;\n"
                       : "=l"(state)
                       : "r"(smem_u32(&sh.full[slot])), "r"(bbytes)
                       : "memory");
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
              "[%3];\n" ::"r"(bS0 + slot * S * pb),
              "l"(src), "r"(bbytes), "r"(smem_u32(&sh.full[slot]))
              : "memory");
          ++gc;
        }
      }
      // no copy outlives the CTA: on success the MMAs have consumed them all;
      // after a failure a copy in flight is given time to land
      if (!ok || *reinterpret_cast<volatile int*>(&sh.fail))
        for (unsigned u = gc > kUSlots ? gc - kUSlots : 0u; u < gc; ++u)
          mbar_wait(smem_u32(&sh.full[u % kUSlots]), (u / kUSlots) & 1u, 4096);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  if (tid == 0 && sh.fail && status) atomicOr(status, 1);
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    tmem_dealloc(tmem);
  }
}

template <int S>
void update_tiles(int m, int* ntiles, int* NT) {
  *ntiles = (int)ceil_div(std::max(m, 1), upd_ntmax<S>());
  *NT = (int)round_up(ceil_div(std::max(m, 1), *ntiles), 16);
}

template <int S>
int update_tc_launch(cudaStream_t st, int64_t n, const SegList& Sg, int s, const double* C,
                     int64_t ldc, int m, double alpha, double beta, const SegList& Y0,
                     const OutList& Y, const int* colexp, void* work, int* status) {
  int ntiles, NT;
  update_tiles<S>(m, &ntiles, &NT);
  const int nch = (int)ceil_div(s, TCK);
  uint16_t* Cs = (uint16_t*)work;
  const size_t cs_elems = (size_t)nch * ntiles * S * KG * (NT / 8) * 64;
  int* Ce = (int*)(Cs + cs_elems);
  int* cxw = Ce + (size_t)ntiles * NT;
  int* ER = cxw + s;
  if (!colexp) {
    int rc = column_exponents(st, n, Sg, s, cxw);
    if (rc) return rc;
    colexp = cxw;
  }
  row_exp_kernel<<<(unsigned)ceil_div(n, 8 * kErRows), 256, 0, st>>>(n, Sg, s, colexp, ER);
  LOB_LAUNCHED();
  {
    const int64_t warps = (int64_t)ntiles * NT;
    split_c_tc_kernel<S><<<(unsigned)ceil_div(warps * 32, 256), 256, 0, st>>>(
        C, ldc, s, m, ntiles, NT, alpha, colexp, Cs, Ce);
    LOB_LAUNCHED();
  }
  // the attribute is per device: set it once on every device that launches
  static bool configured[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !configured[dev]) {
    auto configure = [](auto* kernel, int one_s) -> int {
      LOB_CUDA_OK(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)upd_smem_bytes<S>(upd_ntmax<S>(), one_s)));
      cudaFuncAttributes at;  // a launch with other registers would wait for its shares forever
      LOB_CUDA_OK(cudaFuncGetAttributes(&at, kernel));
      return at.numRegs == kURegs ? LOBPCG_OK : LOBPCG_ERR_CUDA;
    };
    int rc = configure(ozaki_update_tc_kernel<S, true, false>, kBlock);
    if (!rc) rc = configure(ozaki_update_tc_kernel<S, false, false>, kMaxUpdateK);
    if (!rc) rc = configure(ozaki_update_tc_kernel<S, true, true>, kBlock);
    if (!rc) rc = configure(ozaki_update_tc_kernel<S, false, true>, kMaxUpdateK);
    if (rc) return rc;
    if (dev >= 0 && dev < 64) configured[dev] = true;
  }
  const int64_t tiles = ceil_div(n, TCM) * ntiles;
  if (tiles > (1LL << 30) || ceil_div(tiles, 152) * nch > (1LL << 30))
    return LOBPCG_ERR_ARG;  // terabytes of S
  const int64_t grid = std::min<int64_t>(tiles, 152);
  const bool one = s <= kBlock;
  const size_t sm = upd_smem_bytes<S>(NT, s);
  auto launch = [&](auto* kernel) {
    kernel<<<(unsigned)grid, kUThrAll, sm, st>>>(n, Sg, s, colexp, Cs, Ce, ER, m, ntiles, NT,
                                                 (int)tiles, Y0, Y, status);
  };
  if (beta != 0.0)
    one ? launch(ozaki_update_tc_kernel<S, true, true>)
        : launch(ozaki_update_tc_kernel<S, false, true>);
  else
    one ? launch(ozaki_update_tc_kernel<S, true, false>)
        : launch(ozaki_update_tc_kernel<S, false, false>);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

// One CTA waits on the first phase of a barrier that expects one arrival and
// gets none: the bounded wait must run out and report it in *status (bit 0),
// as the Gram and update kernels do, and the CTA must return normally.
__global__ void wait_selftest_kernel(int limit, int* status) {
  __shared__ __align__(8) unsigned long long bar;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n");
  }
  __syncthreads();
  if (threadIdx.x == 0 && !mbar_wait(smem_u32(&bar), 0u, limit)) atomicOr(status, 1);
}

}  // namespace

int wait_selftest(cudaStream_t st, int limit, int* status) {
  wait_selftest_kernel<<<1, 32, 0, st>>>(limit, status);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

int64_t gram_tc_workspace(int64_t n, int p, int q) {
  int64_t need = 0;  // for any slice count
  for (int slices : {6, 7}) {
    const GramPlan g = gram_plan(n, p, q, slices);
    need = std::max(need, (int64_t)g.slabs * p * q * (int64_t)sizeof(int4) + g.nblk * (p + q) * 4);
  }
  return need;
}

int gram_tc(cudaStream_t st, int64_t n, const SegList& U, const SegList& V, double* G,
            int64_t ldg, int slices, void* work, int64_t work_bytes) {
  const int p = U.off[U.nseg], q = V.off[V.nseg];
  if (p <= 0 || q <= 0) return LOBPCG_OK;
  if (slices == 0) slices = 6;
  if (n <= 0) return gram_ozaki(st, n, U, V, G, ldg, slices, work, work_bytes);
  if (work_bytes < gram_tc_workspace(n, p, q)) return LOBPCG_ERR_ARG;
  if (slices < 3 || slices > 7) return LOBPCG_ERR_ARG;
  const GramPlan g = gram_plan(n, p, q, slices);
  int4* partial = (int4*)work;
  int* EU = (int*)(partial + (int64_t)g.slabs * p * q);
  int* EV = EU + g.nblk * p;
  const dim3 egrid((unsigned)g.nblk, (unsigned)(ceil_div(p, 32) + ceil_div(q, 32)));
  if (g.cpb == kChunksPerBlock)
    block_col_exp_kernel<kBlock / 8><<<egrid, 256, 0, st>>>(n, U, p, V, q, EU, EV);
  else
    block_col_exp_kernel<kBlock / 32><<<egrid, 256, 0, st>>>(n, U, p, V, q, EU, EV);
  LOB_LAUNCHED();
  int rc;
  switch (slices) {
    case 3: rc = gram_tc_launch<3>(st, n, U, p, V, q, g, EU, EV, partial); break;
    case 4: rc = gram_tc_launch<4>(st, n, U, p, V, q, g, EU, EV, partial); break;
    case 5: rc = gram_tc_launch<5>(st, n, U, p, V, q, g, EU, EV, partial); break;
    case 6: rc = gram_tc_launch<6>(st, n, U, p, V, q, g, EU, EV, partial); break;
    default: rc = gram_tc_launch<7>(st, n, U, p, V, q, g, EU, EV, partial); break;
  }
  if (rc) return rc;
  const int64_t total = (int64_t)p * q;
  launch_chained(gram_tc_reduce_kernel, (unsigned)ceil_div(total, 32), 256, 0, st, partial,
                 g.slabs, p, q, G, ldg);
  LOB_LAUNCHED();
  return LOBPCG_OK;
}

int64_t update_tc_workspace(int64_t n, int s, int m, int slices) {
  if (slices == 0) slices = 6;
  int ntiles, NT;
  if (slices >= 7)
    update_tiles<7>(m, &ntiles, &NT);
  else
    update_tiles<6>(m, &ntiles, &NT);
  const int64_t nch = ceil_div(std::max(s, 1), TCK);
  return nch * ntiles * slices * KG * (NT / 8) * 64 * 2 + (int64_t)ntiles * NT * 4 +
         (int64_t)std::max(s, 1) * 4 + std::max<int64_t>(n, 1) * 4 + 256;
}

int update_tc(cudaStream_t st, int64_t n, const SegList& S, const double* C, int64_t ldc, int m,
              double alpha, double beta, const SegList& Y0, const OutList& Y, int slices,
              void* work, int64_t work_bytes, const int* colexp, int* status) {
  const int s = S.off[S.nseg];
  if (n <= 0 || m <= 0) return LOBPCG_OK;
  if (slices == 0) slices = 6;
  if (s == 0) return update_f64(st, n, S, C, ldc, m, alpha, beta, Y0, Y);
  if (s > kMaxUpdateK) return LOBPCG_ERR_ARG;
  if (work_bytes < update_tc_workspace(n, s, m, slices)) return LOBPCG_ERR_ARG;
  if (beta != 0.0 && beta != 1.0) return LOBPCG_ERR_ARG;
  switch (slices) {
    case 3: return update_tc_launch<3>(st, n, S, s, C, ldc, m, alpha, beta, Y0, Y, colexp, work, status);
    case 4: return update_tc_launch<4>(st, n, S, s, C, ldc, m, alpha, beta, Y0, Y, colexp, work, status);
    case 5: return update_tc_launch<5>(st, n, S, s, C, ldc, m, alpha, beta, Y0, Y, colexp, work, status);
    case 6: return update_tc_launch<6>(st, n, S, s, C, ldc, m, alpha, beta, Y0, Y, colexp, work, status);
    case 7: return update_tc_launch<7>(st, n, S, s, C, ldc, m, alpha, beta, Y0, Y, colexp, work, status);
    default: return LOBPCG_ERR_ARG;
  }
}

}  // namespace lob
