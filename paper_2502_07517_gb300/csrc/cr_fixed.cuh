// FP64 dot products on the integer pipe.
//
// GB300 has two FP64 FMA lanes per SM (16 cycles per warp instruction) and
// half-rate 32 x 32 + 64 bit integer multiply-adds (0.5 cycles), so a short dot
// product with constant coefficients is several times cheaper in fixed point:
// the values that enter a sum share an exponent E and become 59-bit integers,
// the coefficients of a matrix 58-bit integers with a common scale, both as two
// signed limbs of about 30 bits; three integer multiply-adds per term (the
// product of the low limbs is dropped) and one rounding at the end.  A sum over
// two lines with matrices A and B takes the exponents so that |A| |x| and |B| |y|
// have one scale, and needs no alignment.  Per term, truncating the value costs
// at most 2^-56 of max|a| times the largest value of that exponent, rounding the
// coefficient 2^-57 and the dropped product 2^-56; an FMA chain rounds every partial sum
// to 2^-53.  Against exact rational arithmetic, lines that reach that exponent have
// half of the FMA chain's mean error (tests/test_fixed_point.py); the element kernel's
// exponent is that of the element and variable, and it sees to lines further down
// (kSpareBits in cr_local64.cuh; tests/test_fixed_point_range.py).
//
// Conversions between FP64 and integers or FP32 run on the same FP64 pipe (18
// cycles), so those are done on the bit patterns as well.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

namespace crk {

#define CRK_HD __host__ __device__ __forceinline__

CRK_HD int hi_word(double x) {
#ifdef __CUDA_ARCH__
  return __double2hiint(x);
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return int(uint32_t(b >> 32));
#endif
}
CRK_HD uint32_t lo_word(double x) {
#ifdef __CUDA_ARCH__
  return uint32_t(__double2loint(x));
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return uint32_t(b);
#endif
}
CRK_HD double from_bits(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}

// Biased exponent (0x7ff: not finite).
CRK_HD int exp_of(double x) { return (hi_word(x) & 0x7fffffff) >> 20; }

// Shared exponents are kept at or above kMinLineExp (a zero then truncates to 0
// in spite of its implicit bit); values with larger ones than kMaxLineExp are
// given up as not finite (NaN results).
constexpr int kMinLineExp = 64, kMaxLineExp = 2000;

constexpr int kLimb = 29;  // bits of a low limb

// x as a fixed-point number (hi 2^29 + lo) 2^(E - 1080), truncated towards
// zero; wants an exponent of x of at most E + 1 (one bit of headroom, so that E stays
// when the values grow less than twofold).
CRK_HD int2 to_fixed(double x, int E) {
  const int h = hi_word(x);
  const uint32_t l = lo_word(x);
  const uint64_t m = (uint64_t(uint32_t((h & 0xfffff) | 0x100000)) << 38) | (uint64_t(l) << 6);
  const int d = E + 1 - ((h >> 20) & 0x7ff);
#ifdef __CUDA_ARCH__
  uint64_t t;
  asm("shr.u64 %0, %1, %2;" : "=l"(t) : "l"(m), "r"(d));  // shifts of 64 and more give 0
#else
  const uint64_t t = d > 63 ? 0 : m >> d;
#endif
  const int s = (h >> 31) | 1;
  int2 r;
  r.x = int(t >> kLimb) * s;
  r.y = int(uint32_t(t) & ((1u << kLimb) - 1)) * s;
  return r;
}

// Accumulators of a dot product: hi limbs' products, and the mixed products.
// |x| < 2^59 and |a| <= 2^58 keep 10 high and 20 mixed products below 2^63.
struct FixAcc {
  long long h, m;
};
CRK_HD void fix_mad(FixAcc& acc, int2 x, int2 a) {
  acc.h += (long long)x.x * a.x;
  acc.m += (long long)x.x * a.y;
  acc.m += (long long)x.y * a.x;
}
// (the mixed products start at half a unit, so that their shift rounds)
CRK_HD FixAcc fix_zero() { return FixAcc{0, 1ll << (kLimb - 1)}; }
CRK_HD long long fix_sum(const FixAcc& acc) { return acc.h + (acc.m >> kLimb); }

// r 2^(e - 1023) rounded to FP64 (nearest, ties away from zero), |r| < 2^63;
// results below the normal range become 0.
CRK_HD double from_fixed(long long r, int e) {
  const uint64_t s = uint64_t(r >> 63);
  uint64_t a = (uint64_t(r) ^ s) - s;
#ifdef __CUDA_ARCH__
  const int lz = __clzll((long long)a);
#else
  const int lz = a ? __builtin_clzll(a) : 64;
#endif
  const int f = e + 62 - lz;  // exponent field less one: the leading bit of a >> 11 adds it
  a <<= lz & 63;
  const uint64_t b = (uint64_t(uint32_t(f) << 20) << 32) + (a >> 11) + ((a >> 10) & 1u);
  return (f < 0 || a == 0) ? 0.0 : from_bits(b | (s << 63));
}

// Coefficients with |a| 2^scale <= 2^58 as a 30-bit and a 29-bit signed limb.
inline int2 fix_coef(double a, int scale) {
  const long long v = llrint(ldexp(a, scale));
  const long long lo = ((v + (1ll << (kLimb - 1))) & ((1ll << kLimb) - 1)) - (1ll << (kLimb - 1));
  return make_int2(int((v - lo) >> kLimb), int(lo));
}
// A coefficient times b in [0, 1], with a scale one less (truncated towards
// zero): several such sums, sum b <= 1, add up without overflow.
CRK_HD int2 fix_scaled(int2 a, double b) {
  const long long v = ((long long)a.x << kLimb) + a.y;
  const uint64_t m = uint64_t(v < 0 ? -v : v), f = uint64_t(b * 9223372036854775808.0);  // b 2^63
#ifdef __CUDA_ARCH__
  const long long t = (long long)__umul64hi(m, f);
#else
  const long long t = (long long)((unsigned __int128)m * f >> 64);
#endif
  const long long w = v < 0 ? -t : t;
  const long long lo = ((w + (1ll << (kLimb - 1))) & ((1ll << kLimb) - 1)) - (1ll << (kLimb - 1));
  return make_int2(int((w - lo) >> kLimb), int(lo));
}

// The scale for coefficients a[0..n): the largest is at least 2^57.
inline int fix_scale(const double* a, int n) {
  double m = 0.0;
  for (int i = 0; i < n; ++i) m = fmax(m, fabs(a[i]));
  int k = 0;
  if (m > 0.0 && m <= 1e300) frexp(m, &k);
  return 58 - k;
}
// Exponent offset of the result: a dot product of values with exponent E and
// coefficients of this scale is fix_sum * 2^(E + fix_exp(scale) - 1023).
CRK_HD constexpr int fix_exp(int scale) { return 1023 - 1080 + 2 * kLimb - scale; }

}  // namespace crk
