// FP32 screens in front of FP64 decisions.  The FP64 pipe issues one warp
// instruction per 16 cycles and SM; a decision whose answer is clear by a margin
// above the FP32 rounding needs none of it.  Every screen answers "clear" or
// "not clear", and what is not clear is decided in FP64 as before, so the
// results do not depend on the screens.  Magnitudes outside FP32's range are never
// clear: truncation makes those from 2^128 on infinite, and every comparison asks for
// values, margins or norms well above 2^-126 (kTinyF and the bounds stated there).  (Some of it also compiles for the host:
// tests/test_screens.py holds the screens against FP64.)
#pragma once
#include "cr_common.cuh"

namespace crk {

// |relative error| allowed for an FP32 comparison of two products or speeds:
// truncated operands (2^-23 each), the approximate square root and a few FP32
// operations stay under half of it.
constexpr float kTieF = 1.9073486e-6f;  // 2^-19
// Margin of the screens below, relative to the magnitudes a value is summed
// from: ten times the FP32 rounding of those sums and products.
constexpr float kMarginF = 2e-5f;

// Magnitudes between which FP32 comparisons of truncated FP64 numbers hold: below
// 2^-126 a truncated number keeps stray bits, and products of two numbers, or of one
// and a mesh factor, stay far from both ends of FP32's range.
constexpr float kTinyF = 1e-30f, kHugeF = 1e30f;

// x as FP32, truncated, from the bit pattern (a conversion instruction runs on
// the FP64 pipe): magnitudes below FP32's normal range give a value below
// 2^-126, those from 2^128 on and NaN an infinity, with which no comparison
// against a margin of its own size holds.
__device__ __forceinline__ float trunc_f32(double x) {
  const int h = __double2hiint(x);
  const int m = max((h & 0x7fffffff) - (896 << 20), 0);
  const unsigned b = __funnelshift_l((unsigned)__double2loint(x), (unsigned)m, 3);
  return __uint_as_float((m < 0x0ff00000 ? b : 0x7f800000u) | (unsigned(h) & 0x80000000u));
}
__device__ __forceinline__ float trunc_f32(float x) { return x; }

// x as FP64 from the bit pattern (below FP32's normal range: a signed 0).
__device__ __forceinline__ double widen_f32(float x) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  const unsigned hi = (m >> 3) + (896u << 20);
  return m < 0x00800000u ? __hiloint2double(int(b & 0x80000000u), 0)
                         : __hiloint2double(int(hi | (b & 0x80000000u)), int(b << 29));
}
// double(x), from the bit pattern in FP32's normal range and for 0.
__device__ __forceinline__ double to_double(float x) {
  const unsigned m = __float_as_uint(x) & 0x7fffffffu;
  return m - 0x00800000u >= 0x7f000000u && m != 0u ? double(x) : widen_f32(x);
}
// float(x) (round to nearest, ties to even), on the bit pattern in FP32's normal
// range and for 0.  A carry out of the largest exponent leaves infinity's pattern.
__device__ __forceinline__ float to_float(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x), m = b & 0x7fffffffffffffffull;
  const unsigned s = unsigned(b >> 32) & 0x80000000u;
  if (unsigned(m >> 32) - 0x38100000u < 0x0fe00000u)
    return __uint_as_float(s | (unsigned((m + 0x0fffffffull + ((m >> 29) & 1ull)) >> 29) - (896u << 23)));
  return m == 0ull ? __uint_as_float(s) : float(x);
}
__device__ __forceinline__ float rcp_f32(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}

__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool finite_bits(float x) { return isfinite(x); }

__device__ __forceinline__ float sqrt_f32(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fmaxf(x, 0.0f)));
  return r;
#else  // (the tests: as the device's, subnormal numbers count as 0)
  return x >= 1.17549435e-38f ? sqrtf(x) : 0.0f;
#endif
}

// minmod of three slopes: the one of smallest magnitude when all three share a
// nonzero sign, else 0.
__device__ __forceinline__ float minmod3(float a, float b, float c) {
  if (a > 0.0f && b > 0.0f && c > 0.0f) return fminf(a, fminf(b, c));
  if (a < 0.0f && b < 0.0f && c < 0.0f) return fmaxf(a, fmaxf(b, c));
  return 0.0f;
}
// FP64 version on the bit patterns (integer pipe; the FP64 pipe is the scarce
// unit): sign bits must agree and no magnitude may be zero; for finite numbers
// of one sign the order of the magnitude bits is the order of the magnitudes.
__device__ __forceinline__ double minmod3(double a, double b, double c) {
  const unsigned long long ia = (unsigned long long)__double_as_longlong(a);
  const unsigned long long ib = (unsigned long long)__double_as_longlong(b);
  const unsigned long long ic = (unsigned long long)__double_as_longlong(c);
  const unsigned long long mag = 0x7fffffffffffffffull;
  const unsigned long long ma = ia & mag, mb = ib & mag, mc = ic & mag;
  if (((ia ^ ib) | (ia ^ ic)) >> 63 || ma == 0ull || mb == 0ull || mc == 0ull) return 0.0;
  unsigned long long mm = ma < mb ? ma : mb;
  mm = mm < mc ? mm : mc;
  return __longlong_as_double((long long)(mm | (ia & ~mag)));
}

// minmod of the slopes d1 b1, d2 b2, d3 b3 (b > 0) with f1, f2, f3 = b in FP32: the
// smallest is picked in FP32 where it is the smallest by kTieF and all three lie in
// the range of kTinyF, kHugeF, else in FP64.
__device__ __forceinline__ double minmod_scaled(double d1, double d2, double d3, double b1, double b2,
                                                double b3, float f1, float f2, float f3) {
  const long long i1 = __double_as_longlong(d1), i2 = __double_as_longlong(d2), i3 = __double_as_longlong(d3);
  if (((i1 ^ i2) | (i1 ^ i3)) < 0 || (i1 << 1) == 0 || (i2 << 1) == 0 || (i3 << 1) == 0) return 0.0;
  const float m1 = fabsf(trunc_f32(d1)) * f1, m2 = fabsf(trunc_f32(d2)) * f2, m3 = fabsf(trunc_f32(d3)) * f3;
  const float lim = fminf(m1, fminf(m2, m3)) * (1.0f + kTieF);
  const bool c1 = m1 <= lim, c2 = m2 <= lim, c3 = m3 <= lim;
  if (!(lim > kTinyF && m1 + m2 + m3 < kHugeF) || int(c1) + int(c2) + int(c3) != 1)
    return minmod3(d1 * b1, d2 * b2, d3 * b3);
  return (c1 ? d1 : (c2 ? d2 : d3)) * (c1 ? b1 : (c2 ? b2 : b3));
}

// max(|vL| + sqrt(cL), |vR| + sqrt(cR)), c <= 0 counted as 0: the larger side
// is picked in FP32 unless the two are within kTieF, one is infinite there, or
// both are so small that a c below 2^-126 (0 in FP32: 2^-63 in the speed) counts.
__device__ __forceinline__ double wave_max(double vL, double cL, double vR, double cR) {
  const float sL = fabsf(trunc_f32(vL)) + sqrt_f32(trunc_f32(cL));
  const float sR = fabsf(trunc_f32(vR)) + sqrt_f32(trunc_f32(cR));
  if (sL + sR > 1e-12f && fabsf(sL - sR) > kTieF * (sL + sR)) {
    const bool left = sL > sR;
    return fabs(left ? vL : vR) + sqrt_pos(left ? cL : cR);
  }
  return fmax(fabs(vL) + sqrt_pos(cL), fabs(vR) + sqrt_pos(cR));
}

// Flux in direction dir, normal velocity and squared sound speed in FP32 (see
// flux_c2; equations without a sound speed: vn is the wave speed).
template <class EQ>
__device__ __forceinline__ void flux_c2_f32(const float* u, int dir, float* f, float* vn, float* c2,
                                            const Phys<float>& ph) {
  if constexpr (IsEuler<EQ>::value) {
    const float rinv = rcp_f32(u[0]);
    float p;
    EQ::flux_r(u, dir, rinv, f, &p, ph);
    *vn = u[1 + dir] * rinv;
    *c2 = ph.gamma * p * rinv;
  } else if constexpr (EQ::M == 6) {
    const float rinv = rcp_f32(u[0]);
    EQ::flux_r(u, dir, rinv, f, ph);
    *vn = u[1 + dir] * rinv;
    *c2 = 3.0f * (2.0f * u[3 + 2 * dir] - u[1 + dir] * *vn) * rinv;
  } else {
    EQ::flux(u, dir, f, ph);
    *vn = EQ::speed(u, dir, ph);
    *c2 = 0.0f;
  }
}

// FP32 screen of the MUSCL-Hancock states: s is a state and A bounds the
// magnitudes its parts are summed from.  True only when the state is admissible
// by a margin above the FP32 rounding of the sums and products (by: more of one).  The products are
// of second order in the state (ten-moment: fourth), so their margin, too, has to be
// in FP32's range: near vacuum (rho p below 1e-25, ten-moment 1e-13) nothing is clear.
template <class EQ>
__device__ __forceinline__ bool clearly_admissible(const float* s, const float* A, float by = kMarginF) {
  if constexpr (EQ::K == 0) return true;
  if (!(s[0] > by * A[0] && A[0] > kTinyF)) return false;
  if constexpr (IsEuler<EQ>::value) {
    constexpr int E = EQ::M - 1;
    const float k2 = E == 3 ? s[1] * s[1] + s[2] * s[2] : s[1] * s[1], a2 = E == 3 ? A[1] * A[1] + A[2] * A[2] : A[1] * A[1];
    const float margin = by * (A[E] * A[0] + a2);
    return fminf(A[E], margin) > kTinyF && s[E] * s[0] - 0.5f * k2 > margin;
  } else if constexpr (EQ::M == 6) {
    const float a11 = 2.0f * s[0] * s[3] - s[1] * s[1], a22 = 2.0f * s[0] * s[5] - s[2] * s[2];
    const float a12 = 2.0f * s[0] * s[4] - s[1] * s[2], a345 = A[3] + A[4] + A[5];
    const float B = 2.0f * A[0] * a345 + A[1] * A[1] + A[2] * A[2], margin = 5.0f * kMarginF * B * B;
    const float b11 = 2.0f * A[0] * A[3] + A[1] * A[1], b22 = 2.0f * A[0] * A[5] + A[2] * A[2];  // (by: of each pressure)
    return fminf(a345, margin) > kTinyF && a11 > fmaxf(kMarginF * B, by * b11) && a22 > by * b22 && a11 * a22 - a12 * a12 > margin;
  }
  return true;
}

// Constraint k of the state s in FP32 and the bound of its error, A[v] bounding
// the magnitudes s[v] is summed from.  kTinyF covers what is below FP32's normal
// range, and in the ten-moment constraint 1e-18 what a flushed h^2 + p12^2 (2^-126)
// takes from its root.
template <class EQ>
__device__ __forceinline__ void screened_constraint(const float* s, const float* A, int k, float gm1, float* P,
                                                    float* err) {
  *P = 1.0f;
  *err = 0.0f;
  if constexpr (EQ::K > 0) {
    if (k == 0) {
      *P = s[0];
      *err = kMarginF * A[0] + kTinyF;
    } else if constexpr (IsEuler<EQ>::value) {
      constexpr int E = EQ::M - 1;
      const float r = __frcp_rn(s[0]), v1 = s[1] * r, v2 = E == 3 ? s[2] * r : 0.0f;
      float kin = s[1] * v1, e = A[E] + fabsf(v1) * A[1] + 0.5f * (v1 * v1 + v2 * v2) * A[0];
      if (E == 3) {
        kin += s[2] * v2;
        e += fabsf(v2) * A[2];
      }
      *P = gm1 * (s[E] - 0.5f * kin);
      *err = kMarginF * gm1 * e + kTinyF;
    } else {
      const float r = __frcp_rn(s[0]), v1 = s[1] * r, v2 = s[2] * r;
      const float p11 = 2.0f * s[3] - s[1] * v1, p12 = 2.0f * s[4] - s[1] * v2, p22 = 2.0f * s[5] - s[2] * v2;
      const float h = 0.5f * (p11 - p22);
      const float w = fabsf(v1) + fabsf(v2);
      *P = 0.5f * (p11 + p22) - sqrt_f32(h * h + p12 * p12);
      *err = kMarginF * (2.0f * (A[3] + A[4] + A[5]) + 2.0f * w * (A[1] + A[2]) + w * w * A[0]) + 1e-18f;
    }
  }
}

// Rusanov flux of two states in FP32, and per variable the magnitudes its rounding
// (truncated states included) is kMarginF of: besides the fluxes and jumps themselves
// the energies, of which pressures are differences, and those times the speeds; and
// what the sound speed loses in that difference, up to 1.1e-6 V^2 / c with V^2 = 2 E /
// rho (Mach 30: half of the rest).
template <class EQ>
__device__ __forceinline__ void rusanov_f32(const float* uL, const float* uR, int dir, const Phys<float>& ph, float* lo,
                                            float* a) {
  constexpr int M = EQ::M, E = M == 3 ? 2 : 3;
  float fL[M], fR[M], vL, vR, c2L, c2R;
  flux_c2_f32<EQ>(uL, dir, fL, &vL, &c2L, ph);
  flux_c2_f32<EQ>(uR, dir, fR, &vR, &c2R, ph);
  const float cL = sqrt_f32(c2L), cR = sqrt_f32(c2R);
  const float lam = fmaxf(fabsf(vL) + cL, fabsf(vR) + cR);
  float SL = 0.0f, SR = 0.0f;
#pragma unroll
  for (int v = E; v < M; ++v) {
    SL += fabsf(uL[v]);
    SR += fabsf(uR[v]);
  }
  const float S = 2.0f * (SL + SR), V2 = 2.0f * fmaxf(SL / uL[0], SR / uR[0]);
  const float V = fmaxf(lam, sqrt_f32(V2)), jump = lam + 0.03f * V2 * rcp_f32(fminf(cL, cR));
#pragma unroll
  for (int v = 0; v < M; ++v) {
    lo[v] = 0.5f * (fL[v] + fR[v]) - 0.5f * lam * (uR[v] - uL[v]);
    a[v] = fabsf(fL[v]) + fabsf(fR[v]) + jump * (fabsf(uL[v]) + fabsf(uR[v])) + (v == 0 ? 0.0f : v < E ? S : S * V);
  }
}

// Whether a node next to u's inside the element is like it: the limiter's bases in
// FP32 (hancock_states_f32) hold the subcell flux between the two, whose rounding the
// margin of the face does not see.  With the density within a factor of 2, energies at
// most twice as large and both states admissible by kLikeF (Mach 25), it is below that
// margin.
constexpr float kLikeF = 2e-3f;
template <class EQ>
__device__ __forceinline__ bool like_neighbour(int v, float u, float nb) {
  constexpr int E = EQ::M - 1;
  if (v == 0) return nb <= 2.0f * u && u <= 2.0f * nb;
  return !(v == E || (EQ::M == 6 && v == 3)) || nb <= 2.0f * u;
}

// Whether the flux limiter of an interior face is clearly idle (theta = 1) for
// the flux F: both candidates base -+ c F clear a tenth of the smaller
// low-order candidate (and those are clearly positive) in every constraint.
// uL, uR: the evolved boundary states, whose Rusanov flux is the low-order flux;
// formed in FP32 here.
template <class EQ>
__device__ __forceinline__ bool flux_limiter_idle(const float* uL, const float* uR, const float* bL, const float* bR,
                                                  const float* F, float cL, float cR, int dir,
                                                  const Phys<double>& phd) {
  constexpr int M = EQ::M;
  Phys<float> ph;
  ph.gamma = trunc_f32(phd.gamma);
  ph.gm1 = trunc_f32(phd.gm1);
  float lo[M], a[M], aL[M], aR[M];
  rusanov_f32<EQ>(uL, uR, dir, ph, lo, a);
#pragma unroll
  for (int v = 0; v < M; ++v) {
    aL[v] = fabsf(bL[v]) + cL * (a[v] + fabsf(F[v]));
    aR[v] = fabsf(bR[v]) + cR * (a[v] + fabsf(F[v]));
  }
  bool idle = fminf(cL, cR) > kTinyF;
#pragma unroll
  for (int k = 0; k < EQ::K; ++k) {
    float c[M], pl, el, pr, er, hl, fl, hr, fr;
#pragma unroll
    for (int v = 0; v < M; ++v) c[v] = bL[v] - cL * lo[v];
    screened_constraint<EQ>(c, aL, k, ph.gm1, &pl, &el);
#pragma unroll
    for (int v = 0; v < M; ++v) c[v] = bR[v] + cR * lo[v];
    screened_constraint<EQ>(c, aR, k, ph.gm1, &pr, &er);
#pragma unroll
    for (int v = 0; v < M; ++v) c[v] = bL[v] - cL * F[v];
    screened_constraint<EQ>(c, aL, k, ph.gm1, &hl, &fl);
#pragma unroll
    for (int v = 0; v < M; ++v) c[v] = bR[v] + cR * F[v];
    screened_constraint<EQ>(c, aR, k, ph.gm1, &hr, &fr);
    const float top = 0.1f * fminf(pl + el, pr + er);
    idle = idle && pl > el && pr > er && hl - fl > top && hr - fr > top;
  }
  return idle;
}

// Whether a point is clearly admissible with both constraints above 1e-12 (the
// scaling limiter's threshold is at most that).
template <class EQ>
__device__ __forceinline__ bool clearly_above_eps(const float* s, const float* A, float gm1) {
  bool ok = true;
#pragma unroll
  for (int k = 0; k < EQ::K; ++k) {
    float P, e;
    screened_constraint<EQ>(s, A, k, gm1, &P, &e);
    ok = ok && P > e + 1e-12f;
  }
  return ok;
}

}  // namespace crk
