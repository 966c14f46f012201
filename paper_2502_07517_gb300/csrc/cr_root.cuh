// The scaling limiter's theta.
#pragma once
#include "cr_common.cuh"

namespace crk {

// First zero of a + b th + c th^2, which is positive at 0 and negative further on.
__device__ __forceinline__ double first_zero(double a, double b, double c) {
  const double w = sqrt_pos(b * b - 4.0 * a * c);
  return b <= 0.0 ? 2.0 * a * recip(w - b) : (b + w) * recip(-2.0 * c);
}

// rho (P_2 - eps) / (gamma - 1) along the segment u(th) = ubar + th (pt - ubar), a quadratic q
// in th (Euler).  at(th) sets f = q(th) and rho(th).  f >= noise means that q is above, f
// <= -noise that -q is above twice the rounding of the constraint as EQ::constraint
// takes it from a point of the segment plus that of f itself: with B_v the larger
// magnitude of the two ends, entries of u(th) are off by 5 2^-53 B_v at most, so rho E -
// m^2 / 2 by 2^-53 (10 B_rho B_E + 7 B_m^2), and f, from its coefficients, by twice as much.
template <class EQ> struct EulerSegment {
  double c0, c1, c2, r0, r1, noise, f, rho;

  __device__ __forceinline__ EulerSegment(const double* ubar, const double* pt, double eps, const Phys<double>& ph) {
    constexpr int E = EQ::M - 1;
    r0 = ubar[0];
    r1 = pt[0] - ubar[0];
    const double e = ubar[E] - eps / ph.gm1, de = pt[E] - ubar[E];
    double m2 = 0.0;
    c0 = r0 * e;
    c1 = r0 * de + r1 * e;
    c2 = r1 * de;
#pragma unroll
    for (int v = 1; v < E; ++v) {
      const double d = pt[v] - ubar[v], b = fmax(fabs(ubar[v]), fabs(pt[v]));
      m2 += b * b;
      c0 -= 0.5 * ubar[v] * ubar[v];
      c1 -= ubar[v] * d;
      c2 -= 0.5 * d * d;
    }
    noise = 4.440892098500626e-15 *  // 40 2^-53
            (fmax(fabs(ubar[0]), fabs(pt[0])) * fmax(fabs(ubar[E]), fabs(pt[E])) + m2);
  }
  __device__ __forceinline__ void at(double th) {
    rho = r0 + th * r1;
    f = c0 + th * (c1 + th * c2);
  }
};

// theta of the scaling limiter (Sec. 3.2) for an admissible mean and a point with
// P_2(pt) < eps: the point that 50 bisections of [0, 1] end at, whose decisions are
// P_2(ubar + theta (pt - ubar)) >= eps as computed.  Their evaluations were most of the
// update kernel on steep ten-moment data, so most are saved:
//
// Euler: bit for bit that point, with about 6 evaluations of the constraint where the
// state allows.  P_2 is concave along the segment, so a point at which q is clear of the
// rounding decides every bisection point on its side; the nearest clear points beside
// q's zero bound what rounding leaves open, and only there does the bisection
// evaluate.  Below a clear point L: P_2 - eps is at least the smaller of its values at 0
// and L and rho the smaller of rho there, so both ends' q, times the ratio of the
// smaller rho to its own, have to be clear.  Above a clear point H: a bisection point c >
// H that is visited has 1 - c >= c - L, so rho(c) >= rho(H) / 2 (rho is linear and not
// negative) and, the constraint falling at least linearly, |q(c)| >= |q(H)| / 2; L stays
// 2^-40 away from 1 so that rho(c) is positive as computed.
//
// Ten-moment, about 3 evaluations: rho (P - eps I) is a matrix of quadratics, and q its
// smaller eigenvalue, the least of x^T (..) x over unit vectors x.  The zero of the one
// that is least at an upper bound of theta is the next upper bound (quadratic
// convergence, 3 or 4 steps).  The result is taken when the constraint as computed
// holds there and fails a few roundings further on, which is where the bisection ends,
// up to that rounding.
//
// Where either gives nothing (values near the ends of FP64's range, a mean at the edge of
// admissibility) the bisection evaluates everywhere.  Out of line, for the registers of
// the limiter.  k_update on steep ten-moment data, N = 3: FP32 bulk, 211 x 173 elements,
// 294 us with 50 evaluations each, 116 so; FP64, 256 x 256, 231 us (242 inlined).
template <class EQ>
__device__ __noinline__ double scaling_root(const double* ubar, const double* pt, double eps,
                                               const Phys<double>& ph) {
  constexpr int M = EQ::M;
  constexpr double kGrid = 1125899906842624.0;  // 2^50
  auto holds = [&](double th) {
    double u[M];
#pragma unroll
    for (int v = 0; v < M; ++v) u[v] = ubar[v] + th * (pt[v] - ubar[v]);
    return EQ::constraint(u, 1, ph) >= eps;
  };
  long long open_lo = 0, open_hi = 1ll << 50;  // decided: holds up to open_lo 2^-50, fails from open_hi 2^-50
  if constexpr (IsEuler<EQ>::value) {
    EulerSegment<EQ> s(ubar, pt, eps, ph);
    auto good = [&](double th) {  // (NaN, infinities and numbers that may have lost bits fail)
      s.at(th);
      const double have = s.f * s.r0, need = s.noise * fmax(s.r0, s.rho), have0 = s.c0 * fmin(s.r0, s.rho),
                   need0 = s.noise * s.r0;
      const bool yes = s.rho > 0.0 && th <= 1.0 - 9.094947017729282e-13 && fmin(need, need0) > 1e-290 &&
                       fmax(have, have0) < 1e290 && have >= need && have0 >= need0;
      if (yes) open_lo = (long long)(th * kGrid);
      return yes;
    };
    auto bad = [&](double th) {
      s.at(th);
      const bool yes = s.rho > 0.0 && s.noise > 1e-290 && s.f <= -s.noise && s.f > -1e290;
      if (yes) open_hi = (long long)ceil(th * kGrid);
      return yes;
    };
    const double th = first_zero(s.c0, s.c1, s.c2);
    if (th > 0.0 && th < 1.0) {
      const double step = 1.25 * s.noise * fabs(recip(s.c1 + 2.0 * th * s.c2)) + 2.0 / kGrid;
      double d = step;
#pragma unroll 1
      for (int k = 0; k < 8 && th - d > 0.0 && !good(th - d); ++k) d *= 2.0;
      d = step;
#pragma unroll 1
      for (int k = 0; k < 8 && th + d < 1.0 && !bad(th + d); ++k) d *= 2.0;
    }
  } else {
    double c0[3], c1[3], c2[3], size = 0.0;  // entries 11, 12, 22
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int i = k < 2 ? 1 : 2, j = k < 1 ? 1 : 2;
      const double r = pt[0] - ubar[0], di = pt[i] - ubar[i], dj = pt[j] - ubar[j];
      const double e = 2.0 * ubar[3 + k] - (k == 1 ? 0.0 : eps), de = 2.0 * (pt[3 + k] - ubar[3 + k]);
      c0[k] = ubar[0] * e - ubar[i] * ubar[j];
      c1[k] = ubar[0] * de + r * e - (ubar[i] * dj + di * ubar[j]);
      c2[k] = r * de - di * dj;
      if (k != 1)
        size += fmax(fabs(ubar[0]), fabs(pt[0])) * fmax(fabs(ubar[3 + k]), fabs(pt[3 + k])) +
                fmax(ubar[i] * ubar[i], pt[i] * pt[i]);
    }
    const double noise = 8.881784197001252e-16 * size;  // 8 2^-53
    double th = 1.0, b = 0.0, c = 0.0;
#pragma unroll 1
    for (int it = 0; it < 6; ++it) {
      const double q11 = c0[0] + th * (c1[0] + th * c2[0]), q12 = c0[1] + th * (c1[1] + th * c2[1]);
      const double q22 = c0[2] + th * (c1[2] + th * c2[2]), h = 0.5 * (q11 - q22);
      const double w = sqrt_pos(h * h + q12 * q12), x1 = h > 0.0 ? -q12 : w - h, x2 = h > 0.0 ? w + h : -q12;
      const double n = recip(x1 * x1 + x2 * x2), m11 = x1 * x1 * n, m12 = 2.0 * x1 * x2 * n, m22 = x2 * x2 * n;
      b = m11 * c1[0] + m12 * c1[1] + m22 * c1[2];
      c = m11 * c2[0] + m12 * c2[1] + m22 * c2[2];
      if (0.5 * (q11 + q22) - w >= -8.0 * noise) break;
      th = first_zero(m11 * c0[0] + m12 * c0[1] + m22 * c0[2], b, c);
    }
    double d = noise * fabs(recip(b + 2.0 * th * c)) + 1.0 / kGrid;
    if (th > 0.0 && th + d < 1.0 && !holds(th + d)) {
#pragma unroll 1
      for (int k = 0; k < 6 && th > 0.0; ++k) {
        if (holds(th)) return th;
        th -= d;
        d *= 2.0;
      }
    }
  }
  long long k = 0;
#pragma unroll 1
  for (int i = 49; i >= 0; --i) {
    const long long c = k + (1ll << i);
    if (c <= open_lo || (c < open_hi && holds(double(c) * (1.0 / kGrid)))) k = c;
  }
  return double(k) * (1.0 / kGrid);
}

}  // namespace crk
