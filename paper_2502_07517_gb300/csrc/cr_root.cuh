// The scaling limiter's theta.
#pragma once
#include "cr_common.cuh"

namespace crk {

// First zero of a + b th + c th^2, which is positive at 0 and negative further on.
__device__ __forceinline__ double first_zero(double a, double b, double c) {
  const double w = sqrt_pos(b * b - 4.0 * a * c);
  return b <= 0.0 ? 2.0 * a * recip(w - b) : (b + w) * recip(-2.0 * c);
}

// The second constraint along the segment u(th) = ubar + th (pt - ubar), without its
// division and root: rho (P - eps) >= 0 as a quadratic q in th (Euler; over gamma - 1), or
// as the matrix rho (P - eps I) of three quadratics (ten-moment; q is its smaller eigenvalue,
// bounded by determinant and trace).  at(th) sets rho(th), and f and t: f >= t means that q is
// above, f <= -t that -q is above twice the rounding of the constraint as EQ::constraint
// takes it from a point of the segment plus that of f itself.
//
// That rounding, with B_v the larger magnitude of the two ends: entries of u(th) are off
// by 5 2^-53 B_v at most, so rho E - m^2 / 2 by 2^-53 (10 B_rho B_E + 7 B_m^2), and q, from its
// coefficients, by twice as much; the ten-moment eigenvalue by 2^-53 (56 .. 80) of the same
// sums over its entries.
template <class EQ> struct ConstraintOnSegment {
  static constexpr bool kEuler = IsEuler<EQ>::value;
  static constexpr int NQ = kEuler ? 1 : 3;
  double c0[NQ], c1[NQ], c2[NQ], r0, r1, noise, f, t, rho;

  __device__ __forceinline__ ConstraintOnSegment(const double* ubar, const double* pt, double eps, const Phys<double>& ph) {
    constexpr int M = EQ::M, E = kEuler ? M - 1 : 3;
    double d[M], be = 0.0, bm = 0.0;
#pragma unroll
    for (int v = 0; v < M; ++v) {
      d[v] = pt[v] - ubar[v];
      const double b = fmax(fabs(ubar[v]), fabs(pt[v]));
      if (v >= E) be += b;
      else if (v > 0) bm += b * b;
    }
    r0 = ubar[0];
    r1 = d[0];
    noise = (kEuler ? 4.440892098500626e-15 : 2.6645352591003757e-14) *  // 40, 240 2^-53
            (fmax(fabs(ubar[0]), fabs(pt[0])) * be + bm);
    if constexpr (kEuler) {
      const double e = ubar[E] - eps / ph.gm1;
      c0[0] = r0 * e;
      c1[0] = r0 * d[E] + r1 * e;
      c2[0] = r1 * d[E];
#pragma unroll
      for (int v = 1; v < E; ++v) {
        c0[0] -= 0.5 * ubar[v] * ubar[v];
        c1[0] -= ubar[v] * d[v];
        c2[0] -= 0.5 * d[v] * d[v];
      }
    } else {
#pragma unroll
      for (int k = 0; k < 3; ++k) {  // entries 11, 12, 22
        const int i = k < 2 ? 1 : 2, j = k < 1 ? 1 : 2;
        const double e = 2.0 * ubar[3 + k] - (k == 1 ? 0.0 : eps), de = 2.0 * d[3 + k];
        c0[k] = r0 * e - ubar[i] * ubar[j];
        c1[k] = r0 * de + r1 * e - (ubar[i] * d[j] + d[i] * ubar[j]);
        c2[k] = r1 * de - d[i] * d[j];
      }
    }
  }
  __device__ __forceinline__ void at(double th) {
    rho = r0 + th * r1;
    if constexpr (kEuler) {
      f = c0[0] + th * (c1[0] + th * c2[0]);
      t = noise;
    } else {
      double a[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) a[k] = c0[k] + th * (c1[k] + th * c2[k]);
      const double tr = a[0] + a[2];
      f = a[0] * a[2] - a[1] * a[1];
      t = 2.0 * noise * tr;  // |q| >= |f| / (2 tr), or |q| > tr
      if (!(tr >= noise)) {  // both eigenvalues about 0 or below: not clear
        f = -fabs(f);
        t = fabs(f) + 1.0;
      }
    }
  }
  // The zero of q between 0 and 1 (about), and how far th moves when q moves by noise.
  // Ten-moment: q is the least of x^T (rho (P - eps I)) x over unit vectors x, each a
  // quadratic in th; the zero of the one that is least at an upper bound is the next upper
  // bound (quadratic convergence, 3 or 4 steps).
  __device__ __forceinline__ double zero(double* step) const {
    double th = 1.0, b, c;
    if constexpr (kEuler) {
      b = c1[0];
      c = c2[0];
      th = first_zero(c0[0], b, c);
    } else {
      b = c = 0.0;
#pragma unroll 1
      for (int it = 0; it < 6; ++it) {
        const double q11 = c0[0] + th * (c1[0] + th * c2[0]), q12 = c0[1] + th * (c1[1] + th * c2[1]);
        const double q22 = c0[2] + th * (c1[2] + th * c2[2]), h = 0.5 * (q11 - q22);
        const double w = sqrt_pos(h * h + q12 * q12), x1 = h > 0.0 ? -q12 : w - h, x2 = h > 0.0 ? w + h : -q12;
        const double n = recip(x1 * x1 + x2 * x2), m11 = x1 * x1 * n, m12 = 2.0 * x1 * x2 * n, m22 = x2 * x2 * n;
        b = m11 * c1[0] + m12 * c1[1] + m22 * c1[2];
        c = m11 * c2[0] + m12 * c2[1] + m22 * c2[2];
        if (0.5 * (q11 + q22) - w >= -0.25 * noise) break;
        th = first_zero(m11 * c0[0] + m12 * c0[1] + m22 * c0[2], b, c);
      }
    }
    *step = noise * fabs(recip(b + 2.0 * th * c));
    return th;
  }
};

// theta of the scaling limiter (Sec. 3.2) for an admissible mean and a point with
// P_2(pt) < eps: the point that 50 bisections of [0, 1] end at, whose decisions are
// P_2(ubar + theta (pt - ubar)) >= eps as computed.  Their evaluations were most of the
// update kernel on steep ten-moment data; bit for bit the same point takes about 6
// (Euler) or 10 (ten-moment) of them where the state allows.  P_2 is concave along the
// segment, so a point at which q (ConstraintOnSegment) is clear of the rounding decides
// every bisection point on its side; the nearest clear points beside q's zero bound what
// rounding leaves open, and only there does the bisection evaluate.  Below a clear
// point L: P_2 - eps is at least the smaller of its values at 0 and L and rho the smaller
// of rho there, so both ends' q, times the ratio of the smaller rho to its own, have to be
// clear.  Above a clear point H: a bisection point c > H that is visited has 1 - c >= c -
// L, so rho(c) >= rho(H) / 2 (rho is linear and not negative) and, the constraint falling at
// least linearly, |q(c)| >= |q(H)| / 2; L stays 2^-40 away from 1 so that rho(c) is positive
// as computed.  Where nothing is clear (values near the ends of FP64's range, a mean at
// the edge of admissibility) the bisection evaluates everywhere.
//
// BULK (the result goes into FP32 values), ten-moment: q's zero is taken as it is, about 3
// evaluations, when the constraint as computed holds there and fails a few roundings
// further on.  That is where the bisection ends, up to the rounding; in FP64 states the
// difference showed (6e-16 instead of 3e-16 from 64 bits over steps on steep data).
//
// Out of line, for the registers of the limiter.
template <class EQ, bool BULK>
__device__ __noinline__ double scaling_root(const double* ubar, const double* pt, double eps, const Phys<double>& ph) {
  constexpr double kGrid = 1125899906842624.0;  // 2^50
  auto holds = [&](double th) {
    double u[EQ::M];
#pragma unroll
    for (int v = 0; v < EQ::M; ++v) u[v] = ubar[v] + th * (pt[v] - ubar[v]);
    return EQ::constraint(u, 1, ph) >= eps;
  };
  long long open_lo = 0, open_hi = 1ll << 50;  // decided: holds up to open_lo 2^-50, fails from open_hi 2^-50
  {
    ConstraintOnSegment<EQ> s(ubar, pt, eps, ph);
    double step;
    const double zero = s.zero(&step);
    if constexpr (BULK && !IsEuler<EQ>::value) {
      double th = zero, d = 0.03125 * step + 1.0 / kGrid;
      if (th > 0.0 && th + d < 1.0 && !holds(th + d)) {
#pragma unroll 1
        for (int k = 0; k < 6 && th > 0.0; ++k) {
          if (holds(th)) return th;
          th -= d;
          d *= 2.0;
        }
      }
    } else if (zero > 0.0 && zero < 1.0) {
      s.at(0.0);
      const double f0 = s.f, t0 = s.t;
      auto good = [&](double th) {  // (NaN, infinities and numbers that may have lost bits fail)
        s.at(th);
        const double have = s.f * s.r0, need = s.t * fmax(s.r0, s.rho), have0 = f0 * fmin(s.r0, s.rho), need0 = t0 * s.r0;
        const bool yes = s.rho > 0.0 && th <= 1.0 - 9.094947017729282e-13 && fmin(need, need0) > 1e-290 &&
                         fmax(have, have0) < 1e290 && have >= need && have0 >= need0;
        if (yes) open_lo = (long long)(th * kGrid);
        return yes;
      };
      auto bad = [&](double th) {
        s.at(th);
        const bool yes = s.rho > 0.0 && s.t > 1e-290 && s.f <= -s.t && s.f > -1e290;
        if (yes) open_hi = (long long)ceil(th * kGrid);
        return yes;
      };
      step = 1.25 * step + 2.0 / kGrid;
      double d = step;
#pragma unroll 1
      for (int k = 0; k < 8 && zero - d > 0.0 && !good(zero - d); ++k) d *= 2.0;
      d = step;
#pragma unroll 1
      for (int k = 0; k < 8 && zero + d < 1.0 && !bad(zero + d); ++k) d *= 2.0;
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
