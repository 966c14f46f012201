// The FP64 element kernel in two dimensions (the body that k_local and the
// batched kernels run for real = double, DIM = 2): the same phases and the same
// outputs as local_body, arranged for the FP64 pipe.
//
// What bounds it: GB300 issues one FP64 warp instruction per SM every 16
// cycles, against two integer or FP32 ones per cycle, and the pipe was 90% busy
// at 10% of the issue slots (2D Euler N = 4, 512 x 512: 12.57 ms, 1,031 FP64
// instructions per solution point).  So every FP64 instruction that integer or
// FP32 work can replace without touching the result is worth 30 of those:
//   - the D contractions (a third of the FP64 work) run in fixed point on the
//     integer pipe (cr_fixed.cuh);
//   - the trace of the time-averaged solution is the average of the stage
//     traces, which the face-node threads form anyway, and the wave speed of
//     the u^n trace shares the first stage's flux;
//   - which of the three slopes minmod takes, which of two wave speeds is the
//     larger and whether the MUSCL-Hancock states are admissible are decided in
//     FP32 where the answer is clear by a margin above the FP32 rounding, and
//     in FP64 where it is not; only the chosen slope and speed are formed;
//   - reciprocals and square roots by one third-order and two Newton steps from
//     the hardware's approximations (recip, sqrt_pos), and factors that depend
//     on the step or the node row alone formed once per block.
//   - an element that is neither blended nor beside a blended face or a boundary
//     needs its low-order scheme only for the flux limiter's inequality, which
//     the face kernel decides in FP32: there the MUSCL-Hancock states and the
//     subcell fluxes next to the faces are formed in FP32 (hancock_states_f32),
//     and the face kernel forms the FP64 data itself where the inequality is not
//     clear (exact_face_data).  The update is the same: alpha = 0 leaves the
//     high-order part alone, and theta is decided as in FP64.
// Measured (k_local, the same workload): the contractions and the first two
// groups of decisions 12.57 -> 8.42 ms (612 FP64 instructions per point), the
// low-order scheme in FP32 -> 5.60 ms; ten-moment N = 3 at 256 x 256 2.61 -> 2.03
// -> 1.56 ms.
#pragma once
#include "cr_common.cuh"
#include "cr_fixed.cuh"
#include "cr_screen.cuh"

namespace crk {

// minmod of the slopes d1 b1, d2 b2, d3 b3 (b > 0) with f1, f2, f3 = b in FP32.
__device__ __forceinline__ double minmod_scaled(double d1, double d2, double d3, double b1, double b2,
                                                double b3, float f1, float f2, float f3) {
  const long long i1 = __double_as_longlong(d1), i2 = __double_as_longlong(d2), i3 = __double_as_longlong(d3);
  if (((i1 ^ i2) | (i1 ^ i3)) < 0 || (i1 << 1) == 0 || (i2 << 1) == 0 || (i3 << 1) == 0) return 0.0;
  const float m1 = fabsf(trunc_f32(d1)) * f1, m2 = fabsf(trunc_f32(d2)) * f2, m3 = fabsf(trunc_f32(d3)) * f3;
  const float lim = fminf(m1, fminf(m2, m3)) * (1.0f + kTieF);
  const bool c1 = m1 <= lim, c2 = m2 <= lim, c3 = m3 <= lim;
  if (int(c1) + int(c2) + int(c3) != 1) return minmod3(d1 * b1, d2 * b2, d3 * b3);
  return (c1 ? d1 : (c2 ? d2 : d3)) * (c1 ? b1 : (c2 ? b2 : b3));
}

// Flux in direction dir with the normal velocity and the squared sound speed
// (the wave speed is |vn| + sqrt(c2)); equations without one: vn = the speed.
template <class EQ>
__device__ __forceinline__ void flux_c2(const double* u, int dir, double* f, double* vn, double* c2,
                                        const Phys<double>& ph) {
  if constexpr (IsEuler<EQ>::value) {
    const double rinv = recip(u[0]);
    double p;
    EQ::flux_r(u, dir, rinv, f, &p, ph);
    *vn = u[1 + dir] * rinv;
    *c2 = ph.gamma * p * rinv;
  } else if constexpr (EQ::M == 6) {
    const double rinv = recip(u[0]);
    EQ::flux_r(u, dir, rinv, f, ph);
    *vn = u[1 + dir] * rinv;
    *c2 = 3.0 * (2.0 * u[3 + 2 * dir] - u[1 + dir] * *vn) * rinv;
  } else {
    EQ::flux(u, dir, f, ph);
    *vn = EQ::speed(u, dir, ph);
    *c2 = 0.0;
  }
}

// max(|vL| + sqrt(cL), |vR| + sqrt(cR)), c <= 0 counted as 0: the larger side
// is picked in FP32 unless the two are within kTieF.
__device__ __forceinline__ double wave_max(double vL, double cL, double vR, double cR) {
  const float sL = fabsf(trunc_f32(vL)) + sqrt_f32(trunc_f32(cL));
  const float sR = fabsf(trunc_f32(vR)) + sqrt_f32(trunc_f32(cR));
  if (fabsf(sL - sR) > kTieF * (sL + sR)) {
    const bool left = sL > sR;
    return fabs(left ? vL : vR) + sqrt_pos(left ? cL : cR);
  }
  return fmax(fabs(vL) + sqrt_pos(cL), fabs(vR) + sqrt_pos(cR));
}

// Twice the Rusanov flux (the factor 1/2 goes into the caller's constants,
// exactly).
template <class EQ>
__device__ __forceinline__ void rusanov_twice(const double* uL, const double* uR, int dir, double* out,
                                              const Phys<double>& ph) {
  double fL[EQ::M], fR[EQ::M], vL, vR, cL, cR, lam;
  flux_c2<EQ>(uL, dir, fL, &vL, &cL, ph);
  flux_c2<EQ>(uR, dir, fR, &vR, &cR, ph);
  if constexpr (EQ::K > 0) lam = wave_max(vL, cL, vR, cR);
  else lam = vL;  // linear advection: the speed does not depend on the state
#pragma unroll
  for (int v = 0; v < EQ::M; ++v) out[v] = fma(-lam, uR[v] - uL[v], fL[v] + fR[v]);
}

// FP32 screen of the MUSCL-Hancock states: s is a state and A bounds the
// magnitudes its parts are summed from.  True only when the state is admissible
// by a margin above the FP32 rounding of the sums and products.
template <class EQ>
__device__ __forceinline__ bool clearly_admissible(const float* s, const float* A) {
  if constexpr (EQ::K == 0) return true;
  if (!(s[0] > kMarginF * A[0])) return false;
  if constexpr (IsEuler<EQ>::value) {
    const float q = s[3] * s[0] - 0.5f * (s[1] * s[1] + s[2] * s[2]);
    return q > kMarginF * (A[3] * A[0] + A[1] * A[1] + A[2] * A[2]);
  } else if constexpr (EQ::M == 6) {
    const float a11 = 2.0f * s[0] * s[3] - s[1] * s[1], a22 = 2.0f * s[0] * s[5] - s[2] * s[2];
    const float a12 = 2.0f * s[0] * s[4] - s[1] * s[2];
    const float B = 2.0f * A[0] * (A[3] + A[4] + A[5]) + A[1] * A[1] + A[2] * A[2];
    return a11 > kMarginF * B && a11 * a22 - a12 * a12 > 5.0f * kMarginF * B * B;
  }
  return true;
}

// MUSCL-Hancock states of one node (Sec. 4.2): the evolved states at the four
// subcell faces, or the node value where one of them is not admissible.  nb(v,
// dir, up) is the neighbour node's value along the line; hx, hy = dt / (2 w h).
template <int N, class EQ, class Nb>
__device__ __forceinline__ void hancock_states(const Mesh& m, const Phys<double>& ph, const Tab<double>& tb,
                                               const double (&un)[EQ::M], double alpha, int p, int q, double hx,
                                               double hy, Nb nb, double (&xm)[EQ::M], double (&xp)[EQ::M],
                                               double (&ym)[EQ::M], double (&yp)[EQ::M]) {
  constexpr int M = EQ::M;
#pragma unroll
  for (int v = 0; v < M; ++v) xm[v] = xp[v] = ym[v] = yp[v] = un[v];
  if (!(m.limiter & kLimMH)) return;
  const double beta = 2.0 - alpha;
  double sx[M], sy[M];
  auto slopes = [&](double (&sl)[M], int c, int dir) {
    const double bm = beta * tb.ihm[c], bc = tb.ihc[c], bp = beta * tb.ihp[c];
    const float fm = trunc_f32(bm), fc = trunc_f32(bc), fp = trunc_f32(bp);
#pragma unroll
    for (int v = 0; v < M; ++v) {
      const double um = nb(v, dir, 0), up = nb(v, dir, 1);
      sl[v] = minmod_scaled(un[v] - um, up - um, up - un[v], bm, bc, bp, fm, fc, fp);
    }
  };
  slopes(sx, p, 0);
  slopes(sy, q, 1);
  double fxm[M], fxp[M], fym[M], fyp[M], Fm[M], Fp[M], ex[M];
  vfma(fxm, tb.dm[p], sx, un);
  vfma(fxp, tb.dp[p], sx, un);
  vfma(fym, tb.dm[q], sy, un);
  vfma(fyp, tb.dp[q], sy, un);
  EQ::flux(fxm, 0, Fm, ph);
  EQ::flux(fxp, 0, Fp, ph);
  vsub(ex, Fp, Fm);
  vmul(ex, ex, hx);
  EQ::flux(fym, 1, Fm, ph);
  EQ::flux(fyp, 1, Fp, ph);
  vsub(Fp, Fp, Fm);
  vfma(ex, hy, Fp);
  bool ok = true;
  if constexpr (EQ::K > 0) {
    float uf[M], xf[M], yf[M], ef[M], A[M], st[M];
    const float dmx = trunc_f32(tb.dm[p]), dpx = trunc_f32(tb.dp[p]);
    const float dmy = trunc_f32(tb.dm[q]), dpy = trunc_f32(tb.dp[q]);
#pragma unroll
    for (int v = 0; v < M; ++v) {
      uf[v] = trunc_f32(un[v]);
      xf[v] = trunc_f32(sx[v]);
      yf[v] = trunc_f32(sy[v]);
      ef[v] = trunc_f32(ex[v]);
      A[v] = fabsf(uf[v]) + fabsf(xf[v]) + fabsf(yf[v]) + fabsf(ef[v]);
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {  // four face states, then evolved
      const float d = (c & 3) == 0 ? dmx : (c & 3) == 1 ? dpx : (c & 3) == 2 ? dmy : dpy;
#pragma unroll
      for (int v = 0; v < M; ++v) {
        st[v] = fmaf(d, (c & 2) ? yf[v] : xf[v], uf[v]);
        if (c & 4) st[v] -= ef[v];
      }
      ok = ok && clearly_admissible<EQ>(st, A);
    }
  }
  double exm[M], exp_[M], eym[M], eyp[M];
  vsub(exm, fxm, ex);
  vsub(exp_, fxp, ex);
  vsub(eym, fym, ex);
  vsub(eyp, fyp, ex);
  if (!ok)
    ok = EQ::admissible_fast(fxm, ph) && EQ::admissible_fast(fxp, ph) && EQ::admissible_fast(exm, ph) &&
         EQ::admissible_fast(exp_, ph) && EQ::admissible_fast(fym, ph) && EQ::admissible_fast(fyp, ph) &&
         EQ::admissible_fast(eym, ph) && EQ::admissible_fast(eyp, ph);
  if (ok) {
#pragma unroll
    for (int v = 0; v < M; ++v) {
      xm[v] = exm[v];
      xp[v] = exp_[v];
      ym[v] = eym[v];
      yp[v] = eyp[v];
    }
  }
}

// The same in FP32, for elements whose low-order scheme only feeds the screen of
// the flux limiter (see the body).  Returns false where admissibility is not
// clear in FP32 (the FP64 form then decides).
template <int N, class EQ, class Nb>
__device__ __forceinline__ bool hancock_states_f32(const Mesh& m, const Phys<float>& ph, const Tab<double>& tb,
                                                   const float (&un)[EQ::M], float alpha, int p, int q, float hx,
                                                   float hy, Nb nb, float (&xm)[EQ::M], float (&xp)[EQ::M],
                                                   float (&ym)[EQ::M], float (&yp)[EQ::M]) {
  constexpr int M = EQ::M;
#pragma unroll
  for (int v = 0; v < M; ++v) xm[v] = xp[v] = ym[v] = yp[v] = un[v];
  if (!(m.limiter & kLimMH)) return EQ::K == 0 || un[0] > 1e-30f;
  const float beta = 2.0f - alpha;
  float sx[M], sy[M], A[M];
  auto slopes = [&](float (&sl)[M], int c, int dir) {
    const float bm = beta * trunc_f32(tb.ihm[c]), bc = trunc_f32(tb.ihc[c]), bp = beta * trunc_f32(tb.ihp[c]);
#pragma unroll
    for (int v = 0; v < M; ++v) {
      const float um = nb(v, dir, 0), up = nb(v, dir, 1);
      sl[v] = minmod3((un[v] - um) * bm, (up - um) * bc, (up - un[v]) * bp);
    }
  };
  slopes(sx, p, 0);
  slopes(sy, q, 1);
  float Fm[M], Fp[M], ex[M], vn, c2;
  vfma(xm, trunc_f32(tb.dm[p]), sx, un);
  vfma(xp, trunc_f32(tb.dp[p]), sx, un);
  vfma(ym, trunc_f32(tb.dm[q]), sy, un);
  vfma(yp, trunc_f32(tb.dp[q]), sy, un);
  flux_c2_f32<EQ>(xm, 0, Fm, &vn, &c2, ph);
  flux_c2_f32<EQ>(xp, 0, Fp, &vn, &c2, ph);
  vsub(ex, Fp, Fm);
  vmul(ex, ex, hx);
  flux_c2_f32<EQ>(ym, 1, Fm, &vn, &c2, ph);
  flux_c2_f32<EQ>(yp, 1, Fp, &vn, &c2, ph);
  vsub(Fp, Fp, Fm);
  vfma(ex, hy, Fp);
#pragma unroll
  for (int v = 0; v < M; ++v) A[v] = fabsf(un[v]) + fabsf(sx[v]) + fabsf(sy[v]) + fabsf(ex[v]);
  bool ok = clearly_admissible<EQ>(xm, A) && clearly_admissible<EQ>(xp, A) && clearly_admissible<EQ>(ym, A) &&
            clearly_admissible<EQ>(yp, A);
  vsub(xm, xm, ex);
  vsub(xp, xp, ex);
  vsub(ym, ym, ex);
  vsub(yp, yp, ex);
  return ok && clearly_admissible<EQ>(xm, A) && clearly_admissible<EQ>(xp, A) && clearly_admissible<EQ>(ym, A) &&
         clearly_admissible<EQ>(yp, A);
}

// FP32 face data carry their density negated (their states are clearly
// admissible); a widened FP32 number also has 29 zero low bits.
__device__ __forceinline__ bool is_f32_face_data(double density) {
  return __double2hiint(density) < 0 && (__double2loint(density) & 0x1fffffff) == 0;
}

// FP64 face data in the place of FP32 ones (hancock_states_f32): the evolved
// boundary state and the limiter base of face node (side, j) of element e, from
// the state in memory into the slots.  For the face kernel, where the screen of
// the limiter leaves a face open; rare, so kept out of line.  Elements beside a
// boundary always have FP64 data and are left as they are.
template <int N, class EQ>
__device__ __noinline__ void exact_face_data(const KParams<double>& P, const Tab<double>& tb, int e, int side, int j,
                                             double dt) {
  constexpr int n = N + 1, NP = n * n, M = EQ::M;
  const Mesh& m = P.m;
#pragma unroll
  for (int f = 0; f < 4; ++f)
    if (neighbour(m, e, f) < 0) return;
  const double alpha = P.b.alpha[e];
  const int dir = side >> 1;
  double st[4][M];  // evolved states towards the face and inwards, of the boundary node and the next one
  double ub[M];
  for (int in = 0; in < 2; ++in) {
    const int c = (side & 1) ? N - in : in;
    const int p = dir == 0 ? c : j, q = dir == 0 ? j : c, k = p + n * q;
    double un[M], xm[M], xp[M], ym[M], yp[M];
#pragma unroll
    for (int v = 0; v < M; ++v) un[v] = P.b.u[((size_t)v * m.ne + e) * NP + k];
    auto nb = [&](int v, int d, int up) {
      const int cc = d == 0 ? p : q, step = d == 0 ? 1 : n;
      int ee = e, kk = k + (up ? step : -step);
      if (cc == (up ? N : 0)) {
        ee = neighbour(m, e, 2 * d + up);
        kk = k + (up ? -N : N) * step;
      }
      return P.b.u[((size_t)v * m.ne + ee) * NP + kk];
    };
    const double hx = dt * (0.5 * tb.invw[p] * P.ph.invdx), hy = dt * (0.5 * tb.invw[q] * P.ph.invdy);
    hancock_states<N, EQ>(m, P.ph, tb, un, alpha, p, q, hx, hy, nb, xm, xp, ym, yp);
#pragma unroll
    for (int v = 0; v < M; ++v) {
      const double lo = dir == 0 ? xm[v] : ym[v], hi = dir == 0 ? xp[v] : yp[v];
      st[2 * in][v] = (side & 1) ? hi : lo;
      st[2 * in + 1][v] = (side & 1) ? lo : hi;
      if (in == 0) ub[v] = un[v];
    }
  }
  double f[M];  // twice the subcell flux between the two nodes
  if (side & 1) rusanov_twice<EQ>(st[2], st[1], dir, f, P.ph);
  else rusanov_twice<EQ>(st[1], st[2], dir, f, P.ph);
  const double c = 0.5 * dt * ((side & 1) ? P.ph.cflim[side] : -P.ph.cflim[side]);
#pragma unroll
  for (int v = 0; v < M; ++v) {
    P.b.slot[slot_index(1 + 2 * M + v, side, e, j, 4, m.ne, n)] = st[0][v];
    P.b.slot[slot_index(1 + 3 * M + v, side, e, j, 4, m.ne, n)] = fma(c, f[v], ub[v]);
  }
}

// Shared memory of the body beyond the five node arrays, in bytes.
template <int N, class EQ>
__host__ __device__ constexpr size_t local64_extra(int epb) {
  constexpr int n = N + 1, S = Tableau<N>::S;
  return (size_t)epb * sizeof(double) + (size_t)(4 * n * n) * sizeof(int2) + (size_t)(S * S + 4 * n) * sizeof(double) +
         (size_t)epb * (5 + 2 * n * EQ::M) * sizeof(int);
}

template <int N, class EQ, int T>
__device__ __forceinline__ void local_body_f64(const KParams<double>& P, const Tab<double>& tb, const int blk) {
  constexpr int n = N + 1, NP = n * n, M = EQ::M, S = Tableau<N>::S, NSLOT = 4 * n;
  constexpr int SPT = (NSLOT + NP - 1) / NP;
  using TB = Tableau<N>;
  const Mesh& m = P.m;
  const Phys<double>& ph = P.ph;
  constexpr int epb = (T + NP - 1) / NP, epr = T / NP;
  const int tid = threadIdx.x;
  const int el = tid / NP, k = tid - el * NP, p = k % n, q = k / n;
  const int e = blk * epr + el;
  const bool valid = el < epr && e < m.ne;
  const int ee = valid ? e : m.ne - 1;
  const int ix = ee % m.nx, iy = ee / m.nx;

  const double dt = P.b.ctl->dt_step;
  if (!gt0(dt)) return;

  // node arrays [M][epb][NP]: u^n; the stage state, then the MUSCL-Hancock
  // states; the stage fluxes in fixed point; the time-averaged solution (for a
  // source), then the y+ states
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int stride = epb * NP, arr = M * stride;
  double* s0 = reinterpret_cast<double*>(smem_raw);
  double* sA = s0 + arr;
  double* sB = sA + arr;
  double* sC = sB + arr;
  double* sD = sC + arr;
  int2* xB = reinterpret_cast<int2*>(sB);
  int2* xC = reinterpret_cast<int2*>(sC);
  double* sAlpha = sD + arr;                                  // [epb]
  int2* tDx = reinterpret_cast<int2*>(sAlpha + epb);          // [n][n] each
  int2* tDy = tDx + n * n;
  int2* tDtx = tDy + n * n;
  int2* tDty = tDtx + n * n;
  double* sAdt = reinterpret_cast<double*>(tDty + n * n);     // dt a_ij
  double* sHx = sAdt + S * S;                                 // dt / (2 w_p dx), dt / (2 w_q dy)
  double* sHy = sHx + n;
  double* sWx = sHy + n;                                      // 1 / (2 w_p dx), 1 / (2 w_q dy)
  double* sWy = sWx + n;
  int* sNbr = reinterpret_cast<int*>(sWy + n);                // [epb][4]
  int* sKx = sNbr + epb * 4;                                  // line keys [epb][n][M]
  int* sKy = sKx + epb * n * M;
  int* sFull = sKy + epb * n * M;                             // [epb] low-order scheme in FP64

  double un[M];
#pragma unroll
  for (int v = 0; v < M; ++v) un[v] = P.b.u[((size_t)v * m.ne + ee) * NP + k];
  for (int t = tid; t < 2 * epb * n * M; t += T) sKx[t] = 0;
  for (int e2 = tid; e2 < epb; e2 += T) {
    const int eg0 = blk * epr + e2;
    const bool v2 = e2 < epr && eg0 < m.ne;
    const int eg = v2 ? eg0 : m.ne - 1;
    int nbs[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) sNbr[e2 * 4 + f] = nbs[f] = neighbour(m, eg, f);
    double al = 0.0;
    if (m.alpha_mode == 1) {
      al = m.alpha_fixed;
    } else if (m.limiter & kLimBlend) {
      al = P.b.alpha_raw[eg];
#pragma unroll
      for (int f = 0; f < 4; ++f)
        if (nbs[f] >= 0) al = fmax(al, 0.5 * P.b.alpha_raw[nbs[f]]);
    }
    sAlpha[e2] = al;
    if (v2) P.b.alpha[eg] = al;
    // An element needs its low-order scheme in FP64 when it is blended, when one
    // of its faces is (a face neighbour is blended: alpha_raw > 0 in it or in a
    // neighbour of it), or beside a boundary (those faces take the FP64 limiter
    // as it stands).  Everywhere else that scheme feeds only the flux limiter's
    // test, which FP32 answers (cr_screen.cuh; the face kernel forms the FP64
    // data itself where it does not).
    bool full = gt0(al);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      if (nbs[f] < 0) full = true;
      else if (!full && m.alpha_mode != 1 && (m.limiter & kLimBlend)) {
        full = gt0(P.b.alpha_raw[nbs[f]]);
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          const int n2 = neighbour(m, nbs[f], g);
          full = full || (n2 >= 0 && gt0(P.b.alpha_raw[n2]));
        }
      }
    }
    sFull[e2] = full;
  }
  for (int t = tid; t < n * n; t += T) {
    tDx[t] = P.ds.fDx[t];
    tDy[t] = P.ds.fDy[t];
    tDtx[t] = P.ds.fDtx[t];
    tDty[t] = P.ds.fDty[t];
  }
  // (per-block factors by threads of the last warps: the first ones smooth alpha)
  for (int t = T - 1 - tid; t < S * S + 2 * n; t += T) {
    if (t < S * S) {
      sAdt[t] = dt * TB::a(t / S, t % S);
    } else {
      const int r = t - S * S, pp = r % n;
      const double w = 0.5 * tb.invw[pp] * (r < n ? ph.invdx : ph.invdy);
      sWx[r] = w;
      sHx[r] = dt * w;
    }
  }
  vst_sh<M, stride>(s0 + tid, un);
  __syncthreads();
  const double alpha = sAlpha[el];
  const bool blend = (m.limiter & kLimBlend) || m.alpha_mode == 1;
  const bool need_lo = blend || (m.limiter & kLimFlux);
  const double a = blend ? alpha : 0.0;

  constexpr bool SRC = EQ::M == 6 || HasGravity<EQ>::value;
  const bool has_src = (EQ::M == 6 && m.source == 1) || (HasGravity<EQ>::value && m.source == 2);
  double dWx = 0.0, dWy = 0.0;
  if (HasGravity<EQ>::value && has_src) {
    dWx = m.grav[0];
    dWy = m.grav[1];
  } else if (SRC && has_src) {
    const double x = m.x0 + (ix + tb.xi[p]) * m.dx, y = m.y0 + (iy + tb.xi[q]) * m.dy;
    source_grad<2, double>(m, x - m.src_cx, y - m.src_cy, &dWx, &dWy);
  }

  // ---------------- local cRK stages -----------------------------------
  double Lst[S > 1 ? S - 1 : 1][M], Fa[M], Ga[M];
  double ea[SPT][M], Ut[SPT][M];
#pragma unroll
  for (int v = 0; v < M; ++v) {
    Fa[v] = Ga[v] = 0.0;
#pragma unroll
    for (int mm = 0; mm < SPT; ++mm) ea[mm][v] = Ut[mm][v] = 0.0;
  }
  int* const kx = sKx + (el * n + q) * M;  // this node's x-line and y-line
  int* const ky = sKy + (el * n + p) * M;
  const int line_x = el * NP + n * q, line_y = el * NP + p;

  // The x and y fluxes of this node into the line arrays in fixed point, and a
  // barrier.  A line keeps its exponent from the first stage until a value
  // needs two more bits; then (rarely: the vote) the line takes the larger one.
  auto put_lines = [&](const double (&f)[M], const double (&g)[M], bool first) {
    if (first) {
#pragma unroll
      for (int v = 0; v < M; ++v) {
        atomicMax(kx + v, mag_key(f[v]));
        atomicMax(ky + v, mag_key(g[v]));
      }
      __syncthreads();
    }
    unsigned over = 0u;  // bit 2v: f[v] outgrew its line's exponent, bit 2v + 1: g[v]
#pragma unroll
    for (int v = 0; v < M; ++v) {
      const int ex = line_exp(kx[v]), ey = line_exp(ky[v]);
      over |= (unsigned((mag_key(f[v]) >> 20) > ex + 1) << (2 * v)) | (unsigned((mag_key(g[v]) >> 20) > ey + 1) << (2 * v + 1));
      xB[v * stride + tid] = to_fixed(f[v], ex);
      xC[v * stride + tid] = to_fixed(g[v], ey);
    }
    if (first) {
      __syncthreads();
    } else if (__syncthreads_or(valid && over)) {
#pragma unroll
      for (int v = 0; v < M; ++v) {
        if ((over >> (2 * v)) & 1u) atomicMax(kx + v, mag_key(f[v]));
        if ((over >> (2 * v + 1)) & 1u) atomicMax(ky + v, mag_key(g[v]));
      }
      __syncthreads();
#pragma unroll
      for (int v = 0; v < M; ++v) {
        xB[v * stride + tid] = to_fixed(f[v], line_exp(kx[v]));
        xC[v * stride + tid] = to_fixed(g[v], line_exp(ky[v]));
      }
      __syncthreads();
    }
  };
  // sum_r Ax[p][r] f(line_x, r) + Ay[q][r] g(line_y, r) of variable v
  auto line_dot = [&](int v, const int2* Ax, const int2* Ay, int ox, int oy) -> double {
    FixAcc ax{0, 0}, ay{0, 0};
#pragma unroll
    for (int r = 0; r < n; ++r) {
      fix_mad(ax, xB[v * stride + line_x + r], Ax[p * n + r]);
      fix_mad(ay, xC[v * stride + line_y + n * r], Ay[q * n + r]);
    }
    const int ex = line_exp(kx[v]), ey = line_exp(ky[v]);
    if (max(ex, ey) > kMaxLineExp) return __longlong_as_double(0x7ff8000000000000ll);
    return from_fixed2(fix_sum(ax), ex + ox, fix_sum(ay), ey + oy);
  };

#pragma unroll
  for (int i = 0; i < S; ++i) {
    double ui[M], f[M], g[M];
#pragma unroll
    for (int v = 0; v < M; ++v) ui[v] = un[v];
#pragma unroll
    for (int j = 0; j < i; ++j)
      if (TB::a(i, j) != 0.0) vfma(ui, -sAdt[i * S + j], Lst[j]);
    EQ::flux_xy(ui, f, g, ph);
    if (TB::b(i) != 0.0) {
      vfma(Fa, TB::b(i), f);
      vfma(Ga, TB::b(i), g);
    }
    if (SRC && has_src) {  // the time-averaged solution, for its source
#pragma unroll
      for (int v = 0; v < M; ++v) {
        double* ua = sD + v * stride + tid;
        if (i == 0) *ua = TB::b(0) * ui[v];
        else if (TB::b(i) != 0.0) *ua = fma(TB::b(i), ui[v], *ua);
      }
    }
    vst_sh<M, stride>(sA + tid, ui);
    if (i < S - 1) put_lines(f, g, i == 0);
    else __syncthreads();
    if (i < S - 1) {
#pragma unroll
      for (int v = 0; v < M; ++v) Lst[i < S - 1 ? i : 0][v] = line_dot(v, tDx, tDy, P.ds.oD[0], P.ds.oD[1]);
      if (SRC && has_src) {
        double us[M], s[M];
        vld_sh<M, stride>(us, sA + tid);
        source_eval<EQ>(us, dWx, dWy, s);
#pragma unroll
        for (int v = 0; v < M; ++v) Lst[i < S - 1 ? i : 0][v] -= s[v];
      }
    }
    if (i == 0 || TB::b(i) != 0.0) {
#pragma unroll
      for (int mm = 0; mm < SPT; ++mm) {
        const FaceSlot fs = face_slot<NSLOT, n>(tid + mm * T);
        const int eg = blk * epr + fs.el;
        if (fs.el < epr && eg < m.ne) {
          const int side = fs.side, j = fs.j;
          double ut[M];
#pragma unroll
          for (int v = 0; v < M; ++v) ut[v] = 0.0;
#pragma unroll
          for (int r = 0; r < n; ++r) {
            const double l = (side & 1) ? tb.l1[r] : tb.l0[r];
            vfma_sh<M, stride>(ut, l, sA + fs.el * NP + (side < 2 ? r + n * j : j + n * r));
          }
          if (TB::b(i) != 0.0) {
            vfma(Ut[mm], TB::b(i), ut);
            if (m.dissipation == 2) {  // D-CSX: the stage trace, for the face kernel
#pragma unroll
              for (int v = 0; v < M; ++v)
                P.b.slot[slot_index(1 + 4 * M + i * M + v, side, eg, j, 4, m.ne, n)] = ut[v];
            }
          }
          if (i == 0 || m.central == 0) {
            double fn[M], vn, c2;
            flux_c2<EQ>(ut, side >> 1, fn, &vn, &c2, ph);
            if (TB::b(i) != 0.0 && m.central == 0) vfma(ea[mm], TB::b(i), fn);  // EA, eq. (evaluate)
            if (i == 0) {  // u^n trace: its wave speed, and the trace itself for D1
              P.b.slot[slot_index(0, side, eg, j, 4, m.ne, n)] = EQ::K > 0 ? fabs(vn) + sqrt_pos(c2) : vn;
              if (m.dissipation == 1) {
#pragma unroll
                for (int v = 0; v < M; ++v) P.b.slot[slot_index(1 + v, side, eg, j, 4, m.ne, n)] = ut[v];
              }
            }
          }
        }
      }
    }
    __syncthreads();
  }

  // ---------------- time averages: high-order volume part, face data ----
  if (m.central == 1) {  // AE: the averages themselves, for their traces
    vst_sh<M, stride>(sA + tid, Fa);
  }
  put_lines(Fa, Ga, false);
  double HO[M];
#pragma unroll
  for (int v = 0; v < M; ++v) HO[v] = line_dot(v, tDtx, tDty, P.ds.oDt[0], P.ds.oDt[1]);
  // HO becomes the high-order part of the update, u^n - dt (1 - a) HO + dt S,
  // with the source of the time-averaged solution (linear in u)
  const double dho = dt * (1.0 - a);
  vfma(HO, -dho, HO, un);
  if (SRC && has_src) {
    double us[M], Sa[M];
    vld_sh<M, stride>(us, sD + tid);
    source_eval<EQ>(us, dWx, dWy, Sa);
    vfma(HO, dt, Sa);
  }
#pragma unroll
  for (int mm = 0; mm < SPT; ++mm) {
    const FaceSlot fs = face_slot<NSLOT, n>(tid + mm * T);
    const int eg = blk * epr + fs.el;
    if (fs.el < epr && eg < m.ne) {
      // slots 1..M: the trace the dissipation jumps over (U; D1 stored u^n's);
      // slots 1+M..: the EA average (AE: below)
#pragma unroll
      for (int v = 0; v < M; ++v) {
        if (m.dissipation != 1) P.b.slot[slot_index(1 + v, fs.side, eg, fs.j, 4, m.ne, n)] = Ut[mm][v];
        if (m.central == 0) P.b.slot[slot_index(1 + M + v, fs.side, eg, fs.j, 4, m.ne, n)] = ea[mm][v];
      }
    }
  }
  if (m.central == 1) {  // AE, eq. (extrapolate): the trace of F on x faces, of G on y faces
    for (int dir = 0; dir < 2; ++dir) {
      if (dir == 1) {
        __syncthreads();
        vst_sh<M, stride>(sA + tid, Ga);
        __syncthreads();
      }
#pragma unroll
      for (int mm = 0; mm < SPT; ++mm) {
        const FaceSlot fs = face_slot<NSLOT, n>(tid + mm * T);
        const int eg = blk * epr + fs.el;
        if (fs.el < epr && eg < m.ne && (fs.side >> 1) == dir) {
          double Ft[M];
#pragma unroll
          for (int v = 0; v < M; ++v) Ft[v] = 0.0;
#pragma unroll
          for (int r = 0; r < n; ++r) {
            const double l = (fs.side & 1) ? tb.l1[r] : tb.l0[r];
            vfma_sh<M, stride>(Ft, l, sA + fs.el * NP + (dir == 0 ? r + n * fs.j : fs.j + n * r));
          }
#pragma unroll
          for (int v = 0; v < M; ++v) P.b.slot[slot_index(1 + M + v, fs.side, eg, fs.j, 4, m.ne, n)] = Ft[v];
        }
      }
    }
  }
  __syncthreads();

  // ---------------- MUSCL-Hancock / first-order subcells -----------------
  double LO[M];
#pragma unroll
  for (int v = 0; v < M; ++v) LO[v] = 0.0;
  if (need_lo) {
    // neighbour nodes of the line: across a face the neighbour element's, at a
    // boundary the side's ghost node (outflow: the own node; wall: its
    // reflection; Dirichlet, inflow: given)
    auto nb = [&](int v, int dir, int up) -> double {
      const int c = dir == 0 ? p : q, step = dir == 0 ? 1 : n;
      if (c != (up ? N : 0)) return s0[v * stride + tid + (up ? step : -step)];
      const int side = 2 * dir + up, e2 = sNbr[el * 4 + side];
      if (e2 >= 0) return P.b.u[((size_t)v * m.ne + e2) * NP + k + (up ? -N : N) * step];
      const int bc = m.bcs[side];
      if (bc == kBcDirichlet || bc == kBcInflow) {
        double g[M];
        ghost_at<M>(m, side, P.b.ctl->t, g);
        return g[v];
      }
      return bc == kBcWall && v == 1 + dir ? -un[v] : un[v];
    };
    auto put_exact = [&]() {
      double xm[M], xp[M], ym[M], yp[M];
      hancock_states<N, EQ>(m, ph, tb, un, alpha, p, q, sHx[p], sHy[q], nb, xm, xp, ym, yp);
      vst_sh<M, stride>(sA + tid, xm);
      vst_sh<M, stride>(sB + tid, xp);
      vst_sh<M, stride>(sC + tid, ym);
      vst_sh<M, stride>(sD + tid, yp);
    };
    // FP32 states sit in the low words of the same slots
    auto low = [&](double* base, int v) -> float& { return *reinterpret_cast<float*>(base + v * stride); };
    Phys<float> phf;
    phf.gamma = trunc_f32(ph.gamma);
    phf.gm1 = trunc_f32(ph.gm1);
    phf.ax = trunc_f32(ph.ax);
    phf.ay = trunc_f32(ph.ay);
    const bool full0 = sFull[el] != 0;
    bool unclear = false;
    if (full0) {
      put_exact();
    } else {
      float uf[M], xm[M], xp[M], ym[M], yp[M];
#pragma unroll
      for (int v = 0; v < M; ++v) uf[v] = trunc_f32(un[v]);
      auto nbf = [&](int v, int dir, int up) { return trunc_f32(nb(v, dir, up)); };
      unclear = !hancock_states_f32<N, EQ>(m, phf, tb, uf, trunc_f32(alpha), p, q, trunc_f32(sHx[p]), trunc_f32(sHy[q]),
                                           nbf, xm, xp, ym, yp);
#pragma unroll
      for (int v = 0; v < M; ++v) {
        low(sA + tid, v) = xm[v];
        low(sB + tid, v) = xp[v];
        low(sC + tid, v) = ym[v];
        low(sD + tid, v) = yp[v];
      }
      if (unclear) sFull[el] = 1;  // the whole element goes to FP64
    }
    if (__syncthreads_or(unclear)) {
      if (!full0 && sFull[el]) put_exact();
      __syncthreads();
    }
    // subcell fluxes (twice their value), numbered across the block: element r /
    // NSF, its N n x-subfaces, then its n N y-subfaces; the flux right of (above)
    // node (p2, q2) overwrites that node's x+ (y+) state, which no other reads.
    // FP32 elements need only those next to the element faces.
    constexpr int NSX = N * n, NSF = 2 * N * n;
    for (int gs = tid; gs < epr * NSF; gs += T) {
      const int el2 = gs / NSF, r = gs - el2 * NSF;
      const bool isx = r < NSX;
      const int rr = isx ? r : r - NSX;
      const int p2 = isx ? rr % N : rr % n, q2 = isx ? rr / N : rr / n;
      const int node = el2 * NP + p2 + n * q2;
      double* sL = (isx ? sB : sD) + node;
      double* sR = (isx ? sA : sC) + node + (isx ? 1 : n);
      if (sFull[el2]) {
        double uL[M], uR[M], fr[M];
        vld_sh<M, stride>(uL, sL);
        vld_sh<M, stride>(uR, sR);
        rusanov_twice<EQ>(uL, uR, isx ? 0 : 1, fr, ph);
        vst_sh<M, stride>(sL, fr);
      } else if (const int c = isx ? p2 : q2; c == 0 || c == N - 1) {
        float uL[M], uR[M], fL[M], fR[M], vL, vR, cL, cR;
#pragma unroll
        for (int v = 0; v < M; ++v) {
          uL[v] = low(sL, v);
          uR[v] = low(sR, v);
        }
        flux_c2_f32<EQ>(uL, isx ? 0 : 1, fL, &vL, &cL, phf);
        flux_c2_f32<EQ>(uR, isx ? 0 : 1, fR, &vR, &cR, phf);
        const float lam = fmaxf(fabsf(vL) + sqrt_f32(cL), fabsf(vR) + sqrt_f32(cR));
#pragma unroll
        for (int v = 0; v < M; ++v) low(sL, v) = fL[v] + fR[v] - lam * (uR[v] - uL[v]);
      }
    }
    __syncthreads();
    // low-order residual of the interior subfaces (eq. (low.order.update)); 0
    // times alpha where the element is not blended
    if (gt0(a)) {
      double fr[M], fl[M];
#pragma unroll
      for (int v = 0; v < M; ++v) fr[v] = fl[v] = 0.0;
      if (p < N) vld_sh<M, stride>(fr, sB + tid);
      if (p > 0) vld_sh<M, stride>(fl, sB + tid - 1);
      vsub(fr, fr, fl);
      vmul(LO, fr, sWx[p]);
#pragma unroll
      for (int v = 0; v < M; ++v) fr[v] = fl[v] = 0.0;
      if (q < N) vld_sh<M, stride>(fr, sD + tid);
      if (q > 0) vld_sh<M, stride>(fl, sD + tid - n);
      vsub(fr, fr, fl);
      vfma(LO, sWy[q], fr);
    }
    // face-node data for the face kernel: evolved boundary state u* and the
    // candidate base of the flux limiter, u_b -+ c f_adj
    const double hdt = 0.5 * dt;
#pragma unroll
    for (int mm = 0; mm < SPT; ++mm) {
      const FaceSlot fs = face_slot<NSLOT, n>(tid + mm * T);
      const int eg = blk * epr + fs.el;
      if (fs.el < epr && eg < m.ne) {
        const int side = fs.side, j = fs.j, base = fs.el * NP;
        const int nb_node = base + (side == 0 ? n * j : side == 1 ? N + n * j : side == 2 ? j : j + n * N);
        const int adj_node = nb_node - (side == 1 ? 1 : side == 3 ? n : 0);
        double* ust = (side == 0 ? sA : side == 1 ? sB : side == 2 ? sC : sD) + nb_node;
        double* adj = (side < 2 ? sB : sD) + adj_node;
        const double c = hdt * ((side & 1) ? ph.cflim[side] : -ph.cflim[side]);
        double us[M], ub[M];
        if (sFull[fs.el]) {
          double fa[M];
          vld_sh<M, stride>(us, ust);
          vld_sh<M, stride>(ub, s0 + nb_node);
          vld_sh<M, stride>(fa, adj);
          vfma(ub, c, fa);
        } else {
          const float cf = trunc_f32(c);
#pragma unroll
          for (int v = 0; v < M; ++v) {
            us[v] = widen_f32(low(ust, v));
            ub[v] = widen_f32(fmaf(cf, low(adj, v), trunc_f32(s0[v * stride + nb_node])));
          }
          if (EQ::K > 0) us[0] = -us[0];  // a negative density marks FP32 face data
        }
#pragma unroll
        for (int v = 0; v < M; ++v) {
          P.b.slot[slot_index(1 + 2 * M + v, side, eg, j, 4, m.ne, n)] = us[v];
          P.b.slot[slot_index(1 + 3 * M + v, side, eg, j, 4, m.ne, n)] = ub[v];
        }
      }
    }
  }

  // ---------------- partial update --------------------------------------
  if (valid) {
    double val[M];
    vfma(val, -(dt * a), LO, HO);
#pragma unroll
    for (int v = 0; v < M; ++v) P.b.P[((size_t)v * m.ne + e) * NP + k] = val[v];
  }
}

}  // namespace crk
