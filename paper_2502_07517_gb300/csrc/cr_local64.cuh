// The FP64 element kernel (the body that k_local and the batched kernels run for
// real = double, except for scalar equations in one dimension): the same phases
// and the same outputs as local_body, arranged for the FP64 pipe.
//
// What bounds it: GB300 issues one FP64 warp instruction per SM every 16
// cycles, against two integer or FP32 ones per cycle, and the pipe was 90% busy
// at 10% of the issue slots (2D Euler N = 4, 512 x 512: 12.57 ms, 1,031 FP64
// instructions per solution point).  So every FP64 instruction that integer or
// FP32 work can replace without touching the result is worth 30 of those:
//   - the D contractions and the face traces (40% of the FP64 work) run in
//     fixed point on the integer pipe (cr_fixed.cuh); the FR volume term takes
//     each stage's fluxes with b_i in its matrices and accumulates in fixed
//     point, so the time-averaged fluxes are never formed; elements whose values
//     spread too far for a common exponent take their stages in FP64 (stages_fp64);
//   - the trace of the time-averaged solution is the average of the stage
//     traces, and the wave speed of the u^n trace shares the first stage's flux;
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
// k_local, before (the general body in FP64) and now: 2D Euler N = 4, 512 x 512, 12.57
// and 4.19 ms (58% of the FP64 pipe, 37% of the issue slots: latency bound);
// ten-moment N = 3, 256 x 256, 2.61 and 1.57 ms; 1D Euler N = 4, 4,000 elements, whole
// step, 73 and 51 us.
#pragma once
#include "cr_common.cuh"
#include "cr_fixed.cuh"
#include "cr_screen.cuh"

namespace crk {

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

// Twice the Rusanov flux (the factor 1/2 goes into the caller's constants,
// exactly).
template <class EQ>
__device__ __forceinline__ void rusanov_twice(const double* uL, const double* uR, int dir, double* out,
                                              const Phys<double>& ph) {
  double fL[EQ::M], fR[EQ::M], vL, vR, cL, cR, lam;
  flux_c2<EQ>(uL, dir, fL, &vL, &cL, ph);
  flux_c2<EQ>(uR, dir, fR, &vR, &cR, ph);
  if constexpr (EQ::K > 0) lam = wave_max(vL, cL, vR, cR);
  else lam = __longlong_as_double(max(__double_as_longlong(vL), __double_as_longlong(vR)));  // (speeds are not negative)
#pragma unroll
  for (int v = 0; v < EQ::M; ++v) out[v] = fma(-lam, uR[v] - uL[v], fL[v] + fR[v]);
}

// MUSCL-Hancock states of one node (Sec. 4.2): the evolved states at its
// subcell faces (in one dimension the y states are not formed), or the node value where one of them is not admissible.  nb(v,
// dir, up) is the neighbour node's value along the line; hx, hy = dt / (2 w h).
template <int DIM, int N, class EQ, class Nb>
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
  if (DIM == 2) slopes(sy, q, 1);
  double fxm[M], fxp[M], fym[M], fyp[M], Fm[M], Fp[M], ex[M];
  vfma(fxm, tb.dm[p], sx, un);
  vfma(fxp, tb.dp[p], sx, un);
  if (DIM == 2) {
    vfma(fym, tb.dm[q], sy, un);
    vfma(fyp, tb.dp[q], sy, un);
  }
  EQ::flux(fxm, 0, Fm, ph);
  EQ::flux(fxp, 0, Fp, ph);
  vsub(ex, Fp, Fm);
  vmul(ex, ex, hx);
  if (DIM == 2) {
    EQ::flux(fym, 1, Fm, ph);
    EQ::flux(fyp, 1, Fp, ph);
    vsub(Fp, Fp, Fm);
    vfma(ex, hy, Fp);
  }
  bool ok = true;
  if constexpr (EQ::K > 0) {
    float uf[M], xf[M], yf[M], ef[M], A[M], st[M];
    const float dmx = trunc_f32(tb.dm[p]), dpx = trunc_f32(tb.dp[p]);
    const float dmy = trunc_f32(tb.dm[q]), dpy = trunc_f32(tb.dp[q]);
#pragma unroll
    for (int v = 0; v < M; ++v) {
      uf[v] = trunc_f32(un[v]);
      xf[v] = trunc_f32(sx[v]);
      yf[v] = DIM == 2 ? trunc_f32(sy[v]) : 0.0f;
      ef[v] = trunc_f32(ex[v]);
      A[v] = fabsf(uf[v]) + fabsf(xf[v]) + fabsf(yf[v]) + fabsf(ef[v]);
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {  // the face states, then evolved
      if (DIM == 1 && (c & 2)) continue;
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
  if (DIM == 2) {
    vsub(eym, fym, ex);
    vsub(eyp, fyp, ex);
  }
  if (!ok) {
    ok = EQ::admissible_fast(fxm, ph) && EQ::admissible_fast(fxp, ph) && EQ::admissible_fast(exm, ph) &&
         EQ::admissible_fast(exp_, ph);
    if (DIM == 2)
      ok = ok && EQ::admissible_fast(fym, ph) && EQ::admissible_fast(fyp, ph) && EQ::admissible_fast(eym, ph) &&
           EQ::admissible_fast(eyp, ph);
  }
  if (ok) {
#pragma unroll
    for (int v = 0; v < M; ++v) {
      xm[v] = exm[v];
      xp[v] = exp_[v];
      if (DIM == 2) {
        ym[v] = eym[v];
        yp[v] = eyp[v];
      }
    }
  }
}

// Value of variable v at the neighbour of node k = (p, q) of a block's element
// along direction dir: from the block's nodes (u points at this node's slot),
// across a face from the neighbour element (nbr: the element's face neighbours),
// at a boundary the side's ghost node (outflow: the own node; wall: its
// reflection; Dirichlet, inflow: given).
template <int DIM, int N, class EQ, int STRIDE>
__device__ __forceinline__ double line_neighbour(const KParams<double>& P, const double* u, const int* nbr, int k, int p,
                                                 int q, int v, int dir, int up) {
  constexpr int n = N + 1, NP = DIM == 2 ? n * n : n, M = EQ::M;
  const Mesh& m = P.m;
  const int c = dir == 0 ? p : q, step = dir == 0 ? 1 : n;
  if (c != (up ? N : 0)) return u[v * STRIDE + (up ? step : -step)];
  const int side = 2 * dir + up, e2 = nbr[side];
  if (e2 >= 0) return P.b.u[((size_t)v * m.ne + e2) * NP + k + (up ? -N : N) * step];
  const int bc = m.bcs[side];
  if (bc == kBcDirichlet || bc == kBcInflow) {
    double g[M];
    ghost_at<M>(m, side, P.b.ctl->t, g);
    return g[v];
  }
  const double x = u[v * STRIDE];
  return bc == kBcWall && v == 1 + dir ? -x : x;
}

// hancock_states of a block's node into the four node arrays at st (M STRIDE
// apart).  Out of line: only blended elements, their neighbours and those beside
// a boundary come here, and the element kernel keeps its registers.
template <int DIM, int N, class EQ, int STRIDE>
__device__ __noinline__ void put_hancock_states(const KParams<double>& P, const Tab<double>& tb, const double* u,
                                                const int* nbr, int k, double alpha, double hx, double hy, double* st) {
  constexpr int M = EQ::M;
  const int p = DIM == 2 ? k % (N + 1) : k, q = DIM == 2 ? k / (N + 1) : 0;
  double un[M], xm[M], xp[M], ym[M], yp[M];
  vld_sh<M, STRIDE>(un, u);
  auto nb = [&](int v, int dir, int up) { return line_neighbour<DIM, N, EQ, STRIDE>(P, u, nbr, k, p, q, v, dir, up); };
  hancock_states<DIM, N, EQ>(P.m, P.ph, tb, un, alpha, p, q, hx, hy, nb, xm, xp, ym, yp);
  vst_sh<M, STRIDE>(st, xm);
  vst_sh<M, STRIDE>(st + M * STRIDE, xp);
  if (DIM == 2) {
    vst_sh<M, STRIDE>(st + 2 * M * STRIDE, ym);
    vst_sh<M, STRIDE>(st + 3 * M * STRIDE, yp);
  }
}

// The same in FP32, for elements whose low-order scheme only feeds the screen of
// the flux limiter (see the body).  Returns false where admissibility is not
// clear in FP32, by the margin that the limiter's bases need, or a boundary node and
// its neighbour inside the element are too unlike for those (like_neighbour); the FP64
// form then decides.
template <int DIM, int N, class EQ, class Nb>
__device__ __forceinline__ bool hancock_states_f32(const Mesh& m, const Phys<float>& ph, const Tab<double>& tb,
                                                   const float (&un)[EQ::M], float alpha, int p, int q, float hx,
                                                   float hy, Nb nb, float (&xm)[EQ::M], float (&xp)[EQ::M],
                                                   float (&ym)[EQ::M], float (&yp)[EQ::M]) {
  constexpr int M = EQ::M;
#pragma unroll
  for (int v = 0; v < M; ++v) xm[v] = xp[v] = ym[v] = yp[v] = un[v];
  bool ok = true;
  if constexpr (EQ::K > 0) {
#pragma unroll
    for (int dir = 0; dir < DIM; ++dir) {
      const int c = dir == 0 ? p : q;
#pragma unroll
      for (int v = 0; v < M; ++v)
        if (v == 0 || v == M - 1 || (M == 6 && v == 3)) {
          if (c == 0) ok = ok && like_neighbour<EQ>(v, un[v], nb(v, dir, 1));
          if (c == N) ok = ok && like_neighbour<EQ>(v, un[v], nb(v, dir, 0));
        }
    }
  }
  if (!(m.limiter & kLimMH)) {
    float A[M];
#pragma unroll
    for (int v = 0; v < M; ++v) A[v] = fabsf(un[v]);
    return ok && clearly_admissible<EQ>(un, A, kLikeF);
  }
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
  if (DIM == 2) slopes(sy, q, 1);
  float Fm[M], Fp[M], ex[M], vn, c2;
  vfma(xm, trunc_f32(tb.dm[p]), sx, un);
  vfma(xp, trunc_f32(tb.dp[p]), sx, un);
  if (DIM == 2) {
    vfma(ym, trunc_f32(tb.dm[q]), sy, un);
    vfma(yp, trunc_f32(tb.dp[q]), sy, un);
  }
  flux_c2_f32<EQ>(xm, 0, Fm, &vn, &c2, ph);
  flux_c2_f32<EQ>(xp, 0, Fp, &vn, &c2, ph);
  vsub(ex, Fp, Fm);
  vmul(ex, ex, hx);
  if (DIM == 2) {
    flux_c2_f32<EQ>(ym, 1, Fm, &vn, &c2, ph);
    flux_c2_f32<EQ>(yp, 1, Fp, &vn, &c2, ph);
    vsub(Fp, Fp, Fm);
    vfma(ex, hy, Fp);
  }
#pragma unroll
  for (int v = 0; v < M; ++v) A[v] = fabsf(un[v]) + fabsf(sx[v]) + (DIM == 2 ? fabsf(sy[v]) : 0.0f) + fabsf(ex[v]);
  auto clear = [&](const float (&s)[M]) { return clearly_admissible<EQ>(s, A, kLikeF); };
  ok = ok && clear(xm) && clear(xp);
  vsub(xm, xm, ex);
  vsub(xp, xp, ex);
  ok = ok && clear(xm) && clear(xp);
  if (DIM == 2) {
    ok = ok && clear(ym) && clear(yp);
    vsub(ym, ym, ex);
    vsub(yp, yp, ex);
    ok = ok && clear(ym) && clear(yp);
  }
  return ok;
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
template <int DIM, int N, class EQ>
__device__ __noinline__ void exact_face_data(const KParams<double>& P, const Tab<double>& tb, int e, int side, int j,
                                             double dt) {
  constexpr int n = N + 1, NP = DIM == 2 ? n * n : n, M = EQ::M;
  const Mesh& m = P.m;
#pragma unroll
  for (int f = 0; f < 2 * DIM; ++f)
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
    const double hx = dt * (0.5 * tb.invw[p] * P.ph.invdx), hy = DIM == 2 ? dt * (0.5 * tb.invw[q] * P.ph.invdy) : 0.0;
    hancock_states<DIM, N, EQ>(m, P.ph, tb, un, alpha, p, q, hx, hy, nb, xm, xp, ym, yp);
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
    P.b.slot[slot_index(1 + 2 * M + v, side, e, j, 2 * DIM, m.ne, DIM == 2 ? n : 1)] = st[0][v];
    P.b.slot[slot_index(1 + 3 * M + v, side, e, j, 2 * DIM, m.ne, DIM == 2 ? n : 1)] = fma(c, f[v], ub[v]);
  }
}

// Stage sums of the N = 4 method over residuals R_j in fixed point: sum_j a_ij R_j
// = m_i sum_j c_ij R_j with small whole c_ij.  |R| stays below 2^61.4 (the rows of D
// sum to at most 2.51 of its largest entry, Gauss-Legendre and Gauss-Lobatto), so
// the sums of stages 1 to 3 (weights up to 3) fit 63 bits as they are; those of 4
// and 5 (12 and 37) are taken 4 bits down.
struct StageSums {
  static __host__ __device__ constexpr int c(int i, int j) {
    return i == 4 ? (j == 0 ? 3 : j == 3 ? 9 : 0)
         : i == 5 ? (j == 0 ? -3 : j == 1 ? 2 : j == 2 ? 12 : j == 3 ? -12 : j == 4 ? 8 : 0) : 0;
  }
  static __host__ __device__ constexpr double m(int i) {
    return i == 1 ? 0.25 : i == 2 ? 0.125 : i == 3 ? 0.5 : i == 4 ? 0.0625 : 1.0 / 7.0;
  }
};

// Shared memory of the body beyond the five node arrays, in bytes.
template <int DIM, int N, class EQ>
__host__ __device__ constexpr size_t local64_extra(int epb) {
  constexpr int n = N + 1, S = Tableau<N>::S;
  constexpr size_t src = (EQ::M == 6 || HasGravity<EQ>::value ? EQ::M * (DIM == 2 ? n * n : n) : 0)  // the averaged source,
                         + (N == 4 ? 3 * EQ::M * (DIM == 2 ? n * n : n) : 0);                      // stage residuals
  return (size_t)epb * (1 + src) * sizeof(double) + (size_t)(2 * (1 + S) * n * n + 2 * n) * sizeof(int2) +
         (size_t)(S * S + 4 * n) * sizeof(double) + (size_t)epb * (6 + 2 * EQ::M) * sizeof(int);
}

// A sum in fixed point is as good as FP64's as long as its largest term lies within
// 2^kSpareBits (a trace: 2^kSpareTrace) of the element's largest value of that variable.
// Error against the FMA chain's, root mean square, for sums so far down, N = 1 .. 4:
// smooth lines 0.22, 0.44, 1.09, 0.30, random ones 0.47 to 0.67, lines through 0 0.55 to
// 0.85; traces 0.73 to 1.02.  An element with a node whose two lines of fluxes, which
// enter one sum, both lie below that, but not all at 0, takes its stages in FP64
// (stages_fp64), unless four units of the sum times dt are below half a unit of the
// node's value, which they are added to.  So does one with such a line of a trace, unless
// the trace's unit, as it enters the update (at most by 1 / dt), is below that of the flux
// sums.  Ten-moment data of steep cells (64 x 64, N = 3): 2 to 6% of the elements; shear
// through 0 beside gravity: none.
constexpr int kSpareBits = 2, kSpareTrace = 3;

// Whether a sum of this node's has lost bits: small has, per variable v, bit 2v where
// the node's own fluxes are below the line, 2v + 1 where its stage state is.  Out of line:
// few nodes are so small.
template <int DIM, int N, int M, int STRIDE>
__device__ __noinline__ bool sums_lose_bits(const int2* xA, int line_x, int line_y, unsigned small) {
  constexpr int n = N + 1;
  const int2* xB = xA + M * STRIDE;
  const int2* xC = xB + M * STRIDE;
  int top, any;
  auto look = [&](const int2* X, int base, int step) {
#pragma unroll 1
    for (int r = 0; r < n; ++r) {
      const int2 x = X[base + step * r];
      top = max(top, abs(x.x));
      any |= x.x | x.y;
    }
  };
  bool lost = false;
#pragma unroll 1
  for (int v = 0; v < M; ++v) {
#pragma unroll 1
    for (int c = 0; c < (DIM == 2 ? 3 : 2); ++c) {  // the fluxes' sum, the traces along x and y
      if (!((small >> (2 * v + (c > 0))) & 1u)) continue;
      top = any = 0;
      look((c == 0 ? xB : xA) + v * STRIDE, c == 2 ? line_y : line_x, c == 2 ? n : 1);
      if (DIM == 2 && c == 0) look(xC + v * STRIDE, line_y, n);
      lost = lost || (top < (1 << (28 - (c == 0 ? kSpareBits : kSpareTrace))) && any != 0);
    }
  }
  return lost;
}

// The stages, traces and the high-order part of the update in FP64 throughout, for the
// elements of the block with redo set: the same quantities as the fixed-point stages
// of local_body_f64, which they overwrite in memory (where the element is blended,
// P.b.P comes with the low-order residual).  Every thread of the block calls it; s0
// holds u^n, the three arrays behind it are free; alpha: the elements' coefficients.
template <int DIM, int N, class EQ, int T>
__device__ __noinline__ void stages_fp64(const KParams<double>& P, const Tab<double>& tb, int blk, double* s0,
                                         const double* alpha, const int* redo) {
  constexpr int n = N + 1, NP = DIM == 2 ? n * n : n, M = EQ::M, S = Tableau<N>::S;
  constexpr int NSIDE = 2 * DIM, NFN = DIM == 2 ? n : 1, NSLOT = NSIDE * NFN, SPT = (NSLOT + NP - 1) / NP;
  constexpr int epb = (T + NP - 1) / NP, epr = T / NP, stride = epb * NP, arr = M * stride;
  using TB = Tableau<N>;
  const Mesh& m = P.m;
  const int tid = threadIdx.x, el = tid / NP, k = tid - el * NP, p = DIM == 2 ? k % n : k, q = DIM == 2 ? k / n : 0;
  const int e = blk * epr + el, line_x = el * NP + n * q, line_y = el * NP + p;
  const bool on = el < epr && e < m.ne && redo[el];
  const double dt = P.b.ctl->dt_step, a = on && ((m.limiter & kLimBlend) || m.alpha_mode == 1) ? alpha[el] : 0.0;
  double* sA = s0 + arr;
  double* sB = sA + arr;
  double* sC = sB + arr;
  const bool has_src = (M == 6 && m.source == 1) || (HasGravity<EQ>::value && m.source == 2);
  double dWx = m.grav[0], dWy = m.grav[1];
  if (M == 6 && has_src) {
    const double x = m.x0 + (e % m.nx + tb.xi[p]) * m.dx, y = DIM == 2 ? m.y0 + (e / m.nx + tb.xi[q]) * m.dy : 0.0;
    source_grad<DIM, double>(m, x - m.src_cx, DIM == 2 ? y - m.src_cy : 0.0, &dWx, &dWy);
  }
  double L[S][M], Fa[M], Ga[M], Sa[M], ea[SPT][M], Ut[SPT][M];
  for (int v = 0; v < M; ++v) {
    Fa[v] = Ga[v] = Sa[v] = 0.0;
    for (int mm = 0; mm < SPT; ++mm) ea[mm][v] = Ut[mm][v] = 0.0;
  }
#pragma unroll 1
  for (int i = 0; i < S; ++i) {
    const double b = TB::b(i);
    double src[M];
    if (on) {
      double u[M], f[M], g[M];
      vld_sh<M, stride>(u, s0 + tid);
      for (int j = 0; j < i; ++j) vfma(u, -dt * TB::a(i, j), L[j]);
      if (DIM == 2) EQ::flux_xy(u, f, g, P.ph);
      else EQ::flux(u, 0, f, P.ph);
      vst_sh<M, stride>(sA + tid, u);
      vst_sh<M, stride>(sB + tid, f);
      vfma(Fa, b, f);
      if (DIM == 2) {
        vst_sh<M, stride>(sC + tid, g);
        vfma(Ga, b, g);
      }
      if (has_src) {
        source_eval<EQ>(u, dWx, dWy, src);
        vfma(Sa, b, src);
      }
    }
    __syncthreads();
    if (on && i < S - 1) {
#pragma unroll
      for (int v = 0; v < M; ++v) {
        double h = 0.0;
#pragma unroll
        for (int r = 0; r < n; ++r) h = fma(P.ds.Dx[p * n + r], sB[v * stride + line_x + r], h);
        if (DIM == 2)
#pragma unroll
          for (int r = 0; r < n; ++r) h = fma(P.ds.Dy[q * n + r], sC[v * stride + line_y + n * r], h);
        L[i][v] = has_src ? h - src[v] : h;
      }
    }
    if (i == 0 || b != 0.0) {
#pragma unroll
      for (int mm = 0; mm < SPT; ++mm) {
        const FaceSlot fs = face_slot<NSLOT, NFN>(tid + mm * T);
        const int eg = blk * epr + fs.el;
        if (fs.el >= epr || eg >= m.ne || !redo[fs.el]) continue;
        const int side = fs.side, j = fs.j, base = fs.el * NP + (side < 2 ? n * j : j), step = side < 2 ? 1 : n;
        auto trace = [&](const double* X, double (&t)[M]) {
#pragma unroll
          for (int v = 0; v < M; ++v) {
            t[v] = 0.0;
#pragma unroll
            for (int r = 0; r < n; ++r) t[v] = fma((side & 1) ? tb.l1[r] : tb.l0[r], X[v * stride + base + step * r], t[v]);
          }
        };
        double ut[M], fn[M];
        trace(sA, ut);
        if (i == 0) {
          P.b.slot[slot_index(0, side, eg, j, NSIDE, m.ne, NFN)] = EQ::speed(ut, side >> 1, P.ph);
          if (m.dissipation == 1)
            for (int v = 0; v < M; ++v) P.b.slot[slot_index(1 + v, side, eg, j, NSIDE, m.ne, NFN)] = ut[v];
        }
        if (b == 0.0) continue;
        vfma(Ut[mm], b, ut);
        if (m.dissipation == 2)
          for (int v = 0; v < M; ++v) P.b.slot[slot_index(1 + 4 * M + i * M + v, side, eg, j, NSIDE, m.ne, NFN)] = ut[v];
        if (m.central == 0) EQ::flux(ut, side >> 1, fn, P.ph);
        else trace(side < 2 ? sB : sC, fn);
        vfma(ea[mm], b, fn);
      }
    }
    __syncthreads();
  }
  vst_sh<M, stride>(sB + tid, Fa);
  if (DIM == 2) vst_sh<M, stride>(sC + tid, Ga);
  __syncthreads();
  if (on) {
#pragma unroll
    for (int v = 0; v < M; ++v) {
      double h = 0.0;
#pragma unroll
      for (int r = 0; r < n; ++r) h = fma(P.ds.Dtx[p * n + r], sB[v * stride + line_x + r], h);
      if (DIM == 2)
#pragma unroll
        for (int r = 0; r < n; ++r) h = fma(P.ds.Dty[q * n + r], sC[v * stride + line_y + n * r], h);
      h = fma(-(dt * (1.0 - a)), h, s0[v * stride + tid]);
      if (has_src) h = fma(dt, Sa[v], h);
      double* val = P.b.P + ((size_t)v * m.ne + e) * NP + k;
      *val = gt0(a) ? fma(-(dt * a), *val, h) : h;
    }
  }
#pragma unroll
  for (int mm = 0; mm < SPT; ++mm) {
    const FaceSlot fs = face_slot<NSLOT, NFN>(tid + mm * T);
    const int eg = blk * epr + fs.el;
    if (fs.el >= epr || eg >= m.ne || !redo[fs.el]) continue;
    for (int v = 0; v < M; ++v) {
      if (m.dissipation != 1) P.b.slot[slot_index(1 + v, fs.side, eg, fs.j, NSIDE, m.ne, NFN)] = Ut[mm][v];
      P.b.slot[slot_index(1 + M + v, fs.side, eg, fs.j, NSIDE, m.ne, NFN)] = ea[mm][v];
    }
  }
}

template <int DIM, int N, class EQ, int T>
__device__ __forceinline__ void local_body_f64(const KParams<double>& P, const Tab<double>& tb, const int blk) {
  constexpr int n = N + 1, NP = DIM == 2 ? n * n : n, M = EQ::M, S = Tableau<N>::S;
  constexpr int NSIDE = 2 * DIM, NFN = DIM == 2 ? n : 1, NSLOT = NSIDE * NFN;
  constexpr int SPT = (NSLOT + NP - 1) / NP;
  using TB = Tableau<N>;
  const Mesh& m = P.m;
  const Phys<double>& ph = P.ph;
  constexpr int epb = (T + NP - 1) / NP, epr = T / NP;
  const int tid = threadIdx.x;
  const int el = tid / NP, k = tid - el * NP, p = DIM == 2 ? k % n : k, q = DIM == 2 ? k / n : 0;
  const int e = blk * epr + el;
  const bool valid = el < epr && e < m.ne;
  const int ee = valid ? e : m.ne - 1;
  const int ix = ee % m.nx, iy = ee / m.nx;

  const double dt = P.b.ctl->dt_step;
  if (!gt0(dt)) return;

  // node arrays [M][epb][NP]: u^n; in fixed point the stage state and fluxes,
  // then the MUSCL-Hancock states; for a source its time average
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int stride = epb * NP, arr = M * stride;
  double* s0 = reinterpret_cast<double*>(smem_raw);
  double* sA = s0 + arr;
  double* sB = sA + arr;
  double* sC = sB + arr;
  double* sD = sC + arr;
  constexpr bool SRC = EQ::M == 6 || HasGravity<EQ>::value;
  constexpr bool kShL = N == 4;  // four residuals are live at a time
  double* sS = sD + arr;
  double* sL = sS + (SRC ? arr : 0);  // stage residuals 0..2 (kept in shared memory at N = 4; 3: sD)
  int2* xA = reinterpret_cast<int2*>(sA);
  int2* xB = reinterpret_cast<int2*>(sB);
  int2* xC = reinterpret_cast<int2*>(sC);
  double* sAlpha = sL + (kShL ? 3 * arr : 0);                 // [epb]
  int2* tDx = reinterpret_cast<int2*>(sAlpha + epb);          // [n][n] each
  int2* tDy = tDx + n * n;
  int2* tB = tDy + n * n;                                     // b_i times the FR matrices [S][2][n][n]
  int2* tL = tB + 2 * S * n * n;                              // l(0), l(1) [2][n]
  double* sAdt = reinterpret_cast<double*>(tL + 2 * n);       // dt a_ij
  double* sHx = sAdt + S * S;                                 // dt / (2 w_p dx), dt / (2 w_q dy)
  double* sHy = sHx + n;
  double* sWx = sHy + n;                                      // 1 / (2 w_p dx), 1 / (2 w_q dy)
  double* sWy = sWx + n;
  int* sNbr = reinterpret_cast<int*>(sWy + n);                // [epb][4]
  int* sKey = sNbr + epb * 4;                                 // exponents [fluxes, state][epb][M]
  int* sFull = sKey + 2 * epb * M;                            // [epb] low-order scheme in FP64
  int* sRedo = sFull + epb;                                   // [epb] stages to be done in FP64

  double un[M];
#pragma unroll
  for (int v = 0; v < M; ++v) un[v] = P.b.u[((size_t)v * m.ne + ee) * NP + k];
  for (int t = tid; t < 2 * epb * M; t += T) sKey[t] = 0;
  for (int t = tid; t < epb; t += T) {
    sFull[t] = sRedo[t] = 0;
    sAlpha[t] = m.alpha_mode == 1 ? m.alpha_fixed : 0.0;
  }
  __syncthreads();
  // alpha_e, smoothed with the face neighbours, and which elements need their
  // low-order scheme in FP64: the blended ones, those with a blended face (a face
  // neighbour is blended: alpha_raw > 0 in it or in a neighbour of it) and those
  // beside a boundary (those faces take the FP64 limiter as it stands).
  // Everywhere else that scheme feeds only the flux limiter's test, which FP32
  // answers (cr_screen.cuh; the face kernel forms the FP64 data itself where it
  // does not).  One thread per element and cell of the 13 within two steps, so
  // that their loads go out together.
  constexpr int NC = DIM == 2 ? 13 : 5;
  for (int t = T - 1 - tid; t < epb * NC; t += T) {
    const int e2 = t / NC, c = DIM == 2 ? t - e2 * NC : (0x65410 >> (4 * (t - e2 * NC))) & 15;
    const int eg0 = blk * epr + e2, eg = e2 < epr && eg0 < m.ne ? eg0 : m.ne - 1;
    // cell offsets: the face neighbours (x-, x+, y-, y+), the element, the second ring
    // plus 2, three bits each
    const int iy = eg / m.nx;
    int cx = eg - iy * m.nx + int(0x32ca502499ull >> (3 * c) & 7) - 2, cy = iy + int(0x364c092652ull >> (3 * c) & 7) - 2;
    bool in = true;
    if (m.bcx == 0) cx = (cx % m.nx + m.nx) % m.nx;
    else in = cx >= 0 && cx < m.nx;
    if (DIM == 1) cy = 0;
    else if (m.bcy == 0) cy = (cy % m.ny + m.ny) % m.ny;
    else in = in && cy >= 0 && cy < m.ny;
    const int ec = in ? cx + m.nx * cy : -1;
    if (c < 4) {
      sNbr[e2 * 4 + c] = ec;
      if (ec < 0) sFull[e2] = 1;
    }
    if (m.alpha_mode != 1 && (m.limiter & kLimBlend) && ec >= 0) {
      const double raw = P.b.alpha_raw[ec];
      if (gt0(raw)) {
        sFull[e2] = 1;
        if (c <= 4)  // bit patterns of positive numbers order as the values
          atomicMax(reinterpret_cast<unsigned long long*>(sAlpha + e2),
                    (unsigned long long)__double_as_longlong(c == 4 ? raw : 0.5 * raw));
      }
    }
  }
  // tables: D / dx, D / dy, b_i times the FR matrices, the trace coefficients
  for (int t = tid; t < 2 * (1 + S) * n * n; t += T) {
    const int i = t / (n * n), r = t - i * (n * n), st = i / 2 - 1;
    if (i < 2) tDx[t] = (i == 0 ? P.ds.fDx : P.ds.fDy)[r];
    else tDx[t] = fix_scaled((i & 1 ? P.ds.fDty : P.ds.fDtx)[r], TB::b(st));
  }
  for (int t = tid; t < 2 * n; t += T) tL[t] = P.ds.fL[t];
  // factors of the step and the node row
  for (int t = tid; t < S * S + 2 * n; t += T) {
    if (t < S) {  // (row 0 of the tableau is empty: the factors of the integer sums)
      sAdt[t] = N == 4 && t > 0 ? dt * StageSums::m(t) : 0.0;
    } else if (t < S * S) {
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
  if (m.alpha_mode == 1 && gt0(m.alpha_fixed)) {
    for (int t = tid; t < epb; t += T) sFull[t] = 1;  // (read after the stages' barriers)
  }
  for (int t = tid; t < epr; t += T)
    if (blk * epr + t < m.ne) P.b.alpha[blk * epr + t] = sAlpha[t];
  const double alpha = sAlpha[el];
  const bool blend = (m.limiter & kLimBlend) || m.alpha_mode == 1;
  const bool need_lo = blend || (m.limiter & kLimFlux);
  const double a = blend ? alpha : 0.0;

  const bool has_src = (EQ::M == 6 && m.source == 1) || (HasGravity<EQ>::value && m.source == 2);
  double dWx = 0.0, dWy = 0.0;
  if (HasGravity<EQ>::value && has_src) {
    dWx = m.grav[0];
    dWy = DIM == 2 ? m.grav[1] : 0.0;
  } else if (SRC && has_src) {
    const double x = m.x0 + (ix + tb.xi[p]) * m.dx, y = DIM == 2 ? m.y0 + (iy + tb.xi[q]) * m.dy : 0.0;
    source_grad<DIM, double>(m, x - m.src_cx, DIM == 2 ? y - m.src_cy : 0.0, &dWx, &dWy);
  }

  // ---------------- local cRK stages -----------------------------------
  double Lst[S > 1 ? S - 1 : 1][M];
  constexpr bool kIntSums = N == 4 && !SRC;  // the residuals stay in fixed point
  long long Rlast[M];                        // (the last one, in registers)
  double ea[SPT][M], Ut[SPT][M];
  long long ho[M];  // sum_i b_i (FR volume part of the stage fluxes), fixed point
#pragma unroll
  for (int v = 0; v < M; ++v) {
    ho[v] = 0;
#pragma unroll
    for (int mm = 0; mm < SPT; ++mm) ea[mm][v] = Ut[mm][v] = 0.0;
  }
  const int line_x = el * NP + n * q, line_y = el * NP + p;
  // Exponents of the element's values in fixed point, per variable: kf is the
  // exponent of the products |D/dx| |f|, |D/dy| |g| (the x and y fluxes so carry
  // exponents kf - oD[0], kf - oD[1], and their sums need no alignment), ku the
  // exponent of the stage state.
  int* const kf = sKey + el * M;
  int* const ku = kf + epb * M;
  const int o0 = P.ds.oD[0], o1 = DIM == 2 ? P.ds.oD[1] : o0;
  const int kmin = kMinLineExp + max(o0, o1), kmax = kMaxLineExp + min(o0, o1), exp_dt = exp_of(dt) - 1023;

  // The fluxes of this node, and where its traces are wanted the stage state,
  // into the node arrays in fixed point, and a barrier.  An element keeps its
  // exponents from the first stage until a value needs two more bits; then
  // (rarely: the vote) it takes the larger ones.  An element in which a sum of this
  // stage loses bits, or whose exponents are out of range, is marked for stages_fp64.
  auto put_nodes = [&](const double (&f)[M], const double (&g)[M], const double (&u)[M], int i, bool traces) {
    const bool first = i == 0;
    auto check_range = [&]() {
#pragma unroll
      for (int v = 0; v < M; ++v)
        if (kf[v] > kmax || ku[v] > kMaxLineExp) sRedo[el] = 1;
    };
    if (first) {
#pragma unroll
      for (int v = 0; v < M; ++v) {
        atomicMax(kf + v, max((DIM == 2 ? max(exp_of(f[v]) + o0, exp_of(g[v]) + o1) : exp_of(f[v]) + o0), kmin));
        atomicMax(ku + v, max(exp_of(u[v]), kMinLineExp));
      }
      __syncthreads();
      check_range();
    }
    // bits 2v: f[v] and g[v] (the larger one), 2v + 1: u[v]: outside the spare bits below
    // the exponent and the one above; over: above; small: below (sums_lose_bits)
    unsigned odd = 0u, over = 0u, small = 0u;
    auto put_all = [&]() {
#pragma unroll
      for (int v = 0; v < M; ++v) {
        const int E = kf[v], own = DIM == 2 ? max(exp_of(f[v]) + o0, exp_of(g[v]) + o1) : exp_of(f[v]) + o0;
        odd |= unsigned(unsigned(own - (E - kSpareBits)) > unsigned(kSpareBits + 1)) << (2 * v);
        xB[v * stride + tid] = to_fixed(f[v], E - o0);
        if (DIM == 2) xC[v * stride + tid] = to_fixed(g[v], E - o1);
        if (traces) {
          const int Eu = ku[v];
          odd |= unsigned(unsigned(exp_of(u[v]) - (Eu - kSpareTrace)) > unsigned(kSpareTrace + 1)) << (2 * v + 1);
          xA[v * stride + tid] = to_fixed(u[v], Eu);
        }
      }
    };
    auto sort_out = [&]() {  // (and a number below the unit becomes one unit: it is not 0)
      over = small = 0u;
      auto unit = [](double x) { return make_int2(0, (__double_as_longlong(x) << 1) == 0 ? 0 : (__double2hiint(x) >> 31) | 1); };
#pragma unroll
      for (int v = 0; v < M; ++v) {
        const int E = kf[v], xf = exp_of(f[v]) + o0, xg = DIM == 2 ? exp_of(g[v]) + o1 : xf, own = max(xf, xg);
        over |= unsigned(own > E + 1) << (2 * v);
        // (the unit of a sum is 2^E, that of a product in it 2^(E + 57))
        small |= unsigned(own < E - kSpareBits && E + exp_dt + 56 > exp_of(u[v])) << (2 * v);
        if (xf < E - 57) xB[v * stride + tid] = unit(f[v]);
        if (DIM == 2 && xg < E - 57) xC[v * stride + tid] = unit(g[v]);
        if (traces) {
          const int Eu = ku[v], xu = exp_of(u[v]);
          over |= unsigned(xu > Eu + 1) << (2 * v + 1);
          small |= unsigned(xu < Eu - kSpareTrace && Eu - exp_dt > E + 57) << (2 * v + 1);
          if (xu < Eu - 57) xA[v * stride + tid] = unit(u[v]);
        }
      }
    };
    put_all();
    if (odd) sort_out();
    if (first) {
      __syncthreads();
    } else if (__syncthreads_or(valid && over)) {
      int before[M];
#pragma unroll
      for (int v = 0; v < M; ++v) before[v] = kf[v];
      __syncthreads();
#pragma unroll
      for (int v = 0; v < M; ++v) {
        if ((over >> (2 * v)) & 1u) atomicMax(kf + v, (DIM == 2 ? max(exp_of(f[v]) + o0, exp_of(g[v]) + o1) : exp_of(f[v]) + o0));
        if ((over >> (2 * v + 1)) & 1u) atomicMax(ku + v, exp_of(u[v]));
      }
      __syncthreads();
      put_all();
      sort_out();
      check_range();
#pragma unroll
      for (int v = 0; v < M; ++v) {
        const int d = min(63, kf[v] - before[v]);
        ho[v] >>= d;
        if (kIntSums) {
          for (int j = 0; j < i && j < 4; ++j)
            reinterpret_cast<long long*>(j == 3 ? sD : sL + j * arr)[v * stride + tid] >>= d;
        }
      }
      __syncthreads();
    }
    if (small && valid && sums_lose_bits<DIM, N, M, stride>(xA, line_x, line_y, small)) sRedo[el] = 1;
  };
  // Trace along the line (base, step) of node values X with exponent E.
  auto trace_dot = [&](const int2* X, int E, int base, int step, const int2* l) -> double {
    FixAcc acc = fix_zero();
#pragma unroll
    for (int r = 0; r < n; ++r) fix_mad(acc, X[base + step * r], l[r]);
    return from_fixed(fix_sum(acc), E + P.ds.oL);
  };

#pragma unroll
  for (int i = 0; i < S; ++i) {
    constexpr bool kSrcEq = SRC;
    const bool avg = TB::b(i) != 0.0;           // the stage enters the time averages
    const bool traces = i == 0 || avg;
    double ui[M], f[M], g[M];
    vld_sh<M, stride>(ui, s0 + tid);
    if (kIntSums && i > 0) {
      // u^n - dt m_i sum_j c_ij R_j (StageSums): the sum is exact in integers, one
      // FP64 instruction per variable
#pragma unroll
      for (int v = 0; v < M; ++v) {
        auto R = [&](int j) {
          return j == 4 ? Rlast[v] : reinterpret_cast<long long*>(j == 3 ? sD : sL + j * arr)[v * stride + tid];
        };
        constexpr int low = 4;  // of the sums that need headroom, the low bits are summed apart
        long long sum = 0, rest = 0;
        if (i == 1) sum = R(0);
        if (i == 2) sum = R(0) + R(1);
        if (i == 3) sum = 2 * R(2) - R(1);
        if (i >= 4) {
#pragma unroll
          for (int j = 0; j < i; ++j) {
            const int c = StageSums::c(i, j);
            if (c == 0) continue;
            const long long r = R(j);
            sum += c * (r >> low);
            rest += c * (r & ((1 << low) - 1));
          }
          sum += rest >> low;
        }
        ui[v] = fma(-sAdt[i], from_fixed(sum, kf[v] + (i >= 4 ? low : 0)), ui[v]);
      }
    } else {
#pragma unroll
      for (int j = 0; j < i; ++j) {
        if (TB::a(i, j) == 0.0) continue;
        if (kShL && j < 4) vfma_sh<M, stride>(ui, -sAdt[i * S + j], (j == 3 ? sD : sL + j * arr) + tid);
        else vfma(ui, -sAdt[i * S + j], Lst[j]);
      }
    }
    if (DIM == 2) EQ::flux_xy(ui, f, g, ph);
    else EQ::flux(ui, 0, f, ph);
    double src[M];
    if (kSrcEq && has_src) {
      source_eval<EQ>(ui, dWx, dWy, src);
#pragma unroll
      for (int v = 0; v < M; ++v) {  // the time-averaged source, sum_i b_i s(u^(i))
        double* sa = sS + v * stride + tid;
        if (i == 0) *sa = TB::b(0) * src[v];
        else if (avg) *sa = fma(TB::b(i), src[v], *sa);
      }
    }
    if (i < S - 1 || avg) put_nodes(f, g, ui, i, traces);
    // one pass over the two lines for the stage residual D f / dx + D g / dy and
    // the stage's part of the FR volume term (its matrices hold the factor b_i),
    // two variables at a time (one load of a coefficient for both)
    const int2* const bx = tB + 2 * i * n * n;
    const int2* const by = bx + n * n;
#pragma unroll
    for (int v0 = 0; v0 < M; v0 += 2) {
      const int W = M - v0 < 2 ? M - v0 : 2;
      FixAcc lo[2], hi[2];
#pragma unroll
      for (int w = 0; w < 2; ++w) lo[w] = hi[w] = fix_zero();
#pragma unroll
      for (int d = 0; d < DIM; ++d) {
#pragma unroll
        for (int r = 0; r < n; ++r) {
          const int c = (d == 0 ? p : q) * n + r;
          int2 cl, ch;
          if (i < S - 1) cl = (d == 0 ? tDx : tDy)[c];
          if (avg) ch = (d == 0 ? bx : by)[c];
#pragma unroll
          for (int w = 0; w < 2; ++w) {
            if (w >= W) break;
            const int2 x = d == 0 ? xB[(v0 + w) * stride + line_x + r] : xC[(v0 + w) * stride + line_y + n * r];
            if (i < S - 1) fix_mad(lo[w], x, cl);
            if (avg) fix_mad(hi[w], x, ch);
          }
        }
      }
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        if (w >= W) break;
        const int v = v0 + w;
        if (avg) ho[v] += fix_sum(hi[w]);
        if (i < S - 1) {
          if (kIntSums) {
            const long long r = fix_sum(lo[w]);
            if (i == 4) Rlast[v] = r;
            else reinterpret_cast<long long*>(i == 3 ? sD : sL + i * arr)[v * stride + tid] = r;
            continue;
          }
          double L = from_fixed(fix_sum(lo[w]), kf[v]);
          if (kSrcEq && has_src) L -= src[v];
          if (kShL && i < 4) (i == 3 ? sD : sL + i * arr)[v * stride + tid] = L;
          else Lst[i < S - 1 ? i : 0][v] = L;
        }
      }
    }
    if (traces) {
#pragma unroll
      for (int mm = 0; mm < SPT; ++mm) {
        const FaceSlot fs = face_slot<NSLOT, NFN>(tid + mm * T);
        const int eg = blk * epr + fs.el;
        if (fs.el < epr && eg < m.ne) {
          const int side = fs.side, j = fs.j;
          const bool isx = side < 2;
          const int base = fs.el * NP + (isx ? n * j : j), step = isx ? 1 : n;
          const int* key = sKey + fs.el * M;
          const int2* l = tL + (side & 1) * n;
          double ut[M];
#pragma unroll
          for (int v = 0; v < M; ++v) ut[v] = trace_dot(xA + v * stride, key[epb * M + v], base, step, l);
          if (avg) {
            vfma(Ut[mm], TB::b(i), ut);
            if (m.dissipation == 2) {  // D-CSX: the stage trace, for the face kernel
#pragma unroll
              for (int v = 0; v < M; ++v)
                P.b.slot[slot_index(1 + 4 * M + i * M + v, side, eg, j, NSIDE, m.ne, NFN)] = ut[v];
            }
          }
          if (i == 0 || m.central == 0) {
            double fn[M], vn, c2;
            flux_c2<EQ>(ut, side >> 1, fn, &vn, &c2, ph);
            if (avg && m.central == 0) vfma(ea[mm], TB::b(i), fn);  // EA, eq. (evaluate)
            if (i == 0) {  // u^n trace: its wave speed, and the trace itself for D1
              P.b.slot[slot_index(0, side, eg, j, NSIDE, m.ne, NFN)] = EQ::K > 0 ? fabs(vn) + sqrt_pos(c2) : vn;
              if (m.dissipation == 1) {
#pragma unroll
                for (int v = 0; v < M; ++v) P.b.slot[slot_index(1 + v, side, eg, j, NSIDE, m.ne, NFN)] = ut[v];
              }
            }
          }
          if (avg && m.central == 1) {  // AE, eq. (extrapolate): the trace of the flux itself
#pragma unroll
            for (int v = 0; v < M; ++v)
              ea[mm][v] = fma(TB::b(i), trace_dot((isx ? xB : xC) + v * stride, key[v] - (isx ? o0 : o1), base, step, l), ea[mm][v]);
          }
        }
      }
    }
    if (i < S - 1) __syncthreads();
  }

  // ---------------- high-order part of the update, face data -------------
  // HO = u^n - dt (1 - a) sum_i b_i (FR volume part) + dt (time-averaged source)
  // (into memory at once: the low-order part is added where alpha > 0)
  {
    const double dho = dt * (1.0 - a);
#pragma unroll
    for (int v = 0; v < M; ++v) {
      double h = fma(-dho, from_fixed(ho[v], kf[v] + P.ds.oDt), s0[v * stride + tid]);
      if (SRC && has_src) h = fma(dt, sS[v * stride + tid], h);
      if (valid) P.b.P[((size_t)v * m.ne + e) * NP + k] = h;
    }
  }
#pragma unroll
  for (int mm = 0; mm < SPT; ++mm) {
    const FaceSlot fs = face_slot<NSLOT, NFN>(tid + mm * T);
    const int eg = blk * epr + fs.el;
    if (fs.el < epr && eg < m.ne) {
      // slots 1..M: the trace the dissipation jumps over (U; D1 stored u^n's);
      // slots 1+M..: the central part (EA or AE average)
#pragma unroll
      for (int v = 0; v < M; ++v) {
        if (m.dissipation != 1) P.b.slot[slot_index(1 + v, fs.side, eg, fs.j, NSIDE, m.ne, NFN)] = Ut[mm][v];
        P.b.slot[slot_index(1 + M + v, fs.side, eg, fs.j, NSIDE, m.ne, NFN)] = ea[mm][v];
      }
    }
  }
  __syncthreads();

  // ---------------- MUSCL-Hancock / first-order subcells -----------------
  if (need_lo) {
    auto nb = [&](int v, int dir, int up) { return line_neighbour<DIM, N, EQ, stride>(P, s0 + tid, sNbr + el * 4, k, p, q, v, dir, up); };
    auto put_exact = [&]() {
      put_hancock_states<DIM, N, EQ, stride>(P, tb, s0 + tid, sNbr + el * 4, k, alpha, sHx[p], sHy[q], sA + tid);
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
      for (int v = 0; v < M; ++v) uf[v] = trunc_f32(s0[v * stride + tid]);
      auto nbf = [&](int v, int dir, int up) { return trunc_f32(nb(v, dir, up)); };
      unclear = !hancock_states_f32<DIM, N, EQ>(m, phf, tb, uf, trunc_f32(alpha), p, q, trunc_f32(sHx[p]), trunc_f32(sHy[q]),
                                           nbf, xm, xp, ym, yp);
#pragma unroll
      for (int v = 0; v < M; ++v) {
        low(sA + tid, v) = xm[v];
        low(sB + tid, v) = xp[v];
        if (DIM == 2) {
          low(sC + tid, v) = ym[v];
          low(sD + tid, v) = yp[v];
        }
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
    constexpr int NSX = N * NFN, NSF = DIM * NSX;
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
    // low-order residual of the interior subfaces (eq. (low.order.update))
    if (valid && gt0(a)) {
      double LO[M], fr[M], fl[M];
#pragma unroll
      for (int v = 0; v < M; ++v) fr[v] = fl[v] = 0.0;
      if (p < N) vld_sh<M, stride>(fr, sB + tid);
      if (p > 0) vld_sh<M, stride>(fl, sB + tid - 1);
      vsub(fr, fr, fl);
      vmul(LO, fr, sWx[p]);
      if (DIM == 2) {
#pragma unroll
        for (int v = 0; v < M; ++v) fr[v] = fl[v] = 0.0;
        if (q < N) vld_sh<M, stride>(fr, sD + tid);
        if (q > 0) vld_sh<M, stride>(fl, sD + tid - n);
        vsub(fr, fr, fl);
        vfma(LO, sWy[q], fr);
      }
#pragma unroll
      for (int v = 0; v < M; ++v) {
        double* val = P.b.P + ((size_t)v * m.ne + e) * NP + k;
        *val = sRedo[el] ? LO[v] : fma(-(dt * a), LO[v], *val);  // (stages_fp64 adds it to its high-order part)
      }
    }
    // face-node data for the face kernel: evolved boundary state u* and the
    // candidate base of the flux limiter, u_b -+ c f_adj
    const double hdt = 0.5 * dt;
#pragma unroll
    for (int mm = 0; mm < SPT; ++mm) {
      const FaceSlot fs = face_slot<NSLOT, NFN>(tid + mm * T);
      const int eg = blk * epr + fs.el;
      if (fs.el < epr && eg < m.ne) {
        const int side = fs.side, j = fs.j, base = fs.el * NP;
        const int nb_node = base + (DIM == 1 ? side * N : side == 0 ? n * j : side == 1 ? N + n * j : side == 2 ? j : j + n * N);
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
          P.b.slot[slot_index(1 + 2 * M + v, side, eg, j, NSIDE, m.ne, NFN)] = us[v];
          P.b.slot[slot_index(1 + 3 * M + v, side, eg, j, NSIDE, m.ne, NFN)] = ub[v];
        }
      }
    }
  }
  // (at the end, where least is alive: called behind the stages it cost 5% of the
  // kernel where no element needs it)
  if (__syncthreads_or(valid && sRedo[el])) stages_fp64<DIM, N, EQ, T>(P, tb, blk, s0, sAlpha, sRedo);
}

}  // namespace crk
