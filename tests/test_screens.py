"""The FP32 screens in front of FP64 decisions (csrc/cr_screen.cuh), compiled for
the host: over all magnitudes of the data, also those outside FP32's range, a
screen that answers must answer as FP64 does.  And the FP64 constraints that decide
where a screen does not.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <cuda_runtime.h>
template <class A, class B> static A bits(B b) { A a; static_assert(sizeof a == sizeof b, ""); memcpy(&a, &b, sizeof a); return a; }
static inline int __double2hiint(double x) { return int(bits<uint64_t>(x) >> 32); }
static inline int __double2loint(double x) { return int(uint32_t(bits<uint64_t>(x))); }
static inline double __hiloint2double(int h, int l) { return bits<double>((uint64_t(uint32_t(h)) << 32) | uint32_t(l)); }
static inline long long __double_as_longlong(double x) { return bits<long long>(x); }
static inline double __longlong_as_double(long long b) { return bits<double>(b); }
static inline unsigned __float_as_uint(float x) { return bits<unsigned>(x); }
static inline float __uint_as_float(unsigned b) { return bits<float>(b); }
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
  return unsigned((((uint64_t(hi) << 32) | lo) << (s & 31)) >> 32);
}
static inline float __frcp_rn(float x) { return 1.0f / x; }
using std::isfinite; using std::max; using std::min;
#include "cr_screen.cuh"
using namespace crk;
using Euler = EqEuler<2>;
extern "C" {
float truncated(double x) { return trunc_f32(x); }
int above_eps(const double* u) {
  float s[4], A[4];
  for (int v = 0; v < 4; ++v) {
    s[v] = trunc_f32(u[v]);
    A[v] = fabsf(s[v]);
  }
  return clearly_above_eps<Euler>(s, A, 0.4f);
}
int admissible(const double* u, int m) {
  float s[6], A[6];
  for (int v = 0; v < m; ++v) {
    s[v] = trunc_f32(u[v]);
    A[v] = fabsf(s[v]);
  }
  return m == 4 ? clearly_admissible<Euler>(s, A) : clearly_admissible<EqTenMoment>(s, A);
}
int idle(const double* d, int m, double cL, double cR) {  // uL, uR, bL, bR, F
  float x[5][6];
  for (int i = 0; i < 5; ++i)
    for (int v = 0; v < m; ++v) x[i][v] = trunc_f32(d[i * m + v]);
  Phys<double> ph{};
  ph.gamma = 1.4;
  ph.gm1 = 0.4;
  const float l = trunc_f32(cL), r = trunc_f32(cR);
  return m == 4 ? flux_limiter_idle<Euler>(x[0], x[1], x[2], x[3], x[4], l, r, 0, ph)
                : flux_limiter_idle<EqTenMoment>(x[0], x[1], x[2], x[3], x[4], l, r, 0, ph);
}
double constraint(const double* u, int m) {
  Phys<double> ph{};
  ph.gm1 = 0.4;
  return m == 4 ? Euler::constraint(u, 1, ph) : EqTenMoment::constraint(u, 1, ph);
}
void low_flux(const double* d, int m, float* lo, float* a) {  // uL, uR
  float x[2][6];
  for (int i = 0; i < 2; ++i)
    for (int v = 0; v < m; ++v) x[i][v] = trunc_f32(d[i * m + v]);
  Phys<float> ph{};
  ph.gamma = 1.4f;
  ph.gm1 = 0.4f;
  if (m == 4) rusanov_f32<Euler>(x[0], x[1], 0, ph, lo, a);
  else rusanov_f32<EqTenMoment>(x[0], x[1], 0, ph, lo, a);
}
int like(const double* d, int m) {  // u, its neighbour: alike, and both admissible by kLikeF
  float x[2][6], A[2][6];
  bool ok = true;
  for (int i = 0; i < 2; ++i)
    for (int v = 0; v < m; ++v) {
      x[i][v] = trunc_f32(d[i * m + v]);
      A[i][v] = fabsf(x[i][v]);
    }
  for (int v = 0; v < m; ++v) ok = ok && (m == 4 ? like_neighbour<Euler>(v, x[0][v], x[1][v]) : like_neighbour<EqTenMoment>(v, x[0][v], x[1][v]));
  for (int i = 0; i < 2; ++i) ok = ok && (m == 4 ? clearly_admissible<Euler>(x[i], A[i], kLikeF) : clearly_admissible<EqTenMoment>(x[i], A[i], kLikeF));
  return ok;
}
double speed(const double* s) { return wave_max(s[0], s[1], s[2], s[3]); }
double minmod(const double* d, const double* b) {
  return minmod_scaled(d[0], d[1], d[2], b[0], b[1], b[2], trunc_f32(b[0]), trunc_f32(b[1]), trunc_f32(b[2]));
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("screens")
    src, out = d / "screens.cpp", d / "libscreens.so"
    src.write_text(SRC)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"),
                    "-I", os.path.join(ROOT, "paper_2502_07517_gb300", "csrc"), str(src), "-o", str(out)], check=True)
    lib = ctypes.CDLL(str(out))
    lib.minmod.restype = lib.speed.restype = lib.constraint.restype = ctypes.c_double
    lib.truncated.restype, lib.truncated.argtypes = ctypes.c_float, [ctypes.c_double]
    return lib


def _p(*values):
    return np.array(values, dtype=np.float64).ctypes.data_as(ctypes.POINTER(ctypes.c_double))


SIZES = [5e-324, 1e-310, 1e-300, 1e-60, 1e-45, 1e-42, 1e-38, 1e-30, 1e-20, 1.0, 1e20, 1e30, 1e38, 1e39, 1e60, 1e290]


@pytest.mark.parametrize("size", SIZES)
@pytest.mark.parametrize("other", [1.0, 1e-12, 1e12])
def test_minmod_takes_the_smallest_slope(lib, size, other):
    rng = np.random.default_rng(3)
    for it in range(400):
        d = size * rng.uniform(0.5, 2.0, 3)
        d[it % 3] *= other
        d = d * rng.choice([-1.0, 1.0]) if it % 8 else d * rng.choice([-1.0, 0.0, 1.0], 3)
        b = rng.uniform(0.5, 8.0, 3)
        s = d * b
        want = 0.0 if not ((s > 0).all() or (s < 0).all()) else s[np.argmin(np.abs(s))]
        assert lib.minmod(_p(*d), _p(*b)) == want, (d, b)


@pytest.mark.parametrize("size", [1e-150, 1e-60, 1e-42, 1e-25, 1e-20, 1e-19, 1e-12, 1.0, 1e12, 1e18, 1e20, 1e30, 1e38, 1e60, 1e150])
@pytest.mark.parametrize("ratio", [1e-4, 1.0, 1e4])
def test_wave_speed_is_the_larger_one(lib, size, ratio):
    rng = np.random.default_rng(5)
    for it in range(400):
        v = size * ratio * rng.uniform(-1.0, 1.0, 2)
        c = (size * rng.uniform(0.1, 3.0, 2)) ** 2 * rng.choice([1.0, 1.0, 0.0, -1.0], 2)
        want = max(abs(v) + np.sqrt(np.maximum(c, 0.0)))
        assert lib.speed(_p(v[0], c[0], v[1], c[1])) == want, (v, c)


@pytest.mark.parametrize("x", [1.0, -3.1415926535, 1e-30, 2.0 ** -126, 3.4e38, -2.0 ** 128, 1e39, -1e300, float("inf"),
                               float("nan"), 0.0, -0.0, 1e-40, -1e-300])
def test_truncation(lib, x):
    y = lib.truncated(x)
    if not abs(x) < 2.0 ** 128:
        assert abs(y) == np.inf and (np.isnan(x) or np.sign(y) == np.sign(x))
    elif abs(x) >= 2.0 ** -126:
        assert 0 <= (x - y) / x < 2.0 ** -23
    else:
        assert abs(y) < 2.0 ** -126


@pytest.mark.parametrize("size", SIZES)
def test_no_inadmissible_state_is_clear(lib, size):
    """Euler states whose pressure is negative, for the reason of one momentum or energy
    of another size than the rest."""
    rng = np.random.default_rng(4)
    for it in range(400):
        with np.errstate(over="ignore"):
            rho, mom, e = np.minimum(size * 10.0 ** (rng.uniform(-40, 40, 3) if it % 2 else rng.uniform([0, 0, 0], [4, 40, 4])), 1e150)
        s = np.array([rho, mom, rng.choice([-1.0, 0.0, 1.0]) * mom, e])
        with np.errstate(over="ignore", divide="ignore", invalid="ignore", under="ignore"):
            p = 0.4 * (s[3] - 0.5 * (s[1] / s[0] * s[1] + s[2] / s[0] * s[2]))
        if not (s[0] >= 1e-12 and p >= 1e-12):
            assert not lib.above_eps(_p(*s)), s


@pytest.mark.parametrize("size", SIZES + [1e-9, 1e-10, 3e-11, 1e-11, 3e-12, 1e-12, 1e-13, 1e-19, 1e-21])
@pytest.mark.parametrize("m", [4, 6])
def test_states_at_and_past_the_edge_are_not_clear(lib, size, m):
    """Pressures (ten-moment: their determinants) of 0 and below, at every size; and
    ordinary states are clear."""
    rng = np.random.default_rng(6)
    for it in range(400):
        rho, v1, v2, a, b = np.exp(rng.uniform(-3.0, 3.0, 5)) * np.array([1.0, *rng.choice([-1.0, 1.0], 2), 1.0, 1.0])
        if it % 2 and m == 6:
            v1 = v2 = 0.0
        over = rng.choice([1.0, 1.0 + 1e-6, 1.0 + 1e-3, 2.0])
        if m == 4:
            u = np.array([rho, rho * v1, rho * v2, 0.5 * rho * (v1 * v1 + v2 * v2) / over])
            good = u + np.array([0.0, 0.0, 0.0, a + u[3]])
        else:
            u = np.array([rho, rho * v1, rho * v2, 0.5 * (a + rho * v1 * v1), 0.5 * (over * np.sqrt(a * b) + rho * v1 * v2),
                          0.5 * (b + rho * v2 * v2)])
            good = np.array([rho, 0.0, 0.0, 0.5 * a, 0.1 * min(a, b), 0.5 * b])
        scale = 2.0 ** np.round(np.log2(size))            # (exactly the same state at another size)
        with np.errstate(under="ignore"):
            assert not lib.admissible(_p(*(u * scale)), m), u
        if 1e-3 < size < 1e3:
            assert lib.admissible(_p(*(good * scale)), m), good


def _flux(u):
    v = u[1] / u[0]
    if len(u) == 4:
        p = 0.4 * (u[3] - 0.5 * (u[1] ** 2 + u[2] ** 2) / u[0])
        return np.array([u[1], u[1] * v + p, u[2] * v, (u[3] + p) * v]), abs(v) + np.sqrt(1.4 * p / u[0])
    v2 = u[2] / u[0]
    p11, p12 = 2 * u[3] - u[1] * v, 2 * u[4] - u[1] * v2
    f = np.array([u[1], p11 + u[1] * v, p12 + u[1] * v2, (u[3] + p11) * v, u[4] * v + 0.5 * (p11 * v2 + p12 * v), u[5] * v + p12 * v2])
    return f, abs(v) + np.sqrt(3 * p11 / u[0])


def _constraints(u):
    if len(u) == 4:
        return np.array([u[0], 0.4 * (u[3] - 0.5 * (u[1] ** 2 + u[2] ** 2) / u[0])])
    p11, p12, p22 = 2 * u[3] - u[1] ** 2 / u[0], 2 * u[4] - u[1] * u[2] / u[0], 2 * u[5] - u[2] ** 2 / u[0]
    return np.array([u[0], 0.5 * (p11 + p22) - np.sqrt((0.5 * (p11 - p22)) ** 2 + p12 ** 2)])


@pytest.mark.parametrize("size", [2.0 ** k for k in (-500, -200, -150, -140, -126, -120, -100, -80, -70, -66, -63, -60, -50, -40,
                                                     -30, 0, 40, 80, 120, 126, 200, 500)])
@pytest.mark.parametrize("m", [4, 6])
def test_idle_flux_limiter(lib, m, size):
    """Where the screen calls the flux limiter idle, both candidates with the flux F
    keep a tenth of the smaller low-order candidate in every constraint (1e-9 of the
    constraint's own rounding aside)."""
    rng = np.random.default_rng(7)

    def state():
        rho, a, b = np.exp(rng.uniform(-2.0, 2.0, 3))
        v1, v2 = rng.uniform(-1.0, 1.0, 2)
        if m == 4:
            return np.array([rho, rho * v1, rho * v2, a / 0.4 + 0.5 * rho * (v1 * v1 + v2 * v2)])
        r = rng.choice([0.0, 0.9, 1.0 - 1e-3, 1.0 - 1e-6]) * rng.choice([-1.0, 1.0]) * np.sqrt(a * b)
        return 0.5 * np.array([2 * rho, 2 * rho * v1, 2 * rho * v2, a + rho * v1 * v1, r + rho * v1 * v2, b + rho * v2 * v2])

    clear = 0
    for it in range(500):
        uL, uR, bL, bR = (state() for _ in range(4))
        (fL, sL), (fR, sR) = _flux(uL), _flux(uR)
        lam = max(sL, sR)
        low = 0.5 * (fL + fR) - 0.5 * lam * (uR - uL)
        F = low + lam * rng.choice([0.01, 0.3, 3.0]) * rng.standard_normal(m)
        c = 10.0 ** rng.uniform(-3.0, -0.3, 2) / lam
        if not lib.idle(_p(*(size * np.concatenate([uL, uR, bL, bR, F]))), m, ctypes.c_double(c[0]), ctypes.c_double(c[1])):
            continue
        clear += 1
        lo = np.minimum(_constraints(bL - c[0] * low), _constraints(bR + c[1] * low))
        hi = np.minimum(_constraints(bL - c[0] * F), _constraints(bR + c[1] * F))
        assert (hi >= 0.1 * lo - 1e-9 * abs(hi)).all(), (it, lo, hi)
    assert clear > 20 or not 2.0 ** -30 <= size <= 2.0 ** 40


@pytest.mark.parametrize("m", [4, 6])
def test_constraints_are_the_formula(lib, m):
    """One rounding per operation (no reciprocal in the place of a division), and no
    number where an entry is none."""
    rng = np.random.default_rng(8)
    for it in range(2000):
        u = rng.standard_normal(m) * 10.0 ** rng.uniform(-3, 3, m)
        u[0] = abs(u[0])
        if m == 4:
            want = 0.4 * (u[3] - 0.5 * (u[1] * u[1] + u[2] * u[2]) / u[0])
        else:
            r = 1.0 / u[0]
            p11, p12, p22 = 2.0 * u[3] - u[1] * u[1] * r, 2.0 * u[4] - u[1] * u[2] * r, 2.0 * u[5] - u[2] * u[2] * r
            h = 0.5 * (p11 - p22)
            want = 0.5 * (p11 + p22) - np.sqrt(h * h + p12 * p12)
        assert lib.constraint(_p(*u), m) == want
        u[rng.integers(0, m)] = np.nan
        assert np.isnan(lib.constraint(_p(*u), m))


@pytest.mark.parametrize("m", [4, 6])
@pytest.mark.parametrize("unlike", [1.0, 2.0, 10.0, 1e3, 1e6])
def test_margins_of_the_low_order_fluxes(lib, m, unlike):
    """The FP32 Rusanov flux of any two states within its own margin, at Mach numbers up
    to 200; and that between a node and an inner neighbour, where the two are alike,
    within the margin of a face whose two sides are like the node."""
    rng = np.random.default_rng(9)
    f32 = lambda k: (ctypes.c_float * k)()  # noqa: E731
    seen = 0
    for it in range(3000):
        pair = []
        for i in range(2):
            rho, mach = unlike ** rng.uniform(-i, i), 10.0 ** rng.uniform(-1.0, 2.3)
            a, b = rho * unlike ** rng.uniform(-i, i) * np.exp(rng.uniform(-1.0, 1.0, 2))
            v1, v2 = mach * np.sqrt(1.4 * a / rho) * rng.uniform(-1.0, 1.0, 2)
            if m == 4:
                pair.append(np.array([rho, rho * v1, rho * v2, a / 0.4 + 0.5 * rho * (v1 * v1 + v2 * v2)]))
            else:
                r = rng.uniform(-0.9, 0.9) * np.sqrt(a * b)
                pair.append(0.5 * np.array([2 * rho, 2 * rho * v1, 2 * rho * v2, a + rho * v1 * v1, r + rho * v1 * v2,
                                            b + rho * v2 * v2]))
        (fL, sL), (fR, sR) = _flux(pair[0]), _flux(pair[1])
        want = 0.5 * (fL + fR) - 0.5 * max(sL, sR) * (pair[1] - pair[0])
        lo, a, lo2, a2 = f32(m), f32(m), f32(m), f32(m)
        lib.low_flux(_p(*np.concatenate(pair)), m, lo, a)
        err = np.abs(np.array(lo[:], dtype=np.float64) - want)
        assert not (err > 2e-5 * np.array(a[:])).any(), (it, pair, err, a[:])
        if lib.like(_p(*np.concatenate(pair)), m):
            seen += 1
            lib.low_flux(_p(*np.concatenate([pair[0], pair[0]])), m, lo2, a2)
            assert not (err > 2e-5 * np.array(a2[:])).any(), (it, pair, err, a2[:])
    assert seen > 100 or unlike > 2.0
