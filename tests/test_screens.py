"""The FP32 screens in front of FP64 decisions (csrc/cr_screen.cuh), compiled for
the host: over all magnitudes of the data, also those outside FP32's range, a
screen that answers must answer as FP64 does.
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
    lib.minmod.restype = lib.speed.restype = ctypes.c_double
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
