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
extern "C" {
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
    lib.minmod.restype = ctypes.c_double
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
