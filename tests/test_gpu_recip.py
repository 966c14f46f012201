"""The reciprocal and the square root of the FP64 kernels (recip, sqrt_pos in
csrc/cr_common.cuh) against the exact values, over all exponents, and at 0, subnormal
numbers, infinities, NaN and negative numbers against IEEE division and square root.

Bound: recip's step leaves e^3 < 2^-60 of the hardware approximation's relative error
e < 2^-20, sqrt_pos's second Newton step a residual of 2^-40 times an error of 2^-20 in its
factor, 2^-60 too: 2^-7 units in the last place, on top of the last FMA's 0.5; twice
that 2^-7 and the rounding of the reference allowed: 0.53 units in the last place.
Outside 2^-1000 .. 2^1000 recip multiplies by a power of two (a second rounding below
2^-1022): one unit.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "cr_common.cuh"
__global__ void k(const double* x, double* r, double* s, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    r[i] = crk::recip(x[i]);
    s[i] = crk::sqrt_pos(x[i]);
  }
}
extern "C" int run(const double* x, double* r, double* s, int n) {
  double* d = nullptr;
  if (cudaMalloc(&d, sizeof(double) * 3 * size_t(n)) != cudaSuccess) return 1;
  cudaMemcpy(d, x, sizeof(double) * n, cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * size_t(n), n);
  cudaMemcpy(r, d + n, sizeof(double) * n, cudaMemcpyDeviceToHost);
  cudaMemcpy(s, d + 2 * size_t(n), sizeof(double) * n, cudaMemcpyDeviceToHost);
  const cudaError_t e = cudaGetLastError();
  cudaFree(d);
  return int(e);
}
"""


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_07517_gb300 import build
    d = tmp_path_factory.mktemp("recip")
    src, out = d / "recip.cu", d / "librecip.so"
    src.write_text(SRC)
    subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS + ["-I" + build.CSRC, "-shared", str(src), "-o", str(out)], check=True)
    run = ctypes.CDLL(str(out)).run
    p = lambda a: a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))  # noqa: E731

    def call(x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        r, s = np.empty_like(x), np.empty_like(x)
        assert run(p(x), p(r), p(s), x.size) == 0
        return r, s
    return call


def _units(got, exact):
    """Error in units in the last place of the exact value."""
    ulp = np.spacing(np.abs(exact.astype(np.float64)))
    return np.abs((got.astype(np.longdouble) - exact) / ulp)


@pytest.mark.parametrize("kind", ["random", "few bits", "next to powers of two"])
def test_error(call, kind):
    rng = np.random.default_rng(1)
    e = np.repeat(np.arange(-1000, 1000), 500)
    m = rng.uniform(1.0, 2.0, e.size)
    if kind == "few bits":
        m = 1.0 + rng.integers(0, 256, e.size) / 256.0
    elif kind == "next to powers of two":
        m = np.where(rng.random(e.size) < 0.5, 1.0 + rng.integers(0, 64, e.size) * 2.0 ** -52, 2.0 - rng.integers(1, 64, e.size) * 2.0 ** -52)
    x = np.ldexp(m, e)
    r, s = call(x)
    assert _units(r, 1.0 / x.astype(np.longdouble)).max() <= 0.53
    inside = e >= -899
    assert _units(s, np.sqrt(x.astype(np.longdouble)))[inside].max() <= 0.53
    assert (s[~inside] == np.sqrt(x[~inside])).all()


def test_edges(call):
    rng = np.random.default_rng(2)
    with np.errstate(all="ignore"):
        x = np.concatenate([[0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.0 ** -1022, 2.0 ** -1024, 2.0 ** 1023,
                             np.finfo(float).max, -1.0, -2.0 ** -1000, 2.0 ** -1000, 2.0 ** 1000],
                            np.ldexp(rng.uniform(1.0, 2.0, 4000), rng.integers(-1074, -990, 4000)),
                            np.ldexp(rng.uniform(1.0, 2.0, 4000), rng.integers(990, 1024, 4000))])
        x = np.concatenate([x, -x])
        r, s = call(x)
        want = 1.0 / x
        same = (r == want) | (np.isnan(r) & np.isnan(want))
        near = np.abs(r - want) <= np.spacing(np.abs(want))
        assert (same | near).all(), x[~(same | near)]
        assert (np.signbit(r) == np.signbit(want))[~np.isnan(want)].all()
        root = np.sqrt(np.where(x > 0, x, 0.0))
        assert ((s == root) | (np.abs(s - root) <= np.spacing(root))).all()
