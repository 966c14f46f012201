"""The fixed-point dot products of the FP64 element kernel (csrc/cr_fixed.cuh),
compiled for the host and compared with exact rational arithmetic.

Bound of one sum over two lines of n terms with a common product scale, from the
format: per term the value's truncation (2^-56 of the larger max|a| max|x| of the
two lines), the coefficient's rounding (2^-57) and the dropped product of the low
limbs (2^-56), the shift at the end (2^-57), and one rounding of the result (2^-53
of it).  Values below 2^-959 keep the unit 2^-1016 of the smallest exponent, and
results below 2^-1022 become 0 (FP64 itself has nothing finer than 2^-1074 there).
"""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

import oracle

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "cr_fixed.cuh"
using namespace crk;
extern "C" double two_lines(const double* A, const double* x, int nx, const double* B, const double* y, int ny,
                            const double* whole_a, const double* whole_b, int nw, int below) {
  const int sa = fix_scale(whole_a, nw), sb = fix_scale(whole_b, nw), oa = fix_exp(sa), ob = fix_exp(sb);
  int k = kMinLineExp + (oa > ob ? oa : ob);
  for (int i = 0; i < nx; ++i) if (exp_of(x[i]) + oa > k) k = exp_of(x[i]) + oa;
  for (int i = 0; i < ny; ++i) if (exp_of(y[i]) + ob > k) k = exp_of(y[i]) + ob;
  if (k - below - (oa > ob ? oa : ob) >= kMinLineExp) k -= below;
  FixAcc acc{0, 0};
  for (int i = 0; i < nx; ++i) fix_mad(acc, to_fixed(x[i], k - oa), fix_coef(A[i], sa));
  for (int i = 0; i < ny; ++i) fix_mad(acc, to_fixed(y[i], k - ob), fix_coef(B[i], sb));
  return from_fixed(fix_sum(acc), k);
}
"""


@pytest.fixture(scope="module")
def two_lines(tmp_path_factory):
    d = tmp_path_factory.mktemp("fixed")
    src, lib = d / "fixed.cpp", d / "libfixed.so"
    src.write_text(SRC)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"), "-I",
                    os.path.join(ROOT, "paper_2502_07517_gb300", "csrc"), str(src), "-o", str(lib)], check=True)
    f = ctypes.CDLL(str(lib)).two_lines
    P, I = ctypes.POINTER(ctypes.c_double), ctypes.c_int
    f.argtypes, f.restype = [P, P, I, P, P, I, P, P, I, I], ctypes.c_double
    p = lambda a: np.ascontiguousarray(a).ctypes.data_as(P)

    def call(A, x, B, y, DA, DB, below):
        A, x, B, y, DA, DB = (np.ascontiguousarray(a, dtype=np.float64) for a in (A, x, B, y, DA, DB))
        return f(p(A), p(x), len(x), p(B), p(y), len(y), p(DA), p(DB), DA.size, below)
    return call


LINES = {
    "smooth": lambda r, n: 1.0 + 0.01 * r.standard_normal(n),
    "rough": lambda r, n: r.standard_normal(n),
    "steep": lambda r, n: np.exp(3.0 * r.standard_normal(n)) * r.choice([-1.0, 1.0], n),
    "huge": lambda r, n: 1e200 * r.standard_normal(n),
    "tiny": lambda r, n: 1e-200 * r.standard_normal(n),
    "mixed": lambda r, n: r.choice([0.0, -0.0, 5e-324, 1e-30, 1.0, -3.0], n),
    "zero": lambda r, n: np.zeros(n),
}


@pytest.mark.parametrize("N", [1, 2, 3, 4])
@pytest.mark.parametrize("kind", sorted(LINES))
@pytest.mark.parametrize("below", [0, 1])
def test_two_line_dot_products(two_lines, N, kind, below):
    rng = np.random.default_rng(N + 10 * below)
    n = N + 1
    D = oracle.tables(N)[4]
    err_fix = err_fma = 0.0
    for it in range(60):
        sx, sy = 10.0 ** rng.uniform(-3, 3, 2)   # 1/dx, 1/dy of an anisotropic mesh
        DA, DB = D * sx, D * sy
        x, y = LINES[kind](rng, n), LINES[kind](rng, n)
        for p in range(n):
            got = two_lines(DA[p], x, DB[p], y, DA, DB, below)
            tx = [Fraction(float(a)) * Fraction(float(b)) for a, b in zip(DA[p], x)]
            ty = [Fraction(float(a)) * Fraction(float(b)) for a, b in zip(DB[p], y)]
            want = sum(tx) + sum(ty)
            tops = Fraction(float(np.abs(DA).max())) * Fraction(float(np.abs(x).max())), \
                Fraction(float(np.abs(DB).max())) * Fraction(float(np.abs(y).max()))
            top = max(tops)
            amax = Fraction(float(max(np.abs(DA).max(), np.abs(DB).max())))
            tops_scale = amax / Fraction(float(min(np.abs(DA).max(), np.abs(DB).max())))
            bound = top * Fraction(5 * 2 * n + 1, 2 ** 57) + abs(want) / 2 ** 53 \
                + (2 * n * amax * max(tops_scale, 1) + 1) / Fraction(2 ** 1016)
            e = abs(Fraction(got) - want)
            assert e <= bound, (it, p, float(e), float(bound))
            if kind in ("smooth", "rough") and top > 0:
                c = 0.0
                for a, b in list(zip(DA[p], x)) + list(zip(DB[p], y)):  # one FMA at a time, exactly rounded
                    c = float(Fraction(float(a)) * Fraction(float(b)) + Fraction(c))
                err_fix += float(e / top)
                err_fma += float(abs(Fraction(c) - want) / top)
    assert err_fix <= err_fma  # no further from the exact sums than the FMA chain, on average
