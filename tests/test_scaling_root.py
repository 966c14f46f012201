"""The scaling limiter's theta (csrc/cr_root.cuh), compiled for the host, against 50
bisections of [0, 1], over jets and near-vacuum points, means next to the edge of
admissibility, points that are barely inadmissible and states of any size; and on
ordinary states with a fraction of their evaluations.

Euler: bit for bit the bisection's point.  Ten-moment: a point at which the
constraint as computed holds and 2^6 steps of d = 8 2^-53 (B_rho B_E + B_m^2) / |dq/dtheta| +
2^-50 further on, at most, it fails; the bisection ends between two such points as
well, so the two are within 2^7 d of each other, where B_v is the larger magnitude of
the two ends and q the smaller eigenvalue of rho (P - eps).
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from tests import test_screens

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = "#define __noinline__\n" + test_screens.SRC.split('#include "cr_screen.cuh"')[0] + r"""
#include "cr_root.cuh"
using namespace crk;
static int evaluations;
template <class EQ> struct Counted : EQ {
  static double constraint(const double* u, int k, const Phys<double>& ph) {
    ++evaluations;
    return EQ::constraint(u, k, ph);
  }
};
namespace crk {
template <int DIM> struct IsEuler<Counted<EqEuler<DIM>>> { static constexpr bool value = true; };
}
template <class EQ> static void both(const double* ubar, const double* pt, double eps, double* out) {
  Phys<double> ph{};
  ph.gm1 = 0.4;
  evaluations = 0;
  out[0] = scaling_root<Counted<EQ>, true>(ubar, pt, eps, ph);
  out[1] = evaluations;
  double lo = 0.0, hi = 1.0, u[6];
  for (int i = 0; i < 50; ++i) {
    const double mid = 0.5 * (lo + hi);
    for (int v = 0; v < EQ::M; ++v) u[v] = ubar[v] + mid * (pt[v] - ubar[v]);
    (EQ::constraint(u, 1, ph) >= eps ? lo : hi) = mid;
  }
  out[2] = lo;
}
extern "C" {
double constraint(const double* u, int m) {
  Phys<double> ph{};
  ph.gm1 = 0.4;
  return m == 3 ? EqEuler<1>::constraint(u, 1, ph) : m == 4 ? EqEuler<2>::constraint(u, 1, ph) : EqTenMoment::constraint(u, 1, ph);
}
void roots(const double* ubar, const double* pt, double eps, int m, double* out) {
  if (m == 3) both<EqEuler<1>>(ubar, pt, eps, out);
  else if (m == 4) both<EqEuler<2>>(ubar, pt, eps, out);
  else both<EqTenMoment>(ubar, pt, eps, out);
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("root")
    src, out = d / "root.cpp", d / "libroot.so"
    src.write_text(SRC)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"),
                    "-I", os.path.join(ROOT, "paper_2502_07517_gb300", "csrc"), str(src), "-o", str(out)], check=True)
    lib = ctypes.CDLL(str(out))
    lib.constraint.restype = ctypes.c_double
    return lib


def _p(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))


def _state(rng, m, speed):
    rho, v = np.exp(rng.uniform(-2, 2)), speed * rng.uniform(-1, 1, 2)
    a, b = np.exp(rng.uniform(-2, 2, 2))
    if m == 3:
        return np.array([rho, rho * v[0], a / 0.4 + 0.5 * rho * v[0] ** 2])
    if m == 4:
        return np.array([rho, rho * v[0], rho * v[1], a / 0.4 + 0.5 * rho * (v @ v)])
    r = rng.uniform(-1, 1) * np.sqrt(a * b)
    return 0.5 * np.array([2 * rho, 2 * rho * v[0], 2 * rho * v[1], a + rho * v[0] ** 2, r + rho * v[0] * v[1], b + rho * v[1] ** 2])


def _step(ubar, pt, eps, theta):
    B = np.maximum(abs(ubar), abs(pt))
    scale = max(B)                             # (q is of second order in the state)

    def q(th):
        u = (ubar + th * (pt - ubar)) / scale
        e = eps / scale
        a, b, c = u[0] * (2 * u[3] - e) - u[1] ** 2, u[0] * 2 * u[4] - u[1] * u[2], u[0] * (2 * u[5] - e) - u[2] ** 2
        return 0.5 * (a + c) - np.hypot(0.5 * (a - c), b)

    h = 1e-6 * min(theta, 1.0 - theta) + 1e-12
    slope = abs(q(theta + h) - q(theta - h)) / (2 * h)
    size = (B[0] * (B[3] + B[5]) + B[1] ** 2 + B[2] ** 2) / scale ** 2
    return 8 * 2.0 ** -53 * size / slope + 2.0 ** -50


@pytest.mark.parametrize("m", [3, 4, 6])
@pytest.mark.parametrize("kind", ["ordinary", "jet", "vacuum", "any size", "barely", "mean at the edge"])
def test_theta_is_the_bisections(lib, m, kind):
    rng = np.random.default_rng(m)
    out, counts = np.zeros(3), []
    for it in range(1500):
        ubar = _state(rng, m, 1.0 if kind == "ordinary" else 10.0 ** rng.uniform(-2.0, 3.5))
        if kind == "any size":
            ubar = ubar * 10.0 ** rng.uniform(-150, 120)
        if kind == "jet":
            pt = ubar * rng.uniform(-0.5, 2.0) + 0.01 * rng.standard_normal(m) * abs(ubar)
        elif kind == "vacuum":
            pt = ubar * rng.uniform(0.5, 1.5, m) * rng.choice([-1.0, 1.0], m)
        elif kind == "barely":
            pt = ubar * (1.0 + rng.standard_normal(m) * 10.0 ** rng.uniform(-12, 0))
            pt[-1] -= abs(ubar[-1]) * 10.0 ** rng.uniform(-12, 0)
        else:
            pt = ubar + rng.standard_normal(m) * abs(ubar)
        floor = min(1e-12, ubar[0])
        if pt[0] < floor:                       # as the limiter's density scaling leaves it
            pt[0] = ubar[0] + (ubar[0] - floor) / (ubar[0] - pt[0]) * (pt[0] - ubar[0])
        if kind == "vacuum" and it % 2:
            pt[0] = 10.0 ** rng.uniform(-16, -2) * rng.choice([1.0, 1.0, 0.0])
        P = lib.constraint(_p(ubar), m)
        if not P > 0:
            continue
        eps = P * rng.choice([1.0, 0.5, 1.0 - 1e-14]) if kind == "mean at the edge" else min(1e-12, P)
        if lib.constraint(_p(pt), m) >= eps:
            continue
        lib.roots(_p(ubar), _p(pt), ctypes.c_double(eps), m, _p(out))
        if m < 6:
            assert out[0] == out[2], (it, ubar, pt, eps, out)
        else:
            off = abs(out[0] - out[2])
            assert off <= 128 * _step(ubar, pt, eps, out[2]), (it, ubar, pt, eps, out, off)
            at = ubar + out[0] * (pt - ubar)
            assert out[0] == out[2] or lib.constraint(_p(at), m) >= eps
        counts.append(out[1])
    # (at most all of the bisection, ten-moment after the seven of the attempt)
    assert len(counts) > 150 and max(counts) <= (50 if m < 6 else 57)
    if kind == "ordinary":
        assert np.mean(counts) < (8 if m < 6 else 6)
