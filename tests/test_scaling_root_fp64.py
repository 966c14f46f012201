"""theta of FP64 ten-moment states (csrc/cr_root.cuh), compiled for the host: bit for bit
the point that 50 bisections end at, over the states of tests/test_scaling_root.py, and on
ordinary ones with a fraction of their evaluations.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from tests import test_scaling_root as tsr


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("root64")
    src, out = d / "root.cpp", d / "libroot.so"
    src.write_text(tsr.SRC.replace("scaling_root<Counted<EQ>, true>", "scaling_root<Counted<EQ>, false>"))
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I", os.path.join(cuda, "include"),
                    "-I", os.path.join(tsr.ROOT, "paper_2502_07517_gb300", "csrc"), str(src), "-o", str(out)], check=True)
    lib = ctypes.CDLL(str(out))
    lib.constraint.restype = ctypes.c_double
    return lib


@pytest.mark.parametrize("kind", ["ordinary", "jet", "vacuum", "any size", "barely", "mean at the edge"])
def test_ten_moment_theta_is_the_bisections(lib, kind):
    rng, out, counts = np.random.default_rng(6), np.zeros(3), []
    for it in range(3000):
        ubar = tsr._state(rng, 6, 1.0 if kind == "ordinary" else 10.0 ** rng.uniform(-2.0, 3.5))
        if kind == "any size":
            ubar = ubar * 10.0 ** rng.uniform(-150, 120)
        if kind == "jet":
            pt = ubar * rng.uniform(-0.5, 2.0) + 0.01 * rng.standard_normal(6) * abs(ubar)
        elif kind == "vacuum":
            pt = ubar * rng.uniform(0.5, 1.5, 6) * rng.choice([-1.0, 1.0], 6)
        elif kind == "barely":
            pt = ubar * (1.0 + rng.standard_normal(6) * 10.0 ** rng.uniform(-12, 0))
            pt[-1] -= abs(ubar[-1]) * 10.0 ** rng.uniform(-12, 0)
        else:
            pt = ubar + rng.standard_normal(6) * abs(ubar)
        floor = min(1e-12, ubar[0])
        if pt[0] < floor:
            pt[0] = ubar[0] + (ubar[0] - floor) / (ubar[0] - pt[0]) * (pt[0] - ubar[0])
        if kind == "vacuum" and it % 2:
            pt[0] = 10.0 ** rng.uniform(-16, -2) * rng.choice([1.0, 1.0, 0.0])
        P = lib.constraint(tsr._p(ubar), 6)
        if not P > 0:
            continue
        eps = P * rng.choice([1.0, 0.5, 1.0 - 1e-14]) if kind == "mean at the edge" else min(1e-12, P)
        if lib.constraint(tsr._p(pt), 6) >= eps:
            continue
        lib.roots(tsr._p(ubar), tsr._p(pt), ctypes.c_double(eps), 6, tsr._p(out))
        assert out[0] == out[2], (it, ubar, pt, eps, out)
        counts.append(out[1])
    assert len(counts) > 300 and max(counts) <= 50
    if kind == "ordinary":
        assert np.mean(counts) < 14
