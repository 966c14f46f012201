"""The FP64 element kernel in two dimensions where its arithmetic changes path:
lines of nodes that outgrow their fixed-point exponent within a step (large
steps: stage values grow by orders of magnitude), strongly anisotropic meshes
(the x and y contractions have very different scales), elements whose nodes
differ by orders of magnitude (MUSCL-Hancock decisions near their limits, all
limiters at work), and steps whose values overflow.

Tolerance: the 1e-12 relative bar of tests/test_gpu_parity.py, per variable of
the largest value and flux increment; in the growth cases the scale is the
largest result (both sides round values of that size).
"""
import numpy as np
import pytest

import oracle
from paper_2502_07517_gb300 import crkfr
from paper_2502_07517_gb300 import workloads as wl
from tests._oracle_util import oracle_desc
from tests.test_gpu_parity import assert_parity, flux_increment, gpu_run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_07517_gb300 import build
    build.build()


@pytest.mark.parametrize("N", [1, 2, 3, 4])
@pytest.mark.parametrize("times", [3.0, 100.0, 1e6])
def test_lines_outgrow_their_exponent(N, times):
    prob, u = wl.linadv_random(nx=13, ny=11, dim=2, degree=N, seed=N, adv=(0.7, -1.2))
    d = oracle_desc(prob)
    dt = times * oracle.dt(d, u)
    ref, st = oracle.step(d, u, dt)[:2]
    assert st == 0
    g = gpu_run(prob, u, dt_fixed=dt)[0]
    assert_parity(g, ref)


@pytest.mark.parametrize("N", [2, 3, 4])
@pytest.mark.parametrize("wide", [1e-4, 1e4])
def test_anisotropic_mesh(N, wide):
    prob, u = wl.euler2d_vortex(nx=9, ny=14, degree=N, seed=N)
    prob = dict(prob, x0=-5.0 * wide, x1=5.0 * wide)
    u = u * np.random.default_rng(N).uniform(0.7, 1.4, (1, u.shape[1], 1))
    d = oracle_desc(prob)
    dt = oracle.dt(d, u)
    ref, st, dg = oracle.step(d, u, dt, want_diag=True)
    assert st == 0
    g = gpu_run(prob, u, dt_fixed=dt)[0]
    assert_parity(g, ref, extra_scale=flux_increment(prob, dg, dt))


@pytest.mark.parametrize("N", [2, 3, 4])
@pytest.mark.parametrize("seed", [0, 1])
def test_steep_nodes(N, seed):
    rng = np.random.default_rng(seed)
    prob, u = wl.euler2d_vortex(nx=12, ny=7, degree=N, seed=seed)
    shape = u.shape[1:]
    p = np.exp(rng.uniform(np.log(1e-3), np.log(10.0), shape))
    rho = np.exp(rng.uniform(np.log(0.3), np.log(3.0), shape))
    u = wl.euler_conservative(rho, rng.uniform(-1, 1, shape), rng.uniform(-1, 1, shape), p, 1.4, 2)
    d = oracle_desc(prob)
    dt = 0.2 * oracle.dt(d, u)
    ref, st, dg = oracle.step(d, u, dt, want_diag=True)
    assert st == 0
    g = gpu_run(prob, u, dt_fixed=dt)[0]
    assert_parity(g, ref, extra_scale=flux_increment(prob, dg, dt))


def test_overflowing_step_is_reported():
    prob, u = wl.linadv_random(nx=6, ny=5, dim=2, degree=4, seed=1, adv=(1.0, 1.0))
    ctx = crkfr.cr_init_mesh(crkfr.desc_from_problem(prob))
    crkfr.cr_set_state(ctx, u)
    with pytest.raises(crkfr.CrError) as err:
        crkfr.cr_step(ctx, 1, 1e300, 1e100)
    assert err.value.status == -3
    crkfr.cr_set_state(ctx, u)       # the context stays usable
    crkfr.cr_step(ctx, 1, 1e300)


@pytest.mark.parametrize("N", [2, 3, 4])
@pytest.mark.parametrize("pressure", [1e-3, 3e-5, 1e-5])
def test_low_pressure_beside_the_screens(N, pressure):
    """Mach 30 to 300: pressures above, about and below the margin of the FP32
    screens (2e-5 of the energies), so limiters and MUSCL-Hancock decide in FP32
    in some nodes and in FP64 in others.  The constraint P is a difference of
    energies E: its relative rounding, a few 2^-53 E / P (ten of them here), goes
    into the limiters' theta on top of the 1e-12 bar."""
    rng = np.random.default_rng(N)
    prob, u = wl.euler2d_vortex(nx=11, ny=9, degree=N, seed=N)
    shape = (u.shape[1], 1)
    one = np.ones(u.shape[1:])
    rho, p = one * rng.uniform(0.8, 1.2, shape), pressure * one * rng.uniform(0.5, 2.0, shape)
    u = wl.euler_conservative(rho, one * rng.uniform(0.9, 1.1, shape), one * rng.uniform(-0.1, 0.1, shape), p, 1.4, 2)
    d = oracle_desc(prob)
    dt = 0.5 * oracle.dt(d, u)
    ref, st, dg = oracle.step(d, u, dt, want_diag=True)
    assert st == 0
    g = gpu_run(prob, u, dt_fixed=dt)[0]
    bar = 1e-12 + 10 * 2.0 ** -53 * u[3].max() / p.min()
    assert_parity(g, ref, rtol=bar, extra_scale=flux_increment(prob, dg, dt))


@pytest.mark.parametrize("eq,N,nx,ny", [("euler", 1, 171, 170), ("euler", 1, 171, 171), ("euler", 2, 113, 112),
                                        ("euler", 2, 113, 114), ("euler", 3, 86, 84), ("euler", 3, 86, 85),
                                        ("tenmoment", 3, 70, 69), ("tenmoment", 3, 70, 70)])
def test_meshes_about_the_resident_blocks(eq, N, nx, ny):
    """Meshes that just fit on the chip at once and that just do not (the element
    kernel then asks for one block more per SM)."""
    make = wl.euler2d_vortex if eq == "euler" else wl.tenmoment2d_voronoi
    prob, u = make(nx=nx, ny=ny, degree=N, seed=N)
    d = oracle_desc(prob)
    dt = 0.5 * oracle.dt(d, u)
    ref, st, dg = oracle.step(d, u, dt, want_diag=True)
    assert st == 0
    g = gpu_run(prob, u, dt_fixed=dt)[0]
    assert_parity(g, ref, extra_scale=flux_increment(prob, dg, dt))


@pytest.mark.parametrize("N", [2, 3, 4])
def test_alpha_beside_its_threshold(N):
    """Elements whose modal energy fraction lies within a few percent of the one
    at which alpha becomes 0: the FP32 screen may call none of them wrongly."""
    rng = np.random.default_rng(N)
    prob, u = wl.euler2d_vortex(nx=16, ny=8, degree=N, seed=N, perturb=0.0)
    prob = dict(prob, limiter=frozenset({"blend", "flux", "scaling", "traces"}))
    T, s = 0.5 * 10.0 ** (-1.8 * (N + 1.0) ** 0.25), np.log((1.0 - 1e-4) / 1e-4)
    edge = T * (1.0 - np.log(999.0) / s)
    xi, _ = wl.gl_nodes01(N)
    top = np.polynomial.legendre.Legendre.basis(N)(2.0 * xi - 1.0)     # along x; rho p = 1 + c L_N(x)
    frac = edge * rng.uniform(0.9, 1.1, u.shape[1])
    c = np.sqrt(frac / (1.0 - frac))
    rho = np.ones(u.shape[1:])
    p = 1.0 + c[:, None] * np.tile(top, N + 1)[None, :]
    u = wl.euler_conservative(rho, 0.1 * rho, 0.0 * rho, p, 1.4, 2)
    d = oracle_desc(prob)
    dt = 0.1 * oracle.dt(d, u)
    ref, st, dg = oracle.step(d, u, dt, want_diag=True)
    assert st == 0 and 0 < np.count_nonzero(dg["alpha_raw"]) < u.shape[1]
    g, alpha = gpu_run(prob, u, dt_fixed=dt)[:2]
    np.testing.assert_allclose(alpha, dg["alpha"], rtol=0, atol=1e-12)
    assert_parity(g, ref, extra_scale=flux_increment(prob, dg, dt))
