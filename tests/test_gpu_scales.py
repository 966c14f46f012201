"""Data far from 1: states scaled by powers of ten, where the comparisons that the
FP64 kernels first make in FP32 leave FP32's range, against the oracle.

The scheme is scale free apart from the limiters' 1e-12, so the bar is the one of
tests/test_gpu_parity.py, relative to the largest value and flux increment of each
variable.  The smoothness indicator's alpha is compared to 1e-9: at its threshold
it changes by s / T = 1e4 times the change of an energy fraction, whose rounding is
a few 1e-16 times the number of modes, and the tiny steps taken move the state by
1e-13.
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


def _modes(prob, cells, lo, hi, seed):
    """1 + c L_N(x), the energy fraction of the top mode between lo and hi."""
    N, rng = prob["degree"], np.random.default_rng(seed)
    top = np.polynomial.legendre.Legendre.basis(N)(2.0 * wl.gl_nodes01(N)[0] - 1.0)
    frac = np.exp(rng.uniform(np.log(lo), np.log(hi), cells))
    c = np.sqrt(frac / (1.0 - frac))[:, None]
    return 1.0 + c * np.tile(top, (N + 1) ** (prob["dim"] - 1))[None, :]


def _check_alpha(prob, u, precisions=(crkfr.CR_FP64,)):
    d = oracle_desc(prob)
    dt = 1e-13 * oracle.dt(d, u)
    dg = oracle.step(d, u, dt, want_diag=True)[2]
    assert 0 < np.count_nonzero(dg["alpha_raw"])
    for precision in precisions:
        for steps in (1, 2):          # alpha from the input, then from the update
            alpha = gpu_run(prob, u, dt_fixed=dt, nsteps=steps, precision=precision)[1]
            if precision == crkfr.CR_FP64:
                np.testing.assert_allclose(alpha, dg["alpha"], rtol=0, atol=1e-9)
            elif steps == 1:
                np.testing.assert_allclose(alpha, dg["alpha"], rtol=0, atol=1e-5)


@pytest.mark.parametrize("N", [3, 4])
@pytest.mark.parametrize("rho_p", [1e-22, 1e-20, 1e-18, 1e-17, 1e-16, 1e-10, 1.0, 1e10, 1e17, 3e19, 1e20, 1e21, 1e23])
def test_indicator_of_scaled_states(N, rho_p):
    prob, u = wl.euler2d_vortex(nx=16, ny=8, degree=N, seed=N, perturb=0.0)
    prob = dict(prob, limiter=frozenset({"blend"}))
    edge = 0.5 * 10.0 ** (-1.8 * (N + 1.0) ** 0.25) * 0.25
    s = np.sqrt(rho_p)
    p = s * _modes(prob, u.shape[1], 0.3 * edge, 8.0 * edge, N)
    rho = s * np.ones_like(p)
    _check_alpha(prob, wl.euler_conservative(rho, 0.1 * np.ones_like(p), 0.0 * p, p, 1.4, 2),
                 (crkfr.CR_FP64, crkfr.CR_FP32_BULK) if 1e-10 <= rho_p <= 1e10 else (crkfr.CR_FP64,))


@pytest.mark.parametrize("dim", [1, 2])
@pytest.mark.parametrize("size", [1e-25, 1e-19, 1e-18, 1e-17, 1e-3, 1e18, 3e19, 1e20, 1e22])
def test_indicator_of_scaled_scalars(dim, size):
    prob, u = wl.linadv_random(nx=24, ny=9, dim=dim, degree=4, seed=1, adv=(0.7, -0.4))
    prob = dict(prob, limiter=frozenset({"blend"}))
    edge = 0.5 * 10.0 ** (-1.8 * 5.0 ** 0.25) * 0.25
    _check_alpha(prob, size * _modes(prob, u.shape[1], 0.3 * edge, 8.0 * edge, dim)[None])


@pytest.mark.parametrize("N", [2, 4])
@pytest.mark.parametrize("size", [1e-60, 1e-42, 1e-38, 1e-30, 1e30, 1e39, 1e60])
def test_slopes_of_scaled_scalars(N, size):
    prob, u = wl.linadv_random(nx=11, ny=7, dim=2, degree=N, seed=3, adv=(0.7, -1.2))
    prob, u = dict(prob, limiter=frozenset({"blend", "mh"})), size * u
    d = oracle_desc(prob, alpha_fixed=1.0)
    dt = 0.5 * oracle.dt(d, u)
    ref, st, dg = oracle.step(d, u, dt, want_diag=True)
    assert st == 0
    g = gpu_run(prob, u, dt_fixed=dt, alpha_fixed=1.0)[0]
    assert_parity(g, ref, extra_scale=flux_increment(prob, dg, dt))


def _random_fluid(prob, ne, npts, seed, spread=4.0):
    rng = np.random.default_rng(seed)
    draw = lambda lo, hi: np.exp(rng.uniform(np.log(lo), np.log(hi), (ne, npts)))  # noqa: E731
    rho, v1, v2 = draw(1.0 / spread, spread), rng.uniform(-1, 1, (ne, npts)), rng.uniform(-1, 1, (ne, npts))
    if prob["equation"] == "euler":
        return wl.euler_conservative(rho, v1, v2, draw(0.1, 3.0), 1.4, 2)
    a, b = draw(0.1, 3.0), draw(0.1, 3.0)
    return wl.tenmoment_conservative(rho, v1, v2, a, rng.uniform(-0.9, 0.9, a.shape) * np.sqrt(a * b), b)


@pytest.mark.parametrize("make", [wl.euler2d_vortex, wl.tenmoment2d_voronoi], ids=["euler", "tenmoment"])
@pytest.mark.parametrize("alpha", [None, 1.0])
@pytest.mark.parametrize("power", [-200, -150, -126, -120, -70, -66, -63, -50, -43, -36, 60, 83, 120, 150])
def test_scaled_fluids(make, alpha, power):
    """A state times a power of two gives the result times that power: no rounding
    changes, only what is decided in FP32 and what in FP64.  The values that enter a
    decision are formed by the same formulas at two places, which a compiler may
    contract differently; the flux limiter's theta multiplies such roundings by up to
    1e4 here (random nodes), so 1e-9 of the largest value is allowed.  A wrong decision
    moves it by percents."""
    prob, u = make(nx=11, ny=9, degree=3, seed=1)
    lim = {"mh", "flux"} | ({"blend"} if alpha else set())
    prob = dict(prob, limiter=frozenset(lim), source=None)
    u = _random_fluid(prob, u.shape[1], u.shape[2], 5)
    d = oracle_desc(prob, alpha_fixed=alpha)
    dt = 0.5 * oracle.dt(d, u)
    if oracle.step(d, u, dt)[1]:     # (a mean went negative: nothing to compare)
        dt *= 0.1
    ref = gpu_run(prob, u, dt_fixed=dt, alpha_fixed=alpha)[0]
    g = gpu_run(prob, u * 2.0 ** power, dt_fixed=dt, alpha_fixed=alpha)[0]
    assert_parity(g * 2.0 ** -power, ref, rtol=1e-9)


@pytest.mark.parametrize("speed", [1e-21, 1e21])
def test_squared_sound_speeds_beyond_the_fp32_range(speed):
    prob, u = wl.euler2d_vortex(nx=11, ny=9, degree=3, seed=1)
    prob = dict(prob, limiter=frozenset({"blend", "mh"}))
    rng, shape = np.random.default_rng(2), u.shape[1:]
    rho, p = rng.uniform(0.5, 2.0, shape), speed ** 2 * np.exp(rng.uniform(-3, 3, shape))
    u = wl.euler_conservative(rho, speed * rng.uniform(-1, 1, shape), speed * rng.uniform(-1, 1, shape), p, 1.4, 2)
    d = oracle_desc(prob, alpha_fixed=1.0)
    dt = 0.5 * oracle.dt(d, u)
    ref, st, dg = oracle.step(d, u, dt, want_diag=True)
    assert st == 0
    g = gpu_run(prob, u, dt_fixed=dt, alpha_fixed=1.0)[0]
    assert_parity(g, ref, extra_scale=flux_increment(prob, dg, dt))


@pytest.mark.parametrize("state", [(1e39, 1e60, 1e60), (1e300, 1e300, 1e40), (1e-45, 1e-30, 1e-45)])
@pytest.mark.parametrize("precision", [crkfr.CR_FP64, crkfr.CR_FP32_BULK], ids=["fp64", "fp32"])
def test_inadmissible_input_is_refused_at_every_scale(state, precision):
    """Negative pressures that FP32 cannot show."""
    rho, mom, E = state
    if precision == crkfr.CR_FP32_BULK and max(state) > 1e38:
        pytest.skip("beyond the bulk type")
    prob, u = wl.euler2d_vortex(nx=4, ny=4, degree=3, seed=1)
    u = np.ones_like(u) * np.array([rho, 0.0, 0.0, E])[:, None, None]
    u[1, 5, 3] = mom
    assert E - 0.5 * mom * mom / rho < 0
    ctx = crkfr.cr_init_mesh(crkfr.desc_from_problem(prob, precision=precision))
    with pytest.raises(crkfr.CrError):
        crkfr.cr_set_state(ctx, u)
        crkfr.cr_step(ctx, 1, 1e300, 1e-300)
