"""Lines of nodes of very different size in one element: the fixed-point sums of the
FP64 element kernel share an exponent per element and variable, and elements in which
that would cost a line bits take their stages in FP64.

Advection along x (y) alone: the rows (columns) of nodes of an element do not act on
one another, so each is held to the 1e-12 of tests/test_gpu_parity.py relative to its
own largest value, whatever lies beside it.  Elsewhere the bar is that of
tests/test_gpu_parity.py.
"""
import numpy as np
import pytest

import oracle
from paper_2502_07517_gb300 import crkfr
from paper_2502_07517_gb300 import workloads as wl
from tests._oracle_util import oracle_desc
from tests.test_gpu_parity import assert_parity, flux_increment, gpu_run

pytestmark = pytest.mark.gpu

DISS = {"D2": (crkfr.CR_DISS_D2, oracle.DISS_D2), "D1": (crkfr.CR_DISS_D1, oracle.DISS_D1),
        "DCSX": (crkfr.CR_DISS_DCSX, oracle.DISS_DCSX)}
CENTRAL = {"EA": (crkfr.CR_CENTRAL_EA, oracle.CENTRAL_EA), "AE": (crkfr.CR_CENTRAL_AE, oracle.CENTRAL_AE)}


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_07517_gb300 import build
    build.build()


@pytest.mark.parametrize("N", [1, 2, 3, 4])
@pytest.mark.parametrize("along", ["x", "y"])
@pytest.mark.parametrize("decades", [0.0, 3.0, 25.0])
@pytest.mark.parametrize("diss,central", [("D2", "EA"), ("D1", "EA"), ("DCSX", "EA"), ("D2", "AE")])
def test_rows_keep_their_own_accuracy(N, along, decades, diss, central):
    nx, ny, n = (13, 6, N + 1) if along == "x" else (6, 13, N + 1)
    prob, u = wl.linadv_random(nx=nx, ny=ny, dim=2, degree=N, seed=N, adv=(1.0, 0.0) if along == "x" else (0.0, 1.0))
    rng = np.random.default_rng(N)
    lines = 10.0 ** -rng.uniform(0.0, decades, (6, n)) * np.where(rng.random((6, n)) < 0.2, 0.0, 1.0)   # some are 0
    u = u.reshape(ny, nx, n, n)
    scale = (lines[:, None, :, None] if along == "x" else lines[None, :, None, :]) * np.ones_like(u)
    u = (u * scale).reshape(1, nx * ny, n * n)
    d = oracle_desc(prob, dissipation=DISS[diss][1], central=CENTRAL[central][1])
    dt = oracle.dt(d, u + 1.0)
    ref, st = oracle.step(d, u, dt)[:2]
    assert st == 0
    g = gpu_run(prob, u, dt_fixed=dt, dissipation=DISS[diss][0], central=CENTRAL[central][0])[0]
    scale = scale.reshape(u[0].shape)
    assert (g[0][scale == 0] == 0).all()
    err = np.abs(g - ref)[0][scale > 0] / scale[scale > 0]
    assert err.max() <= 1e-12 * 4.0, err.max()          # (values up to 4 scale)


def _crossing(prob, u, seed):
    """Velocities that pass through 0 inside the elements, and rows at rest."""
    rng = np.random.default_rng(seed)
    x, y = wl.node_coords(prob)
    lx, ly = prob["x1"] - prob["x0"], prob["y1"] - prob["y0"]
    rho = 1.0 + 0.2 * np.sin(2 * np.pi * (x / lx + y / ly))
    v1, v2 = np.sin(4 * np.pi * y / ly + 0.3), 1e-3 * np.cos(6 * np.pi * x / lx)
    v1[rng.random(v1.shape[0]) < 0.2] = 0.0
    if prob["equation"] == "euler":
        return wl.euler_conservative(rho, v1, v2, 1.0 + 0.1 * rho, prob["gamma"], 2)
    return wl.tenmoment_conservative(rho, v1, v2, 1.0 + 0.1 * rho, 1e-4 * v1, 1.2 - 0.1 * rho)


@pytest.mark.parametrize("N", [1, 2, 3, 4])
@pytest.mark.parametrize("flow", ["vortex", "box", "taylor", "tenmoment"])
@pytest.mark.parametrize("diss,central", [("D2", "EA"), ("D1", "EA"), ("DCSX", "EA"), ("D2", "AE")])
def test_velocities_through_zero(N, flow, diss, central):
    if flow == "taylor" and diss == "D1":
        pytest.skip("the HLLC sides take time averages: refused with D1")
    make = {"vortex": wl.euler2d_vortex, "box": wl.euler2d_vortex, "taylor": wl.rayleigh_taylor,
            "tenmoment": wl.tenmoment2d_voronoi}[flow]
    prob, u = make(nx=13, ny=11, degree=N)
    if flow == "box":
        prob = dict(prob, bc_x="wall", bc_y="outflow")
    u = _crossing(prob, u, N)
    d = oracle_desc(prob, dissipation=DISS[diss][1], central=CENTRAL[central][1])
    dt = oracle.dt(d, u)
    ref, st, dg = oracle.step(d, u, dt, want_diag=True)
    assert st == 0
    g, alpha = gpu_run(prob, u, dt_fixed=dt, dissipation=DISS[diss][0], central=CENTRAL[central][0])[:2]
    assert_parity(g, ref, extra_scale=flux_increment(prob, dg, dt))
    np.testing.assert_allclose(alpha, dg["alpha"], rtol=0, atol=1e-12)


@pytest.mark.parametrize("threads", [128, 256])
@pytest.mark.parametrize("mode", [crkfr.CR_BATCH_PHASES, crkfr.CR_BATCH_FUSED])
def test_batches_take_the_same_elements(threads, mode):
    """An element's result does not depend on those that share its block."""
    ref, ctxs, shapes = [], [], []
    for i, (nx, ny, N) in enumerate([(13, 11, 3), (9, 17, 4), (24, 7, 4), (6, 5, 3)]):
        prob, u = wl.euler2d_vortex(nx=nx, ny=ny, degree=N)
        u = _crossing(prob, u, i)
        ref.append(gpu_run(prob, u, nsteps=3)[0])
        ctx = crkfr.cr_init_mesh(crkfr.desc_from_problem(prob))
        crkfr.cr_set_state(ctx, u)
        ctxs.append(ctx)
        shapes.append(u.shape)
    b = crkfr.cr_batch_init(ctxs)
    crkfr.cr_batch_config(b, threads, mode)
    crkfr.cr_batch_step(b, 3)
    for ctx, shape, r in zip(ctxs, shapes, ref):
        np.testing.assert_array_equal(crkfr.cr_get_state(ctx, shape=shape), r)
