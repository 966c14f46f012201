"""The split of an FP64 state into FP64 means and FP32 fluctuations at the edges of
its rounding: fluctuations in FP32's normal range, across its lower end and below it,
exact zeros, and row counts around the kernel's 128 rows per block.

Tolerance per value: the fluctuation x - mean is rounded to FP32 once (2^-24 of it, or
2^-150 below FP32's normal range), on top of a few FP64 roundings of the row's largest
value in the mean, the difference and the sum (Np + 4 of 2^-53).
"""
import numpy as np
import pytest

from paper_2502_07517_gb300 import crkfr
from paper_2502_07517_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_07517_gb300 import build
    build.build()


@pytest.mark.parametrize("N", [3, 4])
@pytest.mark.parametrize("nx,ny", [(2, 2), (8, 4), (3, 11), (16, 8)])
@pytest.mark.parametrize("size", [1.0, 1e-30, 2.0 ** -126, 1e-41, 0.0])
def test_state_survives_the_split(N, nx, ny, size):
    rng = np.random.default_rng(N)
    prob, u = wl.euler2d_vortex(nx=nx, ny=ny, degree=N, seed=N)
    u = np.array(u)
    u[1:3] = size * rng.uniform(-1, 1, u[1:3].shape)     # momenta; the energy keeps the pressure positive
    u[3] = 2.0 + np.abs(u[3])
    ctx = crkfr.cr_init_mesh(crkfr.desc_from_problem(prob, precision=crkfr.CR_FP32_BULK))
    crkfr.cr_set_state(ctx, u)
    got = crkfr.cr_get_state(ctx, shape=u.shape)
    big = np.abs(u).max(axis=2, keepdims=True)
    bound = 2.0 ** -24 * 2 * big + 2.0 ** -150 + (u.shape[2] + 4) * 2.0 ** -53 * big
    assert (np.abs(got - u) <= bound).all()
