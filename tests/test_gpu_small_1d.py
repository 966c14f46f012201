"""One-dimensional FP64 meshes about the size at which the step kernels change from
64-thread to 256-thread blocks (all 64-thread blocks resident at once: 8 per SM, 152
SMs): one element less, that many, one more, against the oracle with the bar of
tests/test_gpu_parity.py.
"""
import pytest

from paper_2502_07517_gb300 import workloads as wl
from tests.test_gpu_parity import one_step_check

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_07517_gb300 import build
    build.build()


@pytest.mark.parametrize("N", [1, 2, 3, 4])
@pytest.mark.parametrize("more", [-1, 0, 1])
@pytest.mark.parametrize("flow", ["riemann", "advection"])
def test_meshes_about_the_small_blocks(N, more, flow):
    nx = 152 * 8 * (64 // (N + 1)) + more
    prob, u = (wl.euler1d_riemann(nx=nx, degree=N, seed=N) if flow == "riemann" else
               wl.linadv_random(nx=nx, degree=N, seed=N, adv=(1.0, 0.0), bc="periodic"))
    one_step_check(prob, u)
