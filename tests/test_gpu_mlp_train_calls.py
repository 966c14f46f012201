"""cr_mlp_train under the conditions of a training program: long sample orders over
several epochs, also behind other work on the stream.

Tolerance: as in tests/test_gpu_mlp_train.py an Adam step differs by
at most 3e-3 * 1e-4 from the FP64 one; over K steps on parameters of standard
deviation 0.2 that is K * 1.5e-6 of their 2-norm, and a mixed-up order moves them by
far more.
"""
import numpy as np
import pytest

from oracle import mlp
from paper_2502_07517_gb300 import crkfr
from tests.test_gpu_mlp_train import _orders

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_07517_gb300 import build
    build.build()


@pytest.mark.parametrize("behind", [False, True])
def test_orders_of_several_epochs(behind):
    """The host draws the next epoch's order while the device still has earlier
    copies to take (behind: other work of the stream holds them all back)."""
    import torch
    nin, n, batch, epochs, seed = 16, 50000, 1024, 5, 9
    rng = np.random.default_rng(seed)
    p = rng.normal(0.0, 0.2, mlp.param_count(nin)).astype(np.float32)
    X = rng.uniform(0.0, 1.0, (n, nin)).astype(np.float32)
    t = rng.uniform(0.0, 1.0, n).astype(np.float32)
    got, Xd, td = (torch.from_numpy(a).cuda() for a in (p, X, t))
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        if behind:
            torch.cuda._sleep(1_500_000_000)          # most of a second
        loss = crkfr.cr_mlp_train(nin, got, Xd, td, batch=batch, epochs=epochs, lr=3e-3, seed=seed,
                                  stream=stream.cuda_stream)
    torch.cuda.synchronize()
    q, m, v, k = p.astype(np.float64), 0.0, 0.0, 0
    for perm in _orders(n, epochs, seed):
        losses = []
        for b in range(0, n, batch):
            i = perm[b:b + batch]
            losses.append(mlp.loss(q, X[i], t[i]))
            g = mlp.grad(q, X[i].astype(np.float64), t[i])
            k += 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            q = q - 3e-3 * (m / (1.0 - 0.9 ** k)) / (np.sqrt(v / (1.0 - 0.999 ** k)) + 1e-8)
    off = np.linalg.norm(got.cpu().numpy().astype(np.float64) - q) / np.linalg.norm(q)
    assert off <= 1.5e-6 * k, off
    assert abs(loss - np.mean(losses)) <= 1e-5 * np.mean(losses)
