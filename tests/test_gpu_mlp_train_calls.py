"""cr_mlp_train under the conditions of a training program: long sample orders over
several epochs, also behind other work on the stream, and two threads at once.

Tolerance of the first: as in tests/test_gpu_mlp_train.py an Adam step differs by
at most 3e-3 * 1e-4 from the FP64 one; over K steps on parameters of standard
deviation 0.2 that is K * 1.5e-6 of their 2-norm, and a mixed-up order moves them by
far more.
"""
import threading

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


def test_two_threads():
    """Calls with small and large minibatches at once (they need different amounts of
    shared memory) give what each gives alone."""
    import torch
    nin, n = 25, 3000
    rng = np.random.default_rng(1)
    p = rng.normal(0.0, 0.2, mlp.param_count(nin)).astype(np.float32)
    X = torch.from_numpy(rng.uniform(0.0, 1.0, (n, nin)).astype(np.float32)).cuda()
    t = torch.from_numpy(rng.uniform(0.0, 1.0, n).astype(np.float32)).cuda()
    one = {b: torch.from_numpy(p).cuda() for b in (64, 3000)}
    for b, q in one.items():
        crkfr.cr_mlp_train(nin, q, X[:n if b > 64 else 64], t[:n if b > 64 else 64], batch=b, epochs=1, lr=3e-3, seed=3)
    errors = []

    def work(b):
        try:
            stream = torch.cuda.Stream()
            m = n if b > 64 else 64
            for _ in range(150):
                q = torch.from_numpy(p).cuda()
                torch.cuda.synchronize()
                crkfr.cr_mlp_train(nin, q, X[:m], t[:m], batch=b, epochs=1, lr=3e-3, seed=3, stream=stream.cuda_stream)
                if not torch.equal(q, one[b]):
                    raise AssertionError("different parameters at batch %d" % b)
        except Exception as e:          # noqa: BLE001
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(b,)) for b in (64, 3000, 64, 3000)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    assert not errors, errors[:3]
