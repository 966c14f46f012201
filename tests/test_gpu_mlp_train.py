"""Training of the network: a few Adam steps against the FP64 backward pass of
oracle/mlp.py with the same seeded sample order, at the edges of the epoch
kernel's range (chunks of 64 samples, clusters of 1 to 8 blocks, several chunks
per block, a ragged last minibatch, one sample) and past it (minibatches of more
than 48 chunks take one launch per step).

Tolerance: an Adam step moves a parameter by at most about lr = 3e-3, and FP32
changes that by its relative error in m / sqrt(v), below 1e-4 on the whole; six
steps on parameters of standard deviation 0.2 so stay within 6 * 3e-3 * 1e-4 / 0.2
< 1e-5 of their 2-norm, and twice that is allowed.
"""
import numpy as np
import pytest

from oracle import mlp
from paper_2502_07517_gb300 import crkfr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2502_07517_gb300 import build
    build.build()


def _orders(n, epochs, seed):
    s, mask, out = seed, (1 << 64) - 1, []
    for _ in range(epochs):
        perm = np.arange(n)
        for i in range(n - 1, 0, -1):
            s = (s + 0x9e3779b97f4a7c15) & mask
            z = ((s ^ (s >> 30)) * 0xbf58476d1ce4e5b9) & mask
            z = ((z ^ (z >> 27)) * 0x94d049bb133111eb) & mask
            j = (z ^ (z >> 31)) % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        out.append(perm)
    return out


@pytest.mark.parametrize("nin,n,batch,epochs", [
    (16, 1, 1, 3), (2, 63, 64, 3), (3, 64, 64, 3), (4, 129, 65, 2), (5, 256, 256, 3), (9, 700, 513, 2), (16, 1000, 512, 2),
    (25, 1200, 10 ** 9, 3), (16, 3072, 3072, 2), (25, 3100, 3000, 2), (16, 3200, 3200, 2), (5, 2 ** 12, 2 ** 31 - 1, 1)])
def test_adam_steps_match_fp64(nin, n, batch, epochs):
    import torch
    rng = np.random.default_rng(nin + n)
    p = rng.normal(0.0, 0.2, mlp.param_count(nin)).astype(np.float32)
    X = rng.uniform(0.0, 1.0, (n, nin)).astype(np.float32)
    t = rng.uniform(0.0, 1.0, n).astype(np.float32)
    dev = lambda a: torch.from_numpy(a).cuda()
    got, again = dev(p), dev(p)
    loss = crkfr.cr_mlp_train(nin, got, dev(X), dev(t), batch=batch, epochs=epochs, lr=3e-3, seed=n)
    loss2 = crkfr.cr_mlp_train(nin, again, dev(X), dev(t), batch=batch, epochs=epochs, lr=3e-3, seed=n)
    assert torch.equal(got, again) and loss == loss2       # the same bits on every run
    q, m, v, k = p.astype(np.float64), 0.0, 0.0, 0
    for perm in _orders(n, epochs, n):
        losses = []
        for b in range(0, n, batch):
            i = perm[b:b + batch]
            losses.append(mlp.loss(q, X[i], t[i]))
            g = mlp.grad(q, X[i].astype(np.float64), t[i])
            k += 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            q = q - 3e-3 * (m / (1.0 - 0.9 ** k)) / (np.sqrt(v / (1.0 - 0.999 ** k)) + 1e-8)
    off = np.linalg.norm(got.cpu().numpy().astype(np.float64) - q) / np.linalg.norm(q)
    assert off <= 2e-5, off
    assert abs(loss - np.mean(losses)) <= 1e-5 * np.mean(losses)
