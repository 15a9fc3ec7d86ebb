"""Training over batches of different samples: the documented seeded order
(splitmix64, Fisher-Yates) and Adam in 64 bits."""
import math

import numpy as np
import pytest

from gpu_common import make_pair
from oracle import mlp as M
from paper_2211_12867_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _orders(n, epochs, seed):
    mask = 2 ** 64 - 1
    state = seed & mask
    for _ in range(epochs):
        perm = list(range(n))
        for i in range(n - 1, 0, -1):
            state = (state + 0x9E3779B97F4A7C15) & mask
            z = ((state ^ (state >> 30)) * 0xBF58476D1CE4E5B9) & mask
            z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & mask
            j = (z ^ (z >> 31)) % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        yield np.array(perm)


# a last batch of one, ragged and even ones, one batch an epoch
@pytest.mark.parametrize("n,batch", [(33, 8), (1000, 96), (512, 128), (70, 100)])
def test_batches_of_different_samples(n, batch):
    """FP32 gradients are within some 1e-6 of the 64-bit ones, and Adam's step
    is lr times a ratio of gradients: apart from parameters whose gradient is
    rounding noise (1e-5 of them, off by 2 lr a step at most) a step is within
    1e-5 lr.  Another order of the samples moves the parameters by a good part
    of lr: 0.01 lr a step on average tells them apart."""
    g, _ = make_pair(n=(24, 12, 12), nb=(12, 12, 12), x_min=(0.1, math.pi / 6, 0.0),
                     x_max=(2.0, 5 * math.pi / 6, 2 * math.pi), stretch=True)
    rng = np.random.default_rng(n)
    X = rng.uniform(0, 1.0, (n, 64)).astype(np.float32)
    T = (rng.random(n) < 0.4).astype(np.float32)
    theta = I.mlp_init(3).astype(np.float32)
    epochs, lr, seed = 2, float(np.float32(1e-3)), 17
    g.mlp_set_params(theta)
    g.mlp_dataset_clear()
    g.mlp_dataset_add(X, T)
    g.mlp_train(n, epochs, batch=batch, lr=lr, seed=seed)
    th = theta.astype(np.float64)
    m, v, step = np.zeros_like(th), np.zeros_like(th), 0
    for perm in _orders(n, epochs, seed):
        for at in range(0, n, batch):
            rows = perm[at:at + batch]
            gr = M.grad(th, X[rows].astype(np.float64), T[rows].astype(np.float64))
            step += 1
            m, v = 0.9 * m + 0.1 * gr, 0.999 * v + 0.001 * gr * gr
            th = th - lr * (m / (1 - 0.9 ** step)) / (np.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
    assert np.abs(g.mlp_get_params() - th).mean() < 0.01 * lr * step
    assert np.abs(th - theta).mean() > 0.1 * lr * step
