"""Which samples a step of training reads.

Distinct samples in several batches, the last one smaller, over two epochs: the
order of the samples is Fisher-Yates by the 64-bit Mersenne twister of the call's
seed, restated here, and the reference takes the same batches one after the other
by float64 Adam.  Forms: an epoch per launch on clusters of eight and of four, and
the launches per step of batches too large for clusters.

The bound is a hundredth of the parameters' mean movement.  Adam moves a parameter by
about lr a step, and by its gradient's float32 error (1e-6 of the largest entry) only
where the gradient itself is as small: about 1e-5 lr in the mean, 3e-7 over the steps
here, against bounds of 3e-5.  One wrong sample in each batch moves the reference by
6e-5 and more, another order of the samples by 1e-3.
"""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_1404_0812_gb300 import workloads as W

pytestmark = pytest.mark.gpu

M64 = (1 << 64) - 1


def _mt19937_64(seed):
    x = [seed & M64]
    for i in range(1, 312):
        x.append((6364136223846793005 * (x[-1] ^ (x[-1] >> 62)) + i) & M64)
    at = 312
    while True:
        if at == 312:
            for k in range(312):
                y = (x[k] & 0xFFFFFFFF80000000) | (x[(k + 1) % 312] & 0x7FFFFFFF)
                x[k] = x[(k + 156) % 312] ^ (y >> 1) ^ (0xB5026F5AA96619E9 if y & 1 else 0)
            at = 0
        z = x[at]
        at += 1
        z ^= (z >> 29) & 0x5555555555555555
        z ^= (z << 17) & 0x71D67FFFEDA60000
        z ^= (z << 37) & 0xFFF7EEE000000000
        yield z ^ (z >> 43)


def _batches(count, batch, epochs, seed):
    rng, perm = _mt19937_64(seed), list(range(count))
    for _ in range(epochs):
        for i in range(count - 1, 0, -1):
            j = next(rng) % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        yield [np.array(perm[b:b + batch]) for b in range(0, count, batch)]


def _adam(p0, X, y, D, epochs, lr):
    p, m, v, t, losses = p0.copy(), np.zeros_like(p0), np.zeros_like(p0), 0, []
    for batches in epochs:
        total = 0.0
        for sel in batches:
            loss, g = omlp.loss_and_grads(W.mlp_unpack(p, D), X[sel], y[sel])
            g, t, total = W.mlp_pack(g), t + 1, total + loss * len(sel)
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - lr * (m / (1 - 0.9**t)) / (np.sqrt(v / (1 - 0.999**t)) + 1e-8)
        losses.append(total / len(X))
    return p, np.array(losses)


@pytest.mark.parametrize("n,count,batch", [(11, 1000, 256), (31, 300, 65), (11, 5000, 2000), (11, 6000, 2433)])
def test_steps_read_the_samples_of_their_batch(n, count, batch):
    import paper_1404_0812_gb300 as R
    D, lr, seed = 3 * n, 1e-3, 7
    rng = np.random.default_rng(n + count)
    start = W.mlp_pack(W.mlp_init(D, seed=n)).astype(np.float32)
    X = rng.uniform(-1.0, 1.0, (count, D)).astype(np.float32)
    y = np.sin(3.0 * X[:, 0] + np.arange(count) % 17).astype(np.float32)
    net = R.EpsNet(n, start)
    losses = net.train(torch.as_tensor(X, device="cuda"), torch.as_tensor(y, device="cuda"), epochs=2, batch=batch, lr=lr,
                       seed=seed)
    p0, X64, y64 = start.astype(np.float64), X.astype(np.float64), y.astype(np.float64)
    p, want = _adam(p0, X64, y64, D, _batches(count, batch, 2, seed), lr)
    other, _ = _adam(p0, X64, y64, D, _batches(count, batch, 2, seed + 1), lr)
    bound = 0.01 * np.abs(p - p0).mean()
    assert np.abs(other - p).mean() > 10 * bound
    assert np.abs(net.params() - p).mean() < bound
    assert np.abs(np.asarray(losses) - want).max() <= 1e-4 * want.max()
