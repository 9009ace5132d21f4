"""Epochs of mini-batch steps in one launch against the same steps one call at
a time.

The samples of a set are all alike, so their order does not matter, and the
steps of an epoch have to leave the same bits as single-step calls on batches of
the same sizes: the weights of a step have to be complete before the next one
reads them, the moments and the step count have to carry over, and a smaller
last batch leaves clusters idle.  Sizes: one tile and part of one, clusters of
eight and of four and their edges, batches of too many tiles for clusters, the
smallest and the largest network.
"""
import numpy as np
import pytest
import torch

from paper_1404_0812_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_1404_0812_gb300 as R
    return R


@pytest.mark.parametrize("n,count,batch,epochs", [(2, 7, 1, 1), (11, 200, 65, 2), (31, 3000, 1000, 2),
                                                  (50, 2 * 1216, 1216, 1), (50, 3 * 1217 + 5, 1217, 1),
                                                  (101, 5000, 2432, 1), (128, 300, 64, 2), (31, 6000, 2433, 1)])
def test_an_epoch_leaves_the_bits_of_its_steps(R, n, count, batch, epochs):
    rng = np.random.default_rng(n)
    p = W.mlp_pack(W.mlp_init(3 * n, seed=n)).astype(np.float32)
    x = torch.as_tensor(rng.uniform(-1.0, 1.0, 3 * n).astype(np.float32), device="cuda")
    X = x.repeat(count, 1).contiguous()
    y = torch.full((count,), 0.7, device="cuda")
    whole, steps = R.EpsNet(n, p), R.EpsNet(n, p)
    losses = whole.train(X, y, epochs=epochs, batch=batch, lr=1e-3, seed=1)
    for ep in range(epochs):
        total = 0.0
        for b in range(0, count, batch):
            nb = min(batch, count - b)
            total += nb * steps.train(X[:nb], y[:nb], epochs=1, batch=batch, lr=1e-3, seed=1)[0]
        assert abs(losses[ep] - total / count) <= 1e-6 * abs(losses[ep])   # float32 losses, averaged in float64
    assert np.array_equal(whole.params(), steps.params())
    assert not np.array_equal(whole.params(), p)
