"""The gradient of mini-batches on clusters of CTAs against the same gradient
tile by tile: every element is summed over a tile's samples, and over tiles, in
the same order, so a batch split at tile boundaries gives the same sums.

A batch of 38 tiles and more runs a CTA per tile, 20 to 38 tiles clusters of
four, fewer clusters of eight: the sizes below are their edges, with partial
last tiles, the smallest and largest networks, and a stencil size whose
features do not divide among the cluster.
"""
import numpy as np
import pytest
import torch

from oracle import mlp as omlp
from paper_1404_0812_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_1404_0812_gb300 as R
    return R


@pytest.mark.parametrize("n,count", [(2, 1), (2, 65), (11, 64), (31, 1000), (50, 1216), (50, 1217), (101, 2432),
                                     (128, 2433), (50, 4000)])
def test_gradient_matches_float64_at_the_edges_of_each_form(R, n, count):
    rng = np.random.default_rng(n + count)
    p = W.mlp_init(3 * n, seed=n)
    p["b1"], p["b2"] = 0.1 * rng.standard_normal(64), 0.1 * rng.standard_normal(64)
    net = R.EpsNet(n, W.mlp_pack(p).astype(np.float32))
    p32 = W.mlp_unpack(net.params(), 3 * n)
    X = rng.uniform(-1.0, 1.0, (count, 3 * n)).astype(np.float32)
    y = rng.uniform(-1.0, 1.0, count).astype(np.float32)
    g, loss = net.loss_grad(torch.as_tensor(X, device="cuda"), torch.as_tensor(y, device="cuda"))
    ref_loss, ref = omlp.loss_and_grads(p32, X.astype(np.float64), y.astype(np.float64))
    ref = W.mlp_pack(ref)
    assert abs(loss - ref_loss) <= 1e-5 * ref_loss
    assert np.abs(g.cpu().numpy() - ref).max() <= 1e-4 * np.abs(ref).max()   # float32 sums of up to `count` terms


def test_clusters_of_four_and_eight_and_single_ctas_agree_bit_for_bit(R):
    """The sum over all samples of a zero-padded batch: samples with zero
    residual and features add exact zeros, so 64 real samples followed by
    padding give the same gradient times the ratio of the counts, whichever
    form a batch of that size takes (powers of two keep the scaling exact)."""
    n = 31
    rng = np.random.default_rng(5)
    net = R.EpsNet(n, W.mlp_pack(W.mlp_init(3 * n, seed=2)).astype(np.float32))
    zero = net.predict(torch.zeros(1, 3 * n, device="cuda"))
    got = []
    for count in (64, 1024, 2048, 4096):   # 1, 16 (clusters of 8), 32 (of 4), 64 tiles (single CTAs)
        rng = np.random.default_rng(5)
        X = torch.zeros(count, 3 * n, device="cuda")
        X[:64] = torch.as_tensor(rng.uniform(-1, 1, (64, 3 * n)).astype(np.float32), device="cuda")
        y = zero.repeat(count).contiguous()
        y[:64] = torch.as_tensor(rng.uniform(-1, 1, 64).astype(np.float32), device="cuda")
        g, _ = net.loss_grad(X, y)
        got.append(g * count)
    for g in got[1:]:
        assert torch.equal(g, got[0])
