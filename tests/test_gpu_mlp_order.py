"""Gradients of samples that the kernel just ahead on the stream makes.

The gradient of one call is the features of the next, with nothing in between:
the second call has to read what the first one's last kernel (which lets its
dependents start early) wrote, so it gives the bits of a call on a finished copy.
Batches of one and of several tiles on clusters of eight and of four, and one too
large for clusters.
"""
import numpy as np
import pytest
import torch

from paper_1404_0812_gb300 import _lib
from paper_1404_0812_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_small", [(31, 31), (101, 11), (50, 2), (128, 2)])
def test_features_written_by_the_kernel_ahead(n, n_small):
    import paper_1404_0812_gb300 as R
    lib = _lib.load()
    rng = np.random.default_rng(n)
    first = R.EpsNet(n, W.mlp_pack(W.mlp_init(3 * n, seed=n)).astype(np.float32))
    second = R.EpsNet(n_small, W.mlp_pack(W.mlp_init(3 * n_small, seed=1)).astype(np.float32))
    X = torch.as_tensor(rng.uniform(-1.0, 1.0, (65, 3 * n)).astype(np.float32), device="cuda")
    count = first.P // (3 * n_small)
    y = torch.as_tensor(rng.uniform(-1.0, 1.0, count).astype(np.float32), device="cuda")
    stream = torch.cuda.current_stream().cuda_stream

    def grad(net, feats, target, rows, out):
        status = lib.rbffd_mlp_loss_grad(net.handle, feats.data_ptr(), target.data_ptr(), rows, out.data_ptr(), None,
                                         stream)
        assert status == 0

    for k in range(10):
        g1 = torch.zeros(first.P, device="cuda")
        got = torch.empty(second.P, device="cuda")
        want = torch.empty(second.P, device="cuda")
        t = torch.as_tensor(rng.uniform(-1.0, 1.0, 65).astype(np.float32), device="cuda")
        torch.cuda.synchronize()
        grad(first, X, t, 65, g1)
        grad(second, g1, y, count, got)
        torch.cuda.synchronize()
        grad(second, g1.clone(), y, count, want)
        torch.cuda.synchronize()
        assert float(g1.abs().max()) > 0.0
        assert torch.equal(got, want), k
