"""The substitutions by blocks of 32 rows (factors without row interchanges)
against dense solves.

Sizes: less than a block, its edges, more blocks than the cluster has CTAs, a
partial last block, bands narrower than a block and as wide as the matrix.  The
matrix I - beta L has off-diagonal column sums of at most half, so its diagonal
dominates by columns, no row is interchanged and its condition number is below
10: two backward-stable float64 solves agree to
1e-12, float32 right-hand sides and results to 1e-5.
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


@pytest.mark.parametrize("N,n", [(5, 3), (31, 5), (32, 5), (33, 11), (64, 4), (65, 31), (257, 11), (289, 3), (700, 31),
                                 (1500, 11)])
def test_block_substitutions_match_dense(R, N, n):
    ns = W.fibonacci_sphere(N)
    X, Nr = (torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in (ns.X, ns.normals))
    op = R.build_operator(X, Nr, n, kernel="imq", kappa_target=1e4, allow_failures=True)
    idx, w = (t.cpu().numpy() for t in R.get_rows(op))
    L = np.zeros((N, N))
    np.add.at(L, (np.repeat(np.arange(N), n), idx.ravel()), w.ravel())
    beta = 0.5 / np.abs(L).sum(0).max()
    M = np.eye(N) - beta * L
    off = np.abs(M).sum(0) - np.abs(np.diag(M))
    assert (off < np.abs(np.diag(M))).all()
    b = W.uniform_field(N, seed=N)
    ref = np.linalg.solve(M, b)
    for dtype, bound in ((torch.float64, 1e-12), (torch.float32, 1e-5)):
        lu = R.lu_factor(op, 1.0, beta, dtype)
        x = R.lu_solve(lu, torch.as_tensor(b, dtype=dtype, device="cuda")).cpu().numpy().astype(np.float64)
        assert np.abs(x - ref).max() <= bound * np.abs(ref).max()
