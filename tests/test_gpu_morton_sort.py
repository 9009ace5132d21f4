"""The Morton order's device sort at its edges: one tile of 4096 nodes and
less, partial and several tiles, equal keys (ties by index), nodes on a line
and in one point, against a numpy restatement of the order."""
import numpy as np
import pytest
import torch

from paper_1404_0812_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_1404_0812_gb300 as R
    return R


def _reference(X):
    lo = X.min(axis=0)
    ext = (X.max(axis=0) - lo).max()
    scale = 2097151.0 / ext if ext > 0 else 0.0
    q = np.clip(np.floor((X - lo) * scale), 0, 2097151).astype(np.uint64)
    key = np.zeros(len(X), dtype=np.uint64)
    for b in range(21):
        for a in range(3):
            key |= ((q[:, a] >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b + a)
    return np.argsort(key, kind="stable").astype(np.int32)


def _order(R, X):
    return R.morton_order(torch.as_tensor(np.ascontiguousarray(X), device="cuda")).cpu().numpy()


@pytest.mark.parametrize("N", [1, 2, 31, 257, 4095, 4096, 4097, 8192, 12_289, 300_001, 2_000_000])
def test_morton_sort_sizes(R, N):
    rng = np.random.default_rng(N)
    X = W.bumpy_sphere(N).X[rng.permutation(N)]
    assert np.array_equal(_order(R, X), _reference(X))


@pytest.mark.parametrize("N", [1000, 70_000])
def test_morton_sort_ties_and_degenerate_sets(R, N):
    rng = np.random.default_rng(N)
    lattice = rng.integers(0, 5, size=(N, 3)).astype(np.float64)           # many equal keys
    line = np.zeros((N, 3))
    line[:, 1] = rng.uniform(-3.0, 5.0, N)
    for X in (lattice, line, np.full((N, 3), 0.25)):
        assert np.array_equal(_order(R, X), _reference(X))
