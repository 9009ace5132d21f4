"""The Morton order refuses nodes that are not finite, wherever the one
coordinate is and whatever the others are; the largest finite ones it takes."""
import numpy as np
import pytest
import torch

from paper_1404_0812_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_1404_0812_gb300 as R
    return R


@pytest.mark.parametrize("N", [1, 257, 5000, 300_001])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_one_coordinate_that_is_not_finite(R, N, value):
    X = W.fibonacci_sphere(N).X.copy() if N > 1 else np.zeros((1, 3))
    for i, a in ((0, 0), (N // 2, 1), (N - 1, 2)):
        Y = torch.as_tensor(X, device="cuda")
        Y[i, a] = value
        with pytest.raises(R.RbffdError) as e:
            R.morton_order(Y)
        assert e.value.status == 1


def test_large_finite_coordinates(R):
    X = W.fibonacci_sphere(5000).X * 1e300
    perm = R.morton_order(torch.as_tensor(X, device="cuda")).cpu().numpy()
    want = R.morton_order(torch.as_tensor(X * 1e-300, device="cuda")).cpu().numpy()
    assert np.array_equal(np.sort(perm), np.arange(5000)) and (perm == want).mean() > 0.99
