"""The back substitution's quotients by the diagonal.

With beta = 0 the matrix is alpha I and its solution b / alpha: the quotients
themselves, which have to be correctly rounded (the float64 form errs by half an
ulp and 2^-105, so an unequal one among these is out of reach), for divisors
throughout float64's range, the subnormal ones included, and in float32.  A whole
float32 matrix of subnormal entries: 2^-129 (I - beta L) with the dominant
diagonal of the block tests.  Its entries and every operation round to 2^-149,
2^-21 of the diagonal, so with a condition number below 10 and bands of at most 64
the results agree to 10 x 2 x 64 x 2^-21 < 1e-3.
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


def _operator(R, N, n):
    ns = W.fibonacci_sphere(N)
    X, Nr = (torch.as_tensor(np.ascontiguousarray(a), device="cuda") for a in (ns.X, ns.normals))
    return R.build_operator(X, Nr, n, kernel="imq", kappa_target=1e4, allow_failures=True)


@pytest.mark.parametrize("N,n", [(5, 3), (33, 5), (300, 11)])
@pytest.mark.parametrize("alpha", [3.0, 0.1, 1.7e250, 1e-260, 1e-300, 1e290, 5e-310])
def test_quotients_are_correctly_rounded(R, N, n, alpha):
    op = _operator(R, N, n)
    b = alpha * (1.0 + W.uniform_field(N, seed=N))
    lu = R.lu_factor(op, alpha, 0.0)
    x = R.lu_solve(lu, torch.as_tensor(b, device="cuda")).cpu().numpy()
    assert np.array_equal(x, b / alpha)


@pytest.mark.parametrize("alpha", [3.0, 0.1, 2.0**100, 2.0**-120, 2.0**-130])
def test_float32_quotients_are_correctly_rounded(R, alpha):
    op = _operator(R, 300, 11)
    a = np.float32(alpha)
    b = (a * (1.0 + W.uniform_field(300, seed=2))).astype(np.float32)
    lu = R.lu_factor(op, float(a), 0.0, torch.float32)
    x = R.lu_solve(lu, torch.as_tensor(b, device="cuda")).cpu().numpy()
    assert np.array_equal(x, b / a)


@pytest.mark.parametrize("N,n", [(33, 5), (65, 5)])
def test_subnormal_float32_factors(R, N, n):
    op = _operator(R, N, n)
    idx, w = (t.cpu().numpy() for t in R.get_rows(op))
    L = np.zeros((N, N))
    np.add.at(L, (np.repeat(np.arange(N), n), idx.ravel()), w.ravel())
    beta = 0.5 / np.abs(L).sum(0).max()
    scale = 2.0**-129
    b = W.uniform_field(N, seed=N).astype(np.float32)
    ref = np.linalg.solve(np.eye(N) - beta * L, b.astype(np.float64))
    lu = R.lu_factor(op, scale, beta * scale, torch.float32)
    x = R.lu_solve(lu, torch.as_tensor(np.ldexp(b, -129), device="cuda")).cpu().numpy().astype(np.float64)
    assert np.abs(x - ref).max() <= 1e-3 * np.abs(ref).max()


@pytest.mark.parametrize("dtype,e", [(torch.float64, -1030), (torch.float32, -132)])
def test_coefficients_below_the_normal_range(R, dtype, e):
    """Coefficients whose quotients by the diagonal are subnormal: 1.5 I - 2^e L (L
    scaled to at most one).  Their products are far below an ulp of right-hand sides
    between one and two, so the solution is b / 1.5, correctly rounded."""
    N, n = 65, 5
    op = _operator(R, N, n)
    w = R.get_rows(op)[1]
    np_t = np.float64 if dtype == torch.float64 else np.float32
    b = (1.0 + W.uniform_field(N, seed=N) % 1.0).astype(np_t)
    lu = R.lu_factor(op, 1.5, 2.0**e / float(w.abs().max()), dtype)
    x = R.lu_solve(lu, torch.as_tensor(b, device="cuda")).cpu().numpy()
    assert np.array_equal(x, b / np_t(1.5))
