"""The build's team kernels (several lanes per stencil) against the
lane-per-stencil kernels: the same floating-point operations in the same
order, so every result is equal bit for bit.

An explicit launch shape keeps a build on the lane-per-stencil kernel; without
one the kernel follows from the number of rows and the stencil size.  The sizes
below reach every number of lanes per team (32, 16, 8 and 4), stencil sizes
with and without padding, the smallest and the largest, more rows than the
chip holds teams at once, and warps whose last teams have no stencil.
"""
import numpy as np
import pytest
import torch

from paper_1404_0812_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LANE = dict(block_threads=128, blocks_per_sm=4)


@pytest.fixture(scope="module")
def R():
    import paper_1404_0812_gb300 as R
    return R


def _cuda(a, dt=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


def _results(R, op):
    ell = R.get_ell(op)
    info = R.get_stencil_info(op)
    return dict(idx=ell["idx"], w64=ell["w64"], w32=ell["w32"], **info)


def _assert_equal(R, a, b):
    x, y = _results(R, a), _results(R, b)
    for k in x:
        u, v = x[k], y[k]
        if u.dtype.is_floating_point:   # NaN (no kappa at given eps) compares by its bits
            it = torch.int64 if u.dtype == torch.float64 else torch.int32
            u, v = u.view(it), v.view(it)
        assert torch.equal(u, v), (k, int((u != v).sum()))


@pytest.mark.parametrize("kernel", ["imq", "gaussian"])
@pytest.mark.parametrize("N,n,kappa", [
    (5, 2, 1e3), (9, 9, 1e6), (130, 128, 1e12), (300, 31, 1e12),   # 32 lanes
    (901, 17, 1e8), (2003, 50, 1e12), (950, 101, 1e12),            # 16
    (3601, 32, 1e12), (4999, 33, 1e10), (12001, 84, 1e12),         # 8
    (8009, 11, 1e8), (15013, 50, 1e12)])                           # 4
def test_search_on_teams_equals_lanes(R, N, n, kappa, kernel):
    ns = W.fibonacci_sphere(N)
    X, Nr = _cuda(ns.X), _cuda(ns.normals)
    args = dict(kernel=kernel, kappa_target=kappa, allow_failures=True)
    _assert_equal(R, R.build_operator(X, Nr, n, **args), R.build_operator(X, Nr, n, **args, **LANE))


def test_search_options_and_mixed_sizes_on_teams_equal_lanes(R):
    """A search range that leaves roots outside, few evaluations, a loose
    tolerance, kappa_T beyond float64 (failing factorisations), and operators
    of mixed sizes."""
    ns = W.bumpy_sphere(3001)
    X, Nr = _cuda(ns.X), _cuda(ns.normals)
    for args in (dict(kappa_target=1e12, eps_range=(0.3, 0.45)), dict(kappa_target=1e12, max_evals=3),
                 dict(kappa_target=1e9, eps_tol=1e-2), dict(kappa_target=1e17)):
        _assert_equal(R, R.build_operator(X, Nr, 31, **args, allow_failures=True),
                      R.build_operator(X, Nr, 31, **args, allow_failures=True, **LANE))
    for N in (700, 9001):
        ns = W.fibonacci_sphere(N)
        X, Nr = _cuda(ns.X), _cuda(ns.normals)
        npn = torch.as_tensor(W.stencil_size_groups(N, (101, 31, 6, 50)), device="cuda")
        _assert_equal(R, R.build_operator(X, Nr, npn, kappa_target=1e8),
                      R.build_operator(X, Nr, npn, kappa_target=1e8, **LANE))


@pytest.mark.parametrize("N", [800, 2500, 20_000])
def test_learned_start_on_teams_equals_lanes(R, N):
    """Networks with a scatter of errors: guesses accepted early, accepted
    after the full run, and searched on from."""
    ns = W.fibonacci_sphere(N)
    X, Nr = _cuda(ns.X), _cuda(ns.normals)
    op = R.build_operator(X, Nr, 31, kernel="imq", kappa_target=1e12)
    F, Y = R.features(op, X, Nr, 31)
    net = R.EpsNet(31, W.mlp_pack(W.mlp_init(93, seed=1)).astype(np.float32))
    net.train(F, Y, epochs=20, batch=256, lr=3e-3, seed=0)
    a = R.build_operator(X, Nr, 31, kernel="imq", kappa_target=1e12, mlps=[net])
    b = R.build_operator(X, Nr, 31, kernel="imq", kappa_target=1e12, mlps=[net], **LANE)
    _assert_equal(R, a, b)
    status = R.get_stencil_info(a)["status"]
    assert bool((status == 4).any()) and bool((status == 0).any())


@pytest.mark.parametrize("N,n", [(700, 2), (1000, 128), (2501, 31), (3001, 101), (9001, 50), (30_001, 70)])
def test_weights_on_teams_equal_lanes(R, N, n):
    ns = W.fibonacci_sphere(N)
    X, Nr = _cuda(ns.X), _cuda(ns.normals)
    radius = np.sqrt(4.0 * n / N)
    eps = _cuda(np.full(N, max(0.16 * np.sqrt(n) - 0.366, 0.1) / radius))
    for e, fails in ((eps, False), (torch.where(torch.arange(N, device="cuda") % 7 == 3, 1e-9, eps), n > 2)):
        a = R.build_operator(X, Nr, n, eps_override=e, allow_failures=True)
        b = R.build_operator(X, Nr, n, eps_override=e, allow_failures=True, **LANE)
        assert (a.status != 0) == fails or n == 2
        _assert_equal(R, a, b)
    # the same rows through the allocation-free call, in another order
    order = torch.as_tensor(np.random.default_rng(0).permutation(N), device="cuda")
    idx, w = R.get_rows(R.build_operator(X, Nr, n, eps_override=eps))
    got = R.stencil_weights_noalloc(X, Nr, idx[order].contiguous(), eps[order].contiguous())
    assert torch.equal(got, w[order])
