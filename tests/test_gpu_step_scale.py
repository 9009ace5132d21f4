"""Float32 steps of a linear problem whose fields are scaled by a power of two.

Multiplying u and v by 2^e multiplies every vector of a step by 2^e exactly, as
long as no value leaves float32's normal range, and every sum of products by
2^(2e): the iterations and the results have to be the same, scaled, although
squares of the fields (2^-120, 2^140) are outside float32's range.  Sizes: a
cluster and a grid of the resident kernel, and the phase kernels with less than
a row per thread and with more, replayed and from the host's loop.
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


def _cuda(a, dt=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


@pytest.mark.parametrize("N,n,graphs", [(642, 17, (True,)), (12000, 31, (True,)), (60000, 101, (True, False)),
                                        (200_003, 17, (True, False))])
@pytest.mark.parametrize("species", [1, 2])
def test_scaled_fields_take_the_same_iterations(R, N, n, graphs, species):
    ns = W.fibonacci_sphere(N)
    eps = (0.16 * np.sqrt(n) - 0.366) / np.sqrt(4.0 * n / N)
    op = R.build_operator(_cuda(ns.X), _cuda(ns.normals), n, eps_override=_cuda(np.full(N, eps)))
    u0 = (ns.X[:, 2] * (ns.X[:, 0] ** 2 - ns.X[:, 1] ** 2) + 0.1 * W.uniform_field(N, 3)).astype(np.float32)
    v0 = W.uniform_field(N, 4).astype(np.float32)
    for graph in graphs:
        p = R.StepParams(model="linear", nspecies=species, coef=(-1.0, 2.0), dt=0.05 * 4.0 * np.pi / N, delta_u=1.0,
                         delta_v=3.0, dtype=torch.float32, tol=1e-6, use_graph=graph)
        want = None
        for e in (0, -60, 70):
            st = R.StepState.create(_cuda(np.ldexp(u0, e), torch.float32),
                                    _cuda(np.ldexp(v0, e), torch.float32) if species == 2 else None)
            rep = R.step_imex(op, st, p, 5, allow_failure=True)
            assert rep["status"] == 0, e
            fields = [st.u, st.v][:species]
            got = (rep["total_iters"], rep["max_iters_u"], [x.double().cpu().numpy() * 2.0**-e for x in fields])
            want = want or got
            assert got[:2] == want[:2], e
            assert all(np.array_equal(a, b) for a, b in zip(got[2], want[2])), e
