"""Steps of a large operator from the host's loop (use_graph off) against the
replayed graph: the same bits, iterations and reports.  The loop launches an
iteration before it knows whether the one before it was the last; the cases are
its ends: no iteration at all (a field at rest, a zero right-hand side), one
iteration, a cap on the iterations, and ordinary steps of one and two species.
"""
import numpy as np
import pytest
import torch

from paper_1404_0812_gb300 import workloads as W

pytestmark = pytest.mark.gpu

N = 160_003


@pytest.fixture(scope="module")
def R():
    import paper_1404_0812_gb300 as R
    return R


def _cuda(a, dt=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


@pytest.fixture(scope="module")
def op(R):
    ns = W.fibonacci_sphere(N)
    eps = (0.16 * np.sqrt(31) - 0.366) / np.sqrt(4.0 * 31 / N)
    return R.build_operator(_cuda(ns.X), _cuda(ns.normals), 31, eps_override=_cuda(np.full(N, eps)))


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("start,species,kw", [
    ("rest", 1, {}), ("zero", 2, {}), ("noise", 1, dict(tol=0.5)), ("noise", 2, dict(maxit=1)),
    ("noise", 1, dict(maxit=3, tol=1e-15)), ("noise", 1, {}), ("noise", 2, {})])
def test_host_loop_and_graph_agree(R, op, dtype, start, species, kw):
    u0 = {"rest": np.ones(N), "zero": np.zeros(N), "noise": 1.0 + 0.5 * W.uniform_field(N, 1)}[start]
    v0 = 0.25 + 0.1 * W.uniform_field(N, 2)
    out = []
    for graph in (True, False):
        p = R.StepParams(model="none", nspecies=species, dt=0.3 * 4.0 * np.pi / N, delta_u=1.0, delta_v=0.3, dtype=dtype,
                         use_graph=graph, **{"tol": 1e-12 if dtype == torch.float64 else 1e-6, **kw})
        st = R.StepState.create(_cuda(u0, dtype), _cuda(v0, dtype) if species == 2 else None)
        rep = R.step_imex(op, st, p, 3, allow_failure=True)
        out.append((rep, st.u.clone(), None if st.v is None else st.v.clone()))
    assert out[0][0] == out[1][0]
    assert torch.equal(out[0][1], out[1][1])
    assert species == 1 or torch.equal(out[0][2], out[1][2])
