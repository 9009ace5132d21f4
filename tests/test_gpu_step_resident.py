"""The resident step kernel (the operator in shared memory, one launch for all
steps) against the oracle's steps on the operator's own rows, at the sizes
where its plan changes: one slice of 32 rows and less, blocks with a partial
last slice, clusters with blocks without rows, the cooperative grid, mixed
stencil sizes, and operators just too large for it (the phase kernels).

Bounds as for every step path: 1e-9 in float64 (systems solved to 1e-12) and
1e-5 in float32 (to 1e-8), relative to the largest value.
"""
import numpy as np
import pytest
import torch

from oracle import stepping as ostp
from paper_1404_0812_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_1404_0812_gb300 as R
    return R


def _cuda(a, dt=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")


def _operator(R, N, n):
    ns = W.fibonacci_sphere(N)
    sizes = W.stencil_size_groups(N, (41, 17, 30)) if n == 0 else np.full(N, n, dtype=np.int32)
    eps = np.maximum(0.16 * np.sqrt(sizes) - 0.366, 0.1) / np.sqrt(4.0 * sizes / N)
    return ns, R.build_operator(_cuda(ns.X), _cuda(ns.normals), torch.as_tensor(sizes, device="cuda"),
                                eps_override=_cuda(eps))


@pytest.mark.parametrize("dtype,tol,bound", [(torch.float64, 1e-12, 1e-9), (torch.float32, 1e-8, 1e-5)])
@pytest.mark.parametrize("N,n,species,order", [
    (20, 7, 1, 2), (32, 9, 2, 1), (33, 17, 1, 2), (257, 17, 2, 2), (642, 31, 1, 4), (1031, 0, 2, 2), (2562, 31, 2, 3),
    (7001, 31, 1, 2), (9973, 17, 2, 2), (20011, 0, 2, 2), (40344, 50, 2, 2), (60013, 31, 1, 2), (90001, 50, 2, 2)])
def test_resident_steps_match_the_oracle(R, N, n, species, order, dtype, tol, bound):
    ns, op = _operator(R, N, n)
    idx, w = (t.cpu().numpy() for t in R.get_rows(op))
    L = lambda x: np.einsum("ij,ij->i", w, x[idx])
    if species == 1:
        u0, v0 = ns.X[:, 2] * (ns.X[:, 0] ** 2 - ns.X[:, 1] ** 2) + 0.1 * W.uniform_field(N, 3), None
        p = dict(model="none", dt=0.02 * 4.0 * np.pi / N, delta_u=1.0)
        sp = R.StepParams(model="none", nspecies=1, dt=p["dt"], delta_u=1.0)
    else:
        u0, v0 = W.schnakenberg_initial(N, seed=3)
        p = W.SCHNAKENBERG
        name, coef = R.model_coefs(p)
        sp = R.StepParams(model=name, nspecies=2, dt=p["dt"], delta_u=p["delta_u"], delta_v=p["delta_v"], coef=coef)
    sp.dtype, sp.tol, sp.order, sp.use_graph = dtype, tol, order, True
    u0 = u0.astype(np.float32).astype(np.float64)
    v0 = None if v0 is None else v0.astype(np.float32).astype(np.float64)
    state = R.StepState.create(_cuda(u0, dtype), None if v0 is None else _cuda(v0, dtype), order)
    rep = [R.step_imex(op, state, sp, k) for k in (1, 4)]   # two calls continue one run
    assert state.step == 5 and all(r["status"] == 0 and r["failed_step"] == -1 for r in rep)
    ref = ostp.imex_run(L, u0, v0, p, 5, order=order, tol=1e-14)
    for k in ("u", "v")[:species]:
        got, want = getattr(state, k).double().cpu().numpy(), ref[k]
        assert np.abs(got - want).max() <= bound * np.abs(want).max(), k


def test_resident_zero_right_hand_side_failure_and_report(R):
    """b = 0 gives x = 0 for that species only; a capped solve is reported with
    its step and residual while later steps run on."""
    ns, op = _operator(R, 642, 31)
    u0 = ns.X[:, 2]
    st = R.StepState.create(_cuda(u0), _cuda(np.zeros(642)))
    sp = R.StepParams(model="linear", nspecies=2, coef=(0.0, 0.0), dt=1e-3, delta_u=1.0, delta_v=1.0)
    rep = R.step_imex(op, st, sp, 3)
    assert rep["status"] == 0 and rep["max_iters_v"] == 0 and rep["max_iters_u"] >= 1
    assert float(st.v.abs().max()) == 0.0 and float(st.u.abs().max()) > 0.5
    st = R.StepState.create(_cuda(u0 + 0.1 * W.uniform_field(642, 1)))
    sp = R.StepParams(dt=1.0, maxit=1, tol=1e-12)
    rep = R.step_imex(op, st, sp, 2, allow_failure=True)
    assert rep["status"] != 0 and rep["failed_step"] == 0 and rep["max_iters_u"] == 1
    assert rep["last_relres_u"] > 1e-12 and rep["steps_done"] == 2
