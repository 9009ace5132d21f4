"""Calls of several threads, each on its own stream and objects, of sizes that ask
the same kernels for different amounts of shared memory: no call may make another
thread's launch fail, and the results are those of the calls one after the other.
"""
import threading

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


def _operator(R, N, n):
    ns = W.fibonacci_sphere(N)
    eps = (0.16 * np.sqrt(n) - 0.366) / np.sqrt(4.0 * n / N)
    return ns, R.build_operator(_cuda(ns.X), _cuda(ns.normals), n, eps_override=_cuda(np.full(N, eps)))


def _stepper(R, N):
    """Heat steps of a resident operator on one cluster."""
    ns, op = _operator(R, N, 31)
    u0 = _cuda(W.sph_harm_y32(ns.X))
    st = R.StepState.create(u0.clone())
    p = R.StepParams(dt=0.02 * 4.0 * np.pi / N, delta_u=1.0, tol=1e-12)

    def run(stream):
        with torch.cuda.stream(stream):
            st.u.copy_(u0)
            st.has_history, st.step, st.t = 0, 0, 0.0
            R.step_imex(op, st, p, 1, stream=stream)
        stream.synchronize()
        return st.u.clone()
    return run


def _trainer(R, n):
    rng = np.random.default_rng(n)
    start = W.mlp_pack(W.mlp_init(3 * n, seed=n)).astype(np.float32)
    net = R.EpsNet(n, start)
    X = _cuda(rng.uniform(-1.0, 1.0, (300, 3 * n)), torch.float32)
    y = _cuda(rng.uniform(-1.0, 1.0, 300), torch.float32)

    def run(stream):
        net.load(start)
        net.train(X, y, epochs=1, batch=128, lr=1e-3, seed=1, stream=stream)
        return torch.as_tensor(net.params())
    return run


@pytest.mark.parametrize("make,sizes", [(_stepper, (642, 5000) * 4), (_trainer, (11, 101) * 4)])
def test_threads_of_different_sizes(R, make, sizes):
    runs = [make(R, s) for s in sizes]
    streams = [torch.cuda.Stream() for _ in sizes]
    torch.cuda.synchronize()
    want = [run(stream) for run, stream in zip(runs, streams)]
    torch.cuda.synchronize()
    errors = []

    def loop(k):
        try:
            for _ in range(300):
                assert torch.equal(runs[k](streams[k]), want[k])
        except Exception as e:   # handed to the test's own thread
            errors.append(e)

    threads = [threading.Thread(target=loop, args=(k,)) for k in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
