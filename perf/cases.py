"""The workloads by which the library's speed is measured.

A case is a dict of plain values; ``prepare`` makes what a user's program has
in hand before the call, ``run`` is one pass through the public entry points
and returns everything the path computes, ``work`` is what a pass cannot do
without and ``exact`` the same outputs from plain torch in 64 bits.

Kinds and what each stands for in real use:

* build     a new operator on a node set: stencils, shape parameters by the
            plain search, weights.  The convergence studies build on a few
            hundred to tens of thousands of nodes, over and over.
* learned   the same with the search started from trained networks: the large
            production build, all four stencil sizes in one operator.
* reweight  weights of known stencils at known shape parameters without
            allocation: a time loop on an evolving surface, every step.
* apply     y = L u, the explicit part of a time loop.
* step      a simulation from its initial state: heat equation in float64,
            reaction-diffusion in float32, BiCGSTAB, replayed from a graph.
* lu        the same with the direct solver (nodes in an order of small
            bandwidth; the factors live with the operator).
* train     training of an eps network on pairs of a plain search.
* order     a locality ordering of scattered nodes before the build.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

import paper_1404_0812_gb300 as R
from paper_1404_0812_gb300 import workloads as W

KERNELS = ("imq", "gaussian")
MIXED = (31, 50, 70, 101)
MODELS = {"none": None, "schnakenberg": W.SCHNAKENBERG, "gray_scott": W.GRAY_SCOTT}


def listed():
    return [
        # the smallest configuration: 2562-node sphere, Gaussian, kappa_T 1e12
        dict(name="build_sphere_2562", kind="build", surface="sphere", N=2562, n=31, kernel="gaussian",
             kappa=1e12),
        # the 40k torus of the Turing runs
        dict(name="build_torus_40k", kind="build", surface="torus", N=40344, n=50, kernel="imq", kappa=1e12),
        # the headline build: 1M nodes, four stencil sizes, learned start
        dict(name="learned_mixed_1m", kind="learned", N=1_000_000, n=0, kappa=1e12),
        # weights of an evolving 10k-node surface, once per time step
        dict(name="reweight_10k", kind="reweight", N=10242, n=31, kernel="imq"),
        # the smallest call of all: one float64 apply on the small sphere
        dict(name="apply_f64_2562", kind="apply", N=2562, n=31, f64=True),
        # the largest apply: 63M nonzeros in float32
        dict(name="apply_f32_mixed_1m", kind="apply", N=1_000_000, n=0, f64=False),
        # heat equation on the small sphere in float64 (one species)
        dict(name="step_heat_2562_f64", kind="step", surface="sphere", N=2562, n=31, f64=True, model="none",
             order=2, steps=50),
        # Turing patterns on the 40k torus in float32 (two species)
        dict(name="step_turing_torus_f32", kind="step", surface="torus", N=40344, n=50, f64=False,
             model="schnakenberg", order=2, steps=20),
        # the same at production size
        dict(name="step_turing_1m_f32", kind="step", surface="sphere", N=1_000_000, n=0, f64=False,
             model="schnakenberg", order=2, steps=5),
        # direct solves on a small torus (two systems per step)
        dict(name="lu_torus_2400_f64", kind="lu", N=2400, n=31, f64=True, steps=3),
        # one network, 50k pairs, mini-batches of 1024
        dict(name="train_n50_50k", kind="train", n=50, count=50_000, batch=1024, epochs=2),
        # Z-order of 1M scattered nodes
        dict(name="order_1m", kind="order", N=1_000_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _torus(N):
    """The nearest size of a staggered torus grid (N = 6 m^2)."""
    return 6 * max(8, round(math.sqrt(N / 6))) ** 2


def draw(rng):
    kind = rng.choice(("build", "build", "learned", "reweight", "apply", "step", "step", "lu", "train", "order"))
    if kind == "build":
        n = rng.randint(11, 101)
        N = min(_log_int(rng, 642, 100_000), int(1e10 / n**3))
        surface = rng.choice(("sphere", "torus", "bumpy"))
        return dict(kind=kind, surface=surface, N=_torus(N) if surface == "torus" else N, n=n,
                    kernel=rng.choice(KERNELS), kappa=rng.choice((1e8, 1e10, 1e12)))
    if kind == "learned":
        n = rng.choice((0,) + MIXED)
        return dict(kind=kind, N=_log_int(rng, 20_000, 200_000 if n == 101 else 500_000), n=n, kappa=1e12)
    if kind == "reweight":
        n = rng.randint(11, 101)
        return dict(kind=kind, N=min(_log_int(rng, 642, 200_000), int(1e10 / n**3)), n=n,
                    kernel=rng.choice(KERNELS))
    if kind == "apply":
        n = rng.choice((0, rng.randint(11, 101)))
        return dict(kind=kind, N=min(_log_int(rng, 642, 1_000_000), 63_000_000 // (n or 63)), n=n,
                    f64=rng.random() < 0.5)
    if kind == "step":
        surface, model = rng.choice(("sphere", "torus")), rng.choice(tuple(MODELS))
        n = rng.choice((17, 31, 50, 70))
        N = min(_log_int(rng, 642, 600_000), 30_000_000 // n)
        return dict(kind=kind, surface=surface, N=_torus(N) if surface == "torus" else N, n=n,
                    f64=rng.random() < 0.5, model=model, order=rng.choice((2, 2, 3, 4)), steps=rng.randint(4, 12))
    if kind == "lu":
        return dict(kind=kind, N=6 * rng.randint(10, 24) ** 2, n=rng.choice((17, 31)), f64=rng.random() < 0.5,
                    steps=rng.randint(2, 4))
    if kind == "train":
        return dict(kind=kind, n=rng.randint(11, 101), count=_log_int(rng, 2000, 60_000),
                    batch=rng.choice((256, 512, 1024, 2048)), epochs=rng.randint(1, 3))
    return dict(kind=kind, N=_log_int(rng, 1000, 2_000_000))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _cuda(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype).to("cuda")


@functools.lru_cache(maxsize=8)
def _base(surface, N):
    if surface == "torus":
        return W.torus_staggered(round(math.sqrt(N / 6)))
    return W.bumpy_sphere(N) if surface == "bumpy" else W.fibonacci_sphere(N)


def _surface(surface, N, seed):
    """Nodes and unit normals on the device, in an orientation of the seed's."""
    ns = _base(surface, N)
    Q, _ = np.linalg.qr(np.random.default_rng(seed).standard_normal((3, 3)))
    return _cuda(ns.X @ Q), _cuda(ns.normals @ Q)


def _banded_torus(N, seed):
    """The torus numbered along its folded longitude: the nodes of both sides
    in turn, which keeps every stencil within a narrow band."""
    perm = torch.as_tensor(np.argsort(np.abs(_base("torus", N).extra["lam"]), kind="stable")).to("cuda")
    X, Nr = _surface("torus", N, seed)
    return X[perm].contiguous(), Nr[perm].contiguous()


def _sizes(N, n):
    """n, or for n = 0 the four sizes in four latitude bands."""
    return n if n else torch.as_tensor(W.stencil_size_groups(N, MIXED)).to("cuda")


def _fixed_eps(surface, N, n):
    """Shape parameters (one per node) of a condition number of about 1e8 for
    the IMQ on quasi-uniform nodes: eps times the stencil radius grows like
    the square root of the stencil size."""
    area = 4.0 * math.pi**2 / 3.0 if "torus" in surface else 4.0 * math.pi
    size = np.full(N, n) if n else W.stencil_size_groups(N, MIXED)
    radius = np.sqrt(area / N * size / math.pi)
    return (0.16 * np.sqrt(size) - 0.366) / radius


def _nodes(surface, N, seed):
    return _banded_torus(N, seed) if surface == "banded torus" else _surface(surface, N, seed)


def _operator(surface, N, n, seed):
    X, Nr = _nodes(surface, N, seed)
    return R.build_operator(X, Nr, _sizes(N, n), kernel="imq", eps_override=_cuda(_fixed_eps(surface, N, n)))


@functools.lru_cache(maxsize=4)
def _pairs(n):
    """Features and targets of the plain search on three spheres."""
    F, Y = [], []
    for N in (4000, 16000, 64000):
        X, Nr = _surface("sphere", N, n)
        op = R.build_operator(X, Nr, n, kernel="imq", kappa_target=1e12)
        f, y = R.features(op, X, Nr, n)
        F.append(f.clone())
        Y.append(y.clone())
    return torch.cat(F), torch.cat(Y)


@functools.lru_cache(maxsize=8)
def _network(n):
    """A trained network for stencil size n, kept as a program keeps its
    weights: Adam on the pairs, then its last layer by least squares."""
    F, Y = _pairs(n)
    p = {k: _cuda(v, torch.float32).requires_grad_() for k, v in W.mlp_init(3 * n, seed=n).items()}
    gelu = torch.nn.functional.gelu

    def hidden(f, p):
        return gelu(gelu(f @ p["W1"] + p["b1"]) @ p["W2"] + p["b2"])

    mean = Y.mean()
    steps = 600
    adam = torch.optim.Adam(p.values(), lr=3e-3)
    for k in range(steps):
        adam.param_groups[0]["lr"] = 3e-3 * 0.5 * (1.0 + math.cos(math.pi * k / steps))
        adam.zero_grad()
        ((hidden(F, p) @ p["W3"] + p["b3"])[:, 0] - (Y - mean)).square().mean().backward()
        adam.step()
    with torch.no_grad():
        h = torch.nn.functional.pad(hidden(F.double(), {k: v.double() for k, v in p.items()}), (0, 1), value=1.0)
    h = h.cpu().numpy()
    last = np.linalg.solve(h.T @ h + 1e-9 * len(h) * np.eye(65), h.T @ Y.double().cpu().numpy())
    flat = {k: v.detach().cpu().numpy() for k, v in p.items()} | {"W3": last[:-1], "b3": last[-1:]}
    return R.EpsNet(n, W.mlp_pack(flat).astype(np.float32))


def _training_set(case, seed):
    """count pairs: rows of the search's pairs, drawn by the seed, with a
    relative scatter of the offsets as other surfaces would give them."""
    F, Y = _pairs(case["n"])
    g = torch.Generator().manual_seed(seed)
    pick = torch.randint(len(Y), (case["count"],), generator=g)
    f = F[pick.to("cuda")] * (1.0 + 0.02 * torch.randn(case["count"], 3 * case["n"], generator=g).to("cuda"))
    return f, Y[pick.to("cuda")] + 0.01 * torch.randn(case["count"], generator=g).to("cuda")


def _initial(case, seed):
    """Initial fields of a simulation (numpy float64)."""
    ns = _base(case.get("surface", "torus"), case["N"])
    if case.get("model", "schnakenberg") == "none":
        u = W.sph_harm_y32(ns.X) + 0.1 * W.uniform_field(case["N"], seed)
        return u, None
    if case.get("model") == "gray_scott":
        return W.gray_scott_initial(ns.X, seed=seed, spots=min(50, case["N"] // 20), radius=0.05)
    return W.schnakenberg_initial(case["N"], seed=seed)


def _step_params(case):
    """Keyword arguments of the step and (delta_u, delta_v)."""
    s = MODELS[case.get("model", "schnakenberg")]
    if s is None:
        h2 = 4.0 * math.pi / case["N"]   # the 2562-node sphere's 1e-4, scaled with the spacing
        return dict(model="none", nspecies=1, dt=0.02 * h2, delta_u=1.0, delta_v=0.0, coef=())
    name, coef = R.model_coefs(s)
    return dict(model=name, nspecies=2, dt=s["dt"], delta_u=s["delta_u"], delta_v=s["delta_v"], coef=coef)


def prepare(case, seed):
    kind, N, n = case["kind"], case.get("N"), case.get("n")
    s = dict(case)
    if kind == "build":
        s["X"], s["normals"] = _surface(case["surface"], N, seed)
    elif kind == "learned":
        s["X"], s["normals"] = _surface("sphere", N, seed)
        s["sizes"] = _sizes(N, n)
        s["nets"] = [_network(k) for k in ((n,) if n else MIXED)]
    elif kind == "reweight":
        # the sphere the stencils belong to, a moment later: a smooth
        # radial motion, normals of the moved surface up to its slope
        X, s["normals"] = _surface("sphere", N, seed)
        op = R.build_operator(X, s["normals"], n, kernel="imq", eps_override=_cuda(_fixed_eps("sphere", N, n)))
        s["stencils"] = R.get_rows(op)[0]
        s["X"] = (X * (1.0 + 0.01 * torch.sin(3.0 * X[:, :1]))).contiguous()
        s["eps"] = _cuda(_fixed_eps("sphere", N, n)) * (1.0 if case["kernel"] == "imq" else 1.4)
        s["weights"] = torch.empty((N, n), dtype=torch.float64, device="cuda")
    elif kind == "apply":
        s["op"] = _operator("sphere", N, n, seed)
        s["u"] = _cuda(W.uniform_field(N, seed), torch.float64 if case["f64"] else torch.float32)
    elif kind in ("step", "lu"):
        dt = torch.float64 if case["f64"] else torch.float32
        u, v = _initial(case, seed)
        s["op"] = _operator(case.get("surface", "banded torus"), N, n, seed)
        s["u0"], s["v0"] = _cuda(u, dt), None if v is None else _cuda(v, dt)
        order = case.get("order", 2)
        s["state"] = R.StepState.create(s["u0"].clone(), None if v is None else s["v0"].clone(), order)
        s["params"] = R.StepParams(dtype=dt, tol=1e-12 if case["f64"] else 1e-7, use_graph=True, order=order,
                                   solver="lu" if kind == "lu" else "bicgstab", **_step_params(case))
    elif kind == "train":
        f, y = _training_set(case, seed)
        s["feats"], s["target"] = f, y
        s["start"] = W.mlp_pack(W.mlp_init(3 * n, seed=seed)).astype(np.float32)
        s["net"], s["seed"] = R.EpsNet(n, s["start"]), seed
    else:
        X, _ = _surface("bumpy", N, seed)
        s["X"] = X[torch.as_tensor(np.random.default_rng(seed).permutation(N)).to("cuda")].contiguous()
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _built(op):
    ell = R.get_ell(op)   # views that keep op alive
    eps, kappa, _ = R.get_eps(op)
    return dict(row_node=ell["row_node"], idx=ell["idx"], weights=ell["w64"], eps=eps, kappa=kappa)


def run(s):
    kind = s["kind"]
    if kind == "build":
        return _built(R.build_operator(s["X"], s["normals"], s["n"], kernel=s["kernel"], kappa_target=s["kappa"]))
    if kind == "learned":
        return _built(R.build_operator(s["X"], s["normals"], s["sizes"], kernel="imq", kappa_target=s["kappa"],
                                       mlps=s["nets"]))
    if kind == "reweight":
        return dict(weights=R.stencil_weights_noalloc(s["X"], s["normals"], s["stencils"], s["eps"],
                                                      kernel=s["kernel"], weights=s["weights"]))
    if kind == "apply":
        return dict(y=R.apply(s["op"], s["u"]))
    if kind in ("step", "lu"):
        st = s["state"]
        st.u.copy_(s["u0"])
        if st.v is not None:
            st.v.copy_(s["v0"])
        st.has_history, st.step, st.t = 0, 0, 0.0
        R.step_imex(s["op"], st, s["params"], s["steps"])
        # the solution at both levels (the kinetics' past values follow from them)
        return dict(u=st.u, v=st.v, u_prev=st.u_prev, v_prev=st.v_prev)
    if kind == "train":
        s["net"].load(s["start"])
        losses = s["net"].train(s["feats"], s["target"], epochs=s["epochs"], batch=s["batch"], lr=1e-3,
                                seed=s["seed"])
        return dict(params=s["net"].params(), losses=np.asarray(losses, dtype=np.float32))
    return dict(perm=R.morton_order(s["X"]))


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    kind, N, n = case["kind"], case.get("N"), case.get("n")
    size = np.full(N or 1, n, dtype=np.float64) if n else W.stencil_size_groups(N, MIXED).astype(np.float64)
    nnz = float(size.sum())
    # one factorisation, the four solves of a stencil's weights and one pass
    # over its pairs; a plain search needs five evaluations (a factorisation
    # and ten Lanczos solves each), an accepted guess one with seven
    factor, solve, pairs = float((size**3).sum()) / 3, 2 * float((size**2).sum()), 16 * float((size**2).sum())
    weights = factor + 4 * solve + pairs
    if kind == "build":
        return dict(bytes=48.0 * N + nnz * 16 + 24.0 * N, flops=weights + 4 * factor + 55 * solve + 5 * pairs)
    if kind == "learned":
        return dict(bytes=52.0 * N + nnz * 16 + 24.0 * N, flops=weights + 8 * solve + pairs)
    if kind == "reweight":
        return dict(bytes=48.0 * N + nnz * 12 + 8.0 * N, flops=weights + solve + pairs)
    e = 8.0 if case.get("f64") else 4.0
    if kind == "apply":
        return dict(bytes=nnz * (e + 4) + 2 * N * e, flops=2 * nnz)
    if kind == "step":
        species = 1 if MODELS[case["model"]] is None else 2
        # the right-hand side and two BiCGSTAB iterations of two products each
        return dict(bytes=case["steps"] * (5 * nnz * (e + 4) + 40 * species * N * e),
                    flops=case["steps"] * species * 10 * nnz)
    if kind == "lu":
        band = 2.0 * math.sqrt(N * n) * 2   # lower and upper bandwidth after the ordering, about
        return dict(bytes=case["steps"] * 2 * N * 2 * band * 8, flops=case["steps"] * 2 * N * 4 * band)
    if kind == "train":
        samples = float(case["count"]) * case["epochs"]
        return dict(bytes=samples * (3 * n + 1) * 4, flops=samples * 6 * (3 * n * 64 + 64 * 64 + 64))
    return dict(bytes=28.0 * N, flops=0.0)


# ---------------------------------------------------------------------------
# the same outputs in 64 bits from plain torch
# ---------------------------------------------------------------------------

def _nearest(X, n):
    """The node and its n - 1 nearest others by (d^2, index)."""
    N, out = len(X), []
    for i in range(0, N, 2048):
        q = X[i:i + 2048]
        d = q[:, None, :] - X[None, :, :]
        d2 = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
        me = torch.arange(i, i + len(q), device=X.device)
        d2[torch.arange(len(q), device=X.device), me] = -1.0
        j = torch.topk(d2, min(N, n + 16), largest=False).indices.sort(dim=1).values
        order = torch.sort(d2.gather(1, j), dim=1, stable=True).indices
        out.append(j.gather(1, order)[:, :n])
    return torch.cat(out)


def _augmented(X, idx, eps, kernel):
    """Offsets x_i - x_j of each stencil in units of its radius, the radius,
    the kernel's psi and the augmented interpolation matrix."""
    P = X[idx] - X[idx[:, :1]]
    rs = P.square().sum(2).max(1).values.sqrt()
    P = P / rs[:, None, None]
    D = P[:, :, None, :] - P[:, None, :, :]
    e2 = ((eps * rs) ** 2)[:, None, None]
    x = e2 * D.square().sum(3)
    phi = torch.exp(-x) if kernel == "gaussian" else (1.0 + x).rsqrt()
    psi = -2.0 * e2 * phi if kernel == "gaussian" else -e2 * phi**3
    A = torch.nn.functional.pad(phi, (0, 1, 0, 1), value=1.0)
    A[:, -1, -1] = 0.0
    return D, rs, psi, A


def _weights(X, normals, idx, eps, kernel):
    """First row of sum_d G^d G^d of every stencil."""
    D, rs, psi, A = _augmented(X, idx, eps, kernel)
    nv = normals[idx]
    nv = nv / nv.square().sum(2, keepdim=True).sqrt()
    PD = D - nv[:, :, None, :] * (D * nv[:, :, None, :]).sum(3, keepdim=True)   # P(x_i)(x_i - x_j)
    B = psi[..., None] * PD
    LU = torch.linalg.lu_factor(A)
    solve = lambda r: torch.linalg.lu_solve(*LU, torch.nn.functional.pad(r, (0, 0, 0, 1)))[:, :-1]
    g = solve(B[:, 0])                                                         # A^{-1} [B^d row 0; 0]
    v = torch.einsum("sijd,sid->sj", B, g)
    return solve(v[..., None])[..., 0] / (rs * rs)[:, None]


def _ell(a, n):
    """Rows (N x n) in the operator's sliced layout, padded with zeros."""
    N, npad = len(a), -(-n // 4) * 4
    p = a.new_zeros(-(-N // 32) * 32, npad)
    p[:N, :n] = a
    return p.view(-1, 32, npad // 4, 4).permute(0, 2, 1, 3).reshape(-1)


def _exact_build(case, seed):
    if case["N"] > 4000 or case["n"] > 31:
        return None
    X, Nr = _surface(case["surface"], case["N"], seed)
    idx = _nearest(X, case["n"])

    def log_kappa(eps):
        lam = torch.linalg.eigvalsh(_augmented(X, idx, eps, case["kernel"])[3]).abs()
        return (lam.max(1).values / lam.min(1).values).log() - math.log(case["kappa"])

    rs = (X[idx] - X[idx[:, :1]]).square().sum(2).max(1).values.sqrt()
    lo, hi = torch.log(0.01 / rs), torch.log(4.0 / rs)
    for _ in range(40):
        mid = 0.5 * (lo + hi)
        above = log_kappa(mid.exp()) > 0.0
        lo, hi = torch.where(above, mid, lo), torch.where(above, hi, mid)
    eps = (0.5 * (lo + hi)).exp()
    return dict(row_node=None, idx=None, weights=_ell(_weights(X, Nr, idx, eps, case["kernel"]), case["n"]), eps=eps,
                kappa=torch.full_like(eps, case["kappa"]))


def _fixed_rows(surface, N, n, seed):
    """Stencils and weights of _operator, row by row in node order."""
    X, Nr = _nodes(surface, N, seed)
    idx = _nearest(X, n)
    eps = _cuda(_fixed_eps(surface, N, n))
    w = [_weights(X, Nr, idx[i:i + 1024], eps[i:i + 1024], "imq") for i in range(0, N, 1024)]
    return idx, torch.cat(w)


def _react(model, u, v):
    p = MODELS[model]
    if model == "schnakenberg":
        return p["gamma"] * (p["a"] - u + u * u * v), p["gamma"] * (p["b"] - u * u * v)
    if model == "gray_scott":
        return -u * v * v + p["F"] * (1.0 - u), u * v * v - (p["F"] + p["k"]) * v
    return torch.zeros_like(u), None


def _bicgstab(A, b, x):
    r = b - A(x)
    rh, p, q = r.clone(), torch.zeros_like(r), torch.zeros_like(r)
    rho = alpha = omega = 1.0
    for _ in range(400):
        if float(r.norm()) <= 1e-14 * float(b.norm()):
            break
        rho1 = float(rh @ r)
        p = r + (rho1 / rho) * (alpha / omega) * (p - omega * q)
        rho, q = rho1, A(p)
        alpha = rho / float(rh @ q)
        s = r - alpha * q
        if float(s.norm()) <= 1e-14 * float(b.norm()):
            return x + alpha * p
        t = A(s)
        omega = float(t @ s) / float(t @ t)
        x, r = x + alpha * p + omega * s, s - omega * t
    return x


# c0 u^{n+1} - cl dt L u^{n+1} = sum a_j u^{n-j} + cl dt sum b_j f^{n-j}
SBDF = {1: (1, 1, (1,), (1,)), 2: (3, 2, (4, -1), (2, -1)), 3: (11, 6, (18, -9, 2), (3, -3, 1)),
        4: (25, 12, (48, -36, 16, -3), (4, -6, 4, -1))}


def _exact_step(case, seed):
    if case["N"] > 45_000 or not case["n"]:
        return None
    N, model, dt = case["N"], case.get("model", "schnakenberg"), torch.float64 if case["f64"] else torch.float32
    idx, w = _fixed_rows(case.get("surface", "banded torus"), N, case["n"], seed)
    p, fields = _step_params(case), [None if a is None else _cuda(a, dt).double() for a in _initial(case, seed)]
    hist, f_hist = [[fields[0]], [fields[1]]], [[], []]
    for k in range(case["steps"]):
        order = min(case.get("order", 2), k + 1)
        c0, cl, a, b = SBDF[order]
        f = _react(model, fields[0], fields[1])
        for sp in range(p["nspecies"]):
            f_hist[sp].insert(0, f[sp])
        new = [None, None]
        for sp, delta in zip(range(p["nspecies"]), (p["delta_u"], p["delta_v"])):
            rhs = sum(aj * h for aj, h in zip(a, hist[sp])) + cl * p["dt"] * sum(bj * h for bj, h in zip(b, f_hist[sp]))
            new[sp] = _bicgstab(lambda x: c0 * x - cl * p["dt"] * delta * (w * x[idx]).sum(1), rhs, fields[sp])
            hist[sp].insert(0, new[sp])
        fields = new
    two = p["nspecies"] == 2
    return dict(u=fields[0], v=fields[1], u_prev=hist[0][1], v_prev=hist[1][1] if two else None)


def _shuffles(count, epochs, seed):
    """The orders of the training pairs: Fisher-Yates by std::mt19937_64 (the
    64-bit Mersenne twister of Nishimura and Matsumoto)."""
    M64 = (1 << 64) - 1
    x = [seed & M64]
    for i in range(1, 312):
        x.append((6364136223846793005 * (x[-1] ^ (x[-1] >> 62)) + i) & M64)
    at, perm = 312, list(range(count))
    for _ in range(epochs):
        for i in range(count - 1, 0, -1):
            if at == 312:
                for k in range(312):
                    y = (x[k] & 0xFFFFFFFF80000000) | (x[(k + 1) % 312] & 0x7FFFFFFF)
                    x[k] = x[(k + 156) % 312] ^ (y >> 1) ^ (0xB5026F5AA96619E9 if y & 1 else 0)
                at = 0
            z = x[at]
            at += 1
            z ^= (z >> 29) & 0x5555555555555555
            z ^= (z << 17) & 0x71D67FFFEDA60000
            z ^= (z << 37) & 0xFFF7EEE000000000
            j = (z ^ (z >> 43)) % (i + 1)
            perm[i], perm[j] = perm[j], perm[i]
        yield torch.tensor(perm, device="cuda")


def _exact_train(case, seed):
    f, y = (t.double() for t in _training_set(case, seed))
    D = 3 * case["n"]
    start = W.mlp_pack(W.mlp_init(D, seed=seed)).astype(np.float32)
    theta = _cuda(start).requires_grad_()
    shapes = [(D, 64), (64,), (64, 64), (64,), (64, 1), (1,)]
    m, v, t, losses = torch.zeros_like(theta), torch.zeros_like(theta), 0, []
    for perm in _shuffles(case["count"], case["epochs"], seed):
        total = 0.0
        for b in range(0, case["count"], case["batch"]):
            sel = perm[b:b + case["batch"]]
            W1, b1, W2, b2, W3, b3 = (q.view(s) for q, s in
                                      zip(theta.split([math.prod(s) for s in shapes]), shapes))
            gelu = torch.nn.functional.gelu
            out = (gelu(gelu(f[sel] @ W1 + b1) @ W2 + b2) @ W3 + b3)[:, 0]
            sq = (out - y[sel]).square().sum()
            (g,) = torch.autograd.grad(sq / len(sel), theta)
            t, total = t + 1, total + float(sq)
            with torch.no_grad():
                m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
                theta -= 1e-3 * (m / (1 - 0.9**t)) / ((v / (1 - 0.999**t)).sqrt() + 1e-8)
        losses.append(total / case["count"])
    return dict(params=theta.detach(), losses=np.asarray(losses))


def exact(case, seed):
    """None where it would take too long (large searches and simulations, the
    learned build), for whole numbers, and for operators of mixed sizes."""
    kind, N, n = case["kind"], case.get("N"), case.get("n")
    if kind == "build":
        return _exact_build(case, seed)
    if kind == "reweight":
        if N > 45_000:
            return None
        X, Nr = _surface("sphere", N, seed)
        idx = _nearest(X, n)
        X = X * (1.0 + 0.01 * torch.sin(3.0 * X[:, :1]))
        eps = _cuda(_fixed_eps("sphere", N, n)) * (1.0 if case["kernel"] == "imq" else 1.4)
        return dict(weights=torch.cat([_weights(X, Nr, idx[i:i + 1024], eps[i:i + 1024], case["kernel"])
                                       for i in range(0, N, 1024)]))
    if kind == "apply":
        if N > 45_000 or not n:
            return None
        idx, w = _fixed_rows("sphere", N, n, seed)
        u = _cuda(W.uniform_field(N, seed), torch.float64 if case["f64"] else torch.float32).double()
        return dict(y=(w * u[idx]).sum(1))
    if kind in ("step", "lu"):
        return _exact_step(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    return None
