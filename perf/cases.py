"""The work whose speed is followed: products, operators, preconditioner and whole solves through the public API.

A case is a dict of plain values; its "kind" says which call it is:
  apply      birkhoff_apply (or birkhoff_apply_T) on [1, comps, pitch] vectors of a plan of size n
  batch      birkhoff_apply_batch over one plan of each size 2^klo .. 2^khi
  kkt        kkt_apply of the KKT operator at a linearised trajectory
  precond    precond_apply of the KKT preconditioner at a linearised trajectory
  newton     newton_solve of an orbit transfer to radius rf from the spiral guess
"""
import math

import numpy as np
import torch

from paper_2509_01855_gb300 import _lib, api

DTYPES = {"f64": torch.float64, "f32": torch.float32}
THRUST = 0.01            # nominal thrust parameter of the orbit kind (serving's value)
RF_RANGE, TF_RANGE = (1.2, 2.0), (10.0, 30.0)   # target radius and transfer time of served requests


def listed():
    return [
        # one short trajectory's product, four states: latency decides
        dict(name="apply_f64_256", kind="apply", n=256, comps=4, dtype="f64", trans=False),
        # the same chain transposed in single precision at a middle size of the serving mix
        dict(name="applyT_f32_4096", kind="apply", n=4096, comps=4, dtype="f32", trans=True),
        # ordinary double-precision products, both directions
        dict(name="applyT_f64_16384", kind="apply", n=16384, comps=4, dtype="f64", trans=True),
        dict(name="apply_f64_65536", kind="apply", n=65536, comps=4, dtype="f64", trans=False),
        # the million-point product in both precisions
        dict(name="apply_f64_1048576", kind="apply", n=1048576, comps=4, dtype="f64", trans=False),
        dict(name="apply_f32_1048576", kind="apply", n=1048576, comps=4, dtype="f32", trans=False),
        # a grid size that is no power of two (a user's own mesh)
        dict(name="apply_f64_100000", kind="apply", n=100000, comps=4, dtype="f64", trans=False),
        # one product for every size of the serving mix in one call
        dict(name="batch_f32_serving", kind="batch", klo=8, khi=16, comps=4, dtype="f32", trans=False),
        # one Krylov step's two halves on the orbit problem: operator and preconditioner
        dict(name="kkt_orbit_f64_262144", kind="kkt", problem="orbit", n=262144, dtype="f64"),
        dict(name="precond_orbit_f64_131072", kind="precond", problem="orbit", n=131072, dtype="f64"),
        # a served request (single-precision inner solves) and the million-point double-precision solve
        dict(name="newton_f32_4096", kind="newton", n=4096, dtype="f32", rf=1.7),
        dict(name="newton_f64_1048576", kind="newton", n=1048576, dtype="f64", rf=1.5),
    ]


def draw(rng):
    kind = rng.choice(["apply"] * 5 + ["batch", "kkt", "kkt", "precond", "precond", "newton", "newton"])
    dtype = rng.choice(["f64", "f32"])
    if kind == "apply":
        if rng.random() < 0.3:   # any N: dense products up to 1024, Bluestein's convolution above
            n = int(round(2.0 ** rng.uniform(7.0, 19.0))) | 1
        else:
            n = 1 << rng.randint(7, 22)
        return dict(kind=kind, n=n, comps=rng.choice([1, 2, 3, 4, 4, 6]), dtype=dtype, trans=rng.random() < 0.5)
    if kind == "batch":
        klo = rng.randint(8, 11)
        return dict(kind=kind, klo=klo, khi=rng.randint(klo + 2, 16), comps=rng.choice([2, 4, 4]), dtype=dtype,
                    trans=rng.random() < 0.5)
    if kind == "newton":
        return dict(kind=kind, n=1 << rng.randint(8, 19), dtype=dtype, rf=round(rng.uniform(*RF_RANGE), 3))
    return dict(kind=kind, problem=rng.choice(["orbit", "orbit", "orbit", "dblint"]), n=1 << rng.randint(8, 20),
                dtype=dtype)


# --- inputs ------------------------------------------------------------------------------------
def _gen(seed, tag):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + tag) & 0x7FFFFFFFFFFFFFFF)
    return g


def _normal(shape, seed, tag):
    return torch.randn(shape, generator=_gen(seed, tag), dtype=torch.float64, device="cuda")


def _uniform(lo_hi, seed, tag):
    u = float(np.random.default_rng([int(seed), tag]).uniform())
    return lo_hi[0] + (lo_hi[1] - lo_hi[0]) * u


def _tau(n):
    j = torch.arange(n + 1, dtype=torch.float64, device="cuda")
    tau = torch.sin(math.pi * (2 * j - n) / (2 * n))
    tau[0], tau[-1] = -1.0, 1.0
    return tau


def _pitch(n):
    return (n + 1 + 31) // 32 * 32


def _vectors(n, comps, dtype, seed, tag=1):
    v = torch.zeros(1, comps, _pitch(n), dtype=DTYPES[dtype], device="cuda")
    v[:, :, :n + 1] = _normal((1, comps, n + 1), seed, tag).to(v.dtype)
    return v


def _spiral(t, rf, tf):
    """Tangential-thrust spiral from the unit circular orbit to radius rf at tf: states and thrust."""
    ae = (1.0 - rf ** -0.5) / tf
    v = 1.0 - ae * t
    X = torch.stack([1.0 / v**2, (1.0 - v**4) / (4.0 * ae), 2.0 * ae / v**3, v])
    U = torch.zeros(2, t.numel(), dtype=torch.float64, device="cuda")
    U[1] = ae
    return X, U


def _point(case, seed):
    """A trajectory to linearise at: (kind code, t_f, parameters, X, U, lambda, nu)."""
    n = case["n"]
    tau = _tau(n)
    wq = torch.clamp(math.pi / n * torch.sqrt(torch.clamp(1 - tau * tau, min=0.0)), min=1.0 / n**2)
    if case["problem"] == "orbit":
        rf, tf = _uniform(RF_RANGE, seed, 2), _uniform(TF_RANGE, seed, 3)
        X, U = _spiral(0.5 * tf * (tau + 1.0), rf, tf)
        code, params, ne = _lib.BK_ORBIT, (THRUST, rf), 3
    else:
        tf, code, params, ne = 1.0, _lib.BK_DBL_INT, (), 2
        X = torch.stack([0.5 * (tau + 1.0), torch.zeros_like(tau)])
        U = torch.zeros(1, n + 1, dtype=torch.float64, device="cuda")
    X = X + 0.01 * _normal(X.shape, seed, 4)
    U = U + 0.01 * _normal(U.shape, seed, 5)
    lam = wq * _normal(X.shape, seed, 6)
    return code, tf, params, X, U, lam, _normal((ne,), seed, 7)


def _kkt_input(case, seed, nx, nu, ne):
    """A KKT vector [X | U | lambda | nu, padded to 32] with normal entries and zero padding."""
    P, L = _pitch(case["n"]), case["n"] + 1
    z = torch.zeros((2 * nx + nu) * P + 32, dtype=DTYPES[case["dtype"]], device="cuda")
    z[:(2 * nx + nu) * P].view(2 * nx + nu, P)[:, :L] = _normal((2 * nx + nu, L), seed, 8).to(z.dtype)
    z[(2 * nx + nu) * P:(2 * nx + nu) * P + ne] = _normal((ne,), seed, 9).to(z.dtype)
    return z


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=case)
    if kind == "apply":
        st["plan"] = api.Plan(case["n"], n_comp=case["comps"], dtype=DTYPES[case["dtype"]], t0=0.0, tf=20.0)
        st["v"] = _vectors(case["n"], case["comps"], case["dtype"], seed)
        st["out"] = torch.zeros_like(st["v"])
    elif kind == "batch":
        ns = [1 << k for k in range(case["klo"], case["khi"] + 1)]
        st["plans"] = [api.Plan(n, n_comp=case["comps"], dtype=DTYPES[case["dtype"]], t0=0.0, tf=20.0) for n in ns]
        st["v"] = [_vectors(n, case["comps"], case["dtype"], seed, 10 + i) for i, n in enumerate(ns)]
        st["out"] = [torch.zeros_like(v) for v in st["v"]]
    elif kind == "newton":
        n = case["n"]
        rf, tf = case["rf"], _uniform(TF_RANGE, seed, 3)
        p = api.Problem(_lib.BK_ORBIT, n, DTYPES[case["dtype"]], 0.0, tf, (THRUST, rf))
        X, U = _spiral(0.5 * tf * (_tau(n) + 1.0), rf, tf)
        st.update(prob=p, z0=p.pack(X, U), ws=api.newton_workspace(p))
        st["z"] = torch.zeros_like(st["z0"])
    else:
        code, tf, params, X, U, lam, nu = _point(case, seed)
        p = api.Problem(code, case["n"], DTYPES[case["dtype"]], 0.0, tf, params)
        p.linearize(p.pack(X, U, lam, nu))
        st.update(prob=p, x=_kkt_input(case, seed, p.n_x, p.n_u, p.n_e))
        st["out"] = torch.zeros_like(st["x"])
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "apply":
        f = api.birkhoff_apply_T if case["trans"] else api.birkhoff_apply
        return f(state["plan"], state["v"], state["out"])
    if kind == "batch":
        return api.birkhoff_apply_batch(state["plans"], state["v"], state["out"], trans=case["trans"])
    if kind == "kkt":
        return api.kkt_apply(state["prob"], _lib.BK_OP_KKT, state["x"], state["out"])
    if kind == "precond":
        return api.precond_apply(state["prob"], _lib.BK_OP_KKT, state["x"], state["out"])
    state["z"].copy_(state["z0"])
    api.newton_solve(state["prob"], state["z"], workspace=state["ws"])
    return state["z"]


# --- algorithmic work ---------------------------------------------------------------------------
def _product_flops(n, nvec):
    """Two real-even transforms of length n + 1 per vector, 2.5 n log2 n operations each."""
    return nvec * 2 * 2.5 * n * math.log2(n)


def work(case):
    kind = case["kind"]
    es = 8 if case["dtype"] == "f64" else 4
    if kind == "apply":
        n, c = case["n"], case["comps"]
        return dict(bytes=2 * c * (n + 1) * es, flops=_product_flops(n, c))
    if kind == "batch":
        ns = [1 << k for k in range(case["klo"], case["khi"] + 1)]
        c = case["comps"]
        return dict(bytes=sum(2 * c * (n + 1) * es for n in ns), flops=sum(_product_flops(n, c) for n in ns))
    n = case["n"]
    nx, nu = (2, 1) if case.get("problem") == "dblint" else (4, 2)
    vec = (2 * nx + nu) * (n + 1) * es
    point = (2 * nx + nu + 1) * (n + 1) * es     # states, controls, s B^T lambda and weights per node
    if kind == "kkt":
        # two products of nx vectors, and the Jacobian and Hessian products of a node
        return dict(bytes=2 * vec + point, flops=2 * _product_flops(n, nx) + (n + 1) * 2 * (nx + nu) ** 2 * 2)
    if kind == "precond":
        # a backward and a forward sweep: one nx x nx matrix per node each, read once; the terminal columns
        return dict(bytes=2 * vec + point + nx * nx * (n + 1) * es, flops=(n + 1) * (2 * 2 * nx * nx + 8 * nx * 3))
    # the guess read and the solution written; five Newton steps, eleven Krylov steps of one operator and one
    # preconditioner apply each, one residual per Newton step
    prod = 2 * _product_flops(n, nx)
    return dict(bytes=2 * (2 * nx + nu) * (n + 1) * 8, flops=11 * (prod + (n + 1) * 300) + 5 * prod)


# --- the same results in 64 bits ------------------------------------------------------------------
def _b(v, s):
    """B v along the last axis (length n + 1): the integral from the first node of the polynomial through v."""
    n = v.shape[-1] - 1
    sgn = torch.ones(n + 1, dtype=torch.float64, device=v.device)
    sgn[1::2] = -1.0
    half = torch.ones(n + 1, dtype=torch.float64, device=v.device)
    half[0] = half[-1] = 0.5

    def cosines(x):   # sum_m half_m x_m cos(pi k m / n) for k = 0 .. n
        x = x * half
        ext = torch.cat([2 * x[..., :1], x[..., 1:n], 2 * x[..., n:], x[..., 1:n].flip(-1)], -1)
        return 0.5 * torch.fft.rfft(ext).real

    a = cosines(v) * sgn * half * (2.0 / n)     # Chebyshev coefficients (nodes run from -1 to 1)
    k = torch.arange(1, n + 2, dtype=torch.float64, device=v.device)
    lower = torch.cat([2 * a[..., :1], a[..., 1:]], -1)                       # a_{k-1}, k = 1 .. n + 1
    upper = torch.cat([a[..., 2:], torch.zeros_like(a[..., :2])], -1)         # a_{k+1}, k = 1 .. n + 1
    c = (lower - upper) / (2 * k)
    # values at the nodes: T_k(tau_j) = (-1)^k cos(pi k j / n); T_{n+1} equals T_{n-1} there
    c = torch.cat([c[..., :n - 2], c[..., n - 2:n - 1] + c[..., n:], c[..., n - 1:n]], -1)
    y = cosines(torch.cat([torch.zeros_like(c[..., :1]), c], -1) * sgn / half)
    return s * (y - y[..., :1])


def _bt(u, s):
    """B^T u: the gradient of u . (B v) in v."""
    v = torch.zeros_like(u, requires_grad=True)
    return torch.autograd.grad((_b(v, s) * u).sum(), v)[0]


def _f(problem, X, U):
    if problem == "dblint":
        return torch.stack([X[1], U[0]])
    r, vr, vt = X[0], X[2], X[3]
    return torch.stack([vr, vt / r, vt * vt / r - 1 / (r * r) + U[0], -vr * vt / r + U[1]])


def _jx(problem, X):
    """State Jacobians per node, [L, nx, nx]."""
    L = X.shape[1]
    if problem == "dblint":
        J = torch.zeros(L, 2, 2, dtype=torch.float64, device=X.device)
        J[:, 0, 1] = 1
        return J
    r, vr, vt = X[0], X[2], X[3]
    J = torch.zeros(L, 4, 4, dtype=torch.float64, device=X.device)
    J[:, 0, 2] = 1
    J[:, 1, 0], J[:, 1, 3] = -vt / r**2, 1 / r
    J[:, 2, 0], J[:, 2, 3] = -vt**2 / r**2 + 2 / r**3, 2 * vt / r
    J[:, 3, 0], J[:, 3, 2], J[:, 3, 3] = vr * vt / r**2, -vt / r, -vr / r
    return J


def _terminal(problem):
    return (0, 1) if problem == "dblint" else (0, 2, 3)


def _split(z, nx, nu, ne, P, L):
    X = z[:nx * P].view(nx, P)[:, :L]
    U = z[nx * P:(nx + nu) * P].view(nu, P)[:, :L]
    lam = z[(nx + nu) * P:(2 * nx + nu) * P].view(nx, P)[:, :L]
    k = (2 * nx + nu) * P
    return X, U, lam, z[k:k + ne]


def _join(X, U, lam, nu, P):
    nx, L = X.shape
    z = torch.zeros((2 * nx + U.shape[0]) * P + 32, dtype=torch.float64, device=X.device)
    a, b, c, d = _split(z, nx, U.shape[0], nu.numel(), P, L)
    a.copy_(X)
    b.copy_(U)
    c.copy_(lam)
    d.copy_(nu)
    return z


def _exact_kkt(case, seed):
    """Derivative of the gradient of the Lagrangian s w . |u|^2 / 2 + lambda . (X - s B f) + nu . x(t_f)."""
    problem, n = case["problem"], case["n"]
    code, tf, params, X, U, lam, nu = _point(case, seed)
    if case["dtype"] == "f32":   # the operator keeps its linearisation point in its own precision
        X, U = X.float().double(), U.float().double()
    s, P, L = 0.5 * tf, _pitch(n), n + 1
    nx, nu_, ne = X.shape[0], U.shape[0], nu.numel()
    d = _split(_kkt_input(case, seed, nx, nu_, ne).double(), nx, nu_, ne, P, L)
    e = torch.zeros(1, L, dtype=torch.float64, device="cuda")
    e[0, -1] = 1.0
    w = _bt(e, 1.0)[0]
    idx = list(_terminal(problem))

    def lagrangian(X, U, lam, nu):
        return 0.5 * s * (w * U * U).sum() + (lam * (X - _b(_f(problem, X, U), s))).sum() + (nu * X[idx, -1]).sum()

    at = [t.clone().requires_grad_(True) for t in (X, U, lam, nu)]
    g = torch.autograd.grad(lagrangian(*at), at, create_graph=True)
    h = torch.autograd.grad(sum((a * b).sum() for a, b in zip(g, d)), at)   # the Hessian is symmetric
    return _join(*h, P)


def _scan(M, f):
    """States before each step of y <- M_k y + f_k from zero (M [L, nx, nx], f [L, nx, m]), by doubling."""
    L = M.shape[0]
    A, b = M.clone(), f.clone()
    d = 1
    while d < L:
        b = torch.cat([b[:d], b[d:] + A[d:] @ b[:-d]])
        A = torch.cat([A[:d], A[d:] @ A[:-d]])
        d *= 2
    return torch.cat([torch.zeros_like(b[:1]), b[:-1]])


def _exact_precond(case, seed):
    """K-tilde^{-1} r: the KKT matrix with the trapezoidal-like B-tilde in the constraint and the control cost only."""
    problem, n = case["problem"], case["n"]
    code, tf, params, X, U, lam, nu = _point(case, seed)
    if case["dtype"] == "f32":
        X, U = X.float().double(), U.float().double()
    s, P, L = 0.5 * tf, _pitch(n), n + 1
    nx, nu_, ne = X.shape[0], U.shape[0], nu.numel()
    rx, ru, rl, rn = _split(_kkt_input(case, seed, nx, nu_, ne).double(), nx, nu_, ne, P, L)
    e = torch.zeros(1, L, dtype=torch.float64, device="cuda")
    e[0, -1] = 1.0
    w = _bt(e, 1.0)[0]
    h = (0.5 * s * w)[:, None, None]
    J = _jx(problem, X)
    eye = torch.eye(nx, dtype=torch.float64, device="cuda")
    K = torch.linalg.inv(eye - h * J)
    D = h * (J @ K)
    Ju = torch.zeros(nx, nu_, dtype=torch.float64, device="cuda")
    for q in range(nu_):
        Ju[nx - nu_ + q, q] = 1.0
    idx = list(_terminal(problem))

    def fwd(Y):      # P xi = Y, Y [L, nx, m]
        return K @ (Y + _scan(eye + 2 * D, 2 * (D @ Y)))

    def bwd(R):      # P^T y = R and B-tilde^T y
        Kt, Dt = K.transpose(1, 2), D.transpose(1, 2)
        rho = _scan((eye + 2 * Dt).flip(0), (Kt @ R).flip(0)).flip(0)
        y = Kt @ R + 2 * (Dt @ rho)
        return y, w[:, None, None] * (0.5 * y + rho)

    def btilde(g):   # running sum with half weight at the node itself
        t = w[:, None, None] * g
        return torch.cumsum(t, 0) - 0.5 * t

    R = torch.zeros(L, nx, 1 + ne, dtype=torch.float64, device="cuda")
    R[:, :, 0] = rx.T
    for r, i in enumerate(idx):
        R[-1, i, 1 + r] = 1.0
    y, b = bwd(R)
    # controls: (s w) yu = r_u + s Ju^T B-tilde^T y (first column), minus that for the terminal columns
    yu = (s * (Ju.T @ b))
    yu[:, :, 0] += ru.T
    yu = yu / (s * w)[:, None, None]
    Y = s * btilde(Ju @ yu)
    Y[:, :, 0] += rl.T
    xi = fwd(Y)
    x0, Q = xi[:, :, 0], -xi[:, :, 1:]
    S = Q[-1, idx, :]
    m = torch.linalg.solve(-S, x0[-1, idx] - rn)
    return _join((x0 + Q @ m).T, (yu[:, :, 0] - yu[:, :, 1:] @ m).T, (y[:, :, 0] - y[:, :, 1:] @ m).T, m, P)


def exact(case, seed):
    kind = case["kind"]
    if kind == "apply":
        return _product(_vectors(case["n"], case["comps"], case["dtype"], seed), case["n"], case["trans"])
    if kind == "batch":
        return [_product(_vectors(1 << k, case["comps"], case["dtype"], seed, 10 + i), 1 << k, case["trans"])
                for i, k in enumerate(range(case["klo"], case["khi"] + 1))]
    if kind == "kkt":
        return _exact_kkt(case, seed)
    if kind == "precond":
        return _exact_precond(case, seed)
    return None   # a nonlinear solve: no closed form, and a second solver at these sizes takes minutes


def _product(v, n, trans):
    out = torch.zeros(v.shape, dtype=torch.float64, device=v.device)
    x = v[:, :, :n + 1].double()
    out[:, :, :n + 1] = _bt(x, 10.0) if trans else _b(x, 10.0)
    return out
