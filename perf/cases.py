"""Performance cases: the work a user of this library has it do, through its public entry points.

Every case is a dict with a ``family`` and its sizes:

* ``solve``    Mesh.pcg_solve from zero, all right-hand sides of a batch of independent box problems (the whole call);
* ``apply``    Mesh.apply_operator, the operator a user's own Krylov method or time loop calls;
* ``edge``     the same on a batch of edge neighbourhoods of uneven degree (graded geometric meshes, corner sets);
* ``precond``  Mesh.apply_preconditioner, element blocks or the separable form;
* ``residual`` autograd.ResidualMap, forward and backward, on a batch of problems of uneven degree;
* ``gradient`` autograd.Solve and its backward: the data gradient of a solution functional;
* ``setup``    new coefficients on a mesh: set_data, the element-block preconditioner, one application of it.

``exact`` restates the method in plain 64-bit torch (Gauss-Lobatto-Legendre rules, the weighted residual on the
(2W+1)-point grid, the face forms on the nodal face grid, preconditioned CG to the attainable level).
"""
from __future__ import annotations

import math
from functools import lru_cache
from types import SimpleNamespace

import numpy as np
import torch
from numpy.polynomial import legendre as npleg

from paper_1110_2316_gb300 import api
from paper_1110_2316_gb300 import autograd as ag

DEV = "cuda"
F64 = torch.float64
PREC = {"f64": (api.FP64, torch.float64), "f32": (api.FP32, torch.float32)}
KIND = {"laplace": api.COEF_LAPLACE, "scalar": api.COEF_SCALAR, "general": api.COEF_GENERAL}


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # one small Poisson problem to 1e-10 in FP64 with the default preconditioner: the smallest solve, bound by
        # latency and launches
        dict(name="solve_poisson_small", family="solve", kind="laplace", nx=2, ny=2, nz=2, W=4, rhs=1, problems=1,
             prec="f64", pre="separable"),
        # a parameter study: many independent small problems in one mixed-precision solve, default preconditioner
        dict(name="solve_poisson_batch", family="solve", kind="laplace", nx=2, ny=2, nz=2, W=4, rhs=1, problems=1024,
             prec="f32", pre="separable"),
        # the ordinary production solve: variable coefficient, many right-hand sides, element blocks, FP32 applies
        # with FP64 refinement
        dict(name="solve_varcoef", family="solve", kind="scalar", nx=8, ny=8, nz=8, W=8, rhs=16, problems=1,
             prec="f32", pre="block"),
        # operator applies: the largest batch of the benchmark in FP32 ...
        dict(name="apply_varcoef_f32", family="apply", kind="scalar", nx=8, ny=8, nz=8, W=8, rhs=64, prec="f32"),
        # ... a few right-hand sides in FP64 (the refinement residual, FP64 solves) ...
        dict(name="apply_varcoef_f64", family="apply", kind="scalar", nx=8, ny=8, nz=8, W=8, rhs=4, prec="f64"),
        # ... the general non-self-adjoint operator with mixed derivatives and Neumann faces ...
        dict(name="apply_general_f32", family="apply", kind="general", nx=8, ny=8, nz=8, W=8, rhs=16, prec="f32"),
        # ... and a batch of edge neighbourhoods of degree 2 to 8 (low degrees, small elements, several launches)
        dict(name="apply_edge_f32", family="edge", wmin=2, wmax=8, copies=146, prec="f32"),
        # the element-block preconditioner inside a many-right-hand-side solve, and on a few right-hand sides
        dict(name="precond_block_f32", family="precond", pre="block", nx=8, ny=8, nz=8, W=8, rhs=64, prec="f32"),
        dict(name="precond_block_few", family="precond", pre="block", nx=8, ny=8, nz=8, W=8, rhs=4, prec="f32"),
        # training-style use: residual map forward and backward over a batch of uneven degrees
        dict(name="residual_f64", family="residual", wmin=4, wmax=10, problems=8, n=4, prec="f64"),
        # the data gradient of a solution functional (forward solve, adjoint solve, pointwise gradients)
        dict(name="gradient_f64", family="gradient", wmin=4, wmax=6, problems=8, n=3),
        # a new coefficient field: data, right-hand side, element blocks, one preconditioner application
        dict(name="setup_block", family="setup", nx=4, ny=4, nz=4, W=8, rhs=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))


def _boxes(rng, hi):
    return {k: rng.randint(1, hi) for k in ("nx", "ny", "nz")}


def _dofs(c):
    return c["nx"] * c["ny"] * c["nz"] * (c["W"] + 1) ** 3


def draw(rng):
    while True:
        fam = rng.choice(["solve", "solve", "apply", "apply", "apply", "edge", "precond", "precond", "residual",
                          "gradient", "setup"])
        if fam == "solve":
            kind = rng.choice(["laplace", "scalar"])
            c = dict(family=fam, kind=kind, **_boxes(rng, 3 if kind == "laplace" else 6),
                     W=rng.randint(2, 6 if kind == "laplace" else 8),
                     rhs=_log(rng, 1, 4 if kind == "laplace" else 16),
                     problems=_log(rng, 1, 512) if kind == "laplace" else 1, prec=rng.choice(["f64", "f32"]),
                     pre="separable" if kind == "laplace" else "block")
            if _dofs(c) * c["rhs"] * c["problems"] > (1_500_000 if c["prec"] == "f32" else 60_000):
                continue
        elif fam == "apply":
            kind, prec = rng.choice(["laplace", "scalar", "general"]), rng.choice(["f64", "f32"])
            c = dict(family=fam, kind=kind, **_boxes(rng, 8), W=rng.randint(1, 9 if kind == "general" else 10),
                     rhs=_log(rng, 1, 96), prec=prec)
            most = {"f32": 20_000_000, "f64": 1_500_000}[prec] // (4 if kind == "general" else 1)
            if _dofs(c) * c["rhs"] > most:
                continue
        elif fam == "edge":
            lo, hi = sorted((rng.randint(2, 8), rng.randint(2, 8)))
            c = dict(family=fam, wmin=lo, wmax=hi, copies=_log(rng, 1, 146), prec=rng.choice(["f64", "f32"]))
        elif fam == "precond":
            c = dict(family=fam, pre=rng.choice(["block", "block", "separable"]), **_boxes(rng, 8),
                     W=rng.randint(2, 10), rhs=_log(rng, 1, 80), prec=rng.choice(["f64", "f32"]))
            n = (c["W"] + 1) ** 3
            if _dofs(c) * n > 2.5e8 or _dofs(c) * n * c["rhs"] > (1.6e10 if c["prec"] == "f32" else 1.5e9):
                continue
        elif fam == "residual":
            lo, hi = sorted((rng.randint(2, 10), rng.randint(2, 10)))
            c = dict(family=fam, wmin=lo, wmax=hi, problems=_log(rng, 1, 8), n=rng.randint(1, 4),
                     prec=rng.choice(["f64", "f32"]))
        elif fam == "gradient":
            lo, hi = sorted((rng.randint(2, 6), rng.randint(2, 6)))
            c = dict(family=fam, wmin=lo, wmax=hi, problems=_log(rng, 1, 8), n=rng.randint(1, 3))
        else:
            c = dict(family=fam, **_boxes(rng, 5), W=rng.randint(2, 8), rhs=_log(rng, 1, 40))
            if _dofs(c) * (c["W"] + 1) ** 3 > 3.0e7:
                continue
        return c


# ---------------------------------------------------------------------------
# meshes
# ---------------------------------------------------------------------------
def _box_desc(nx, ny, nz, Ws, lo=0.0, hi=1.0):
    """len(Ws) independent problems on nx x ny x nz boxes of [lo, hi]^3, degree Ws[p] in problem p."""
    E = nx * ny * nz
    idx = np.stack(np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij"), -1).reshape(E, 3)[:, ::-1]
    n3, step = np.array([nx, ny, nz]), np.array([1, nx, nx * ny])
    cuts = [np.linspace(lo, hi, m + 1) for m in n3]
    elo = np.stack([cuts[a][idx[:, a]] for a in range(3)], 1)
    ehi = np.stack([cuts[a][idx[:, a] + 1] for a in range(3)], 1)
    nbr = np.full((E, 6), -1, dtype=np.int64)
    for a in range(3):
        m = idx[:, a] > 0
        nbr[m, 2 * a] = np.nonzero(m)[0] - step[a]
        m = idx[:, a] < n3[a] - 1
        nbr[m, 2 * a + 1] = np.nonzero(m)[0] + step[a]
    K = len(Ws)
    allnbr = np.where(nbr[None] >= 0, nbr[None] + (np.arange(K) * E)[:, None, None], -1).reshape(-1, 6)
    return SimpleNamespace(elem_lo=np.tile(elo, (K, 1)), elem_hi=np.tile(ehi, (K, 1)),
                           elem_W=np.repeat(np.asarray(Ws, dtype=np.int32), E), elem_nbr=allnbr.astype(np.int32),
                           elem_problem=np.repeat(np.arange(K, dtype=np.int32), E), n_problem=K)


def _edge_desc(Ws, mu=0.15):
    """Independent edge neighbourhoods 0 < r < 1, 0 < theta < pi/2, 0 < x3 < 1: 2 W + 4 layers graded by mu toward the
    edge, one corner set each, boxes in (ln r, theta, x3)."""
    lo, hi, W, nbr, prob, off = [], [], [], [], [], 0
    for p, w in enumerate(Ws):
        N = 2 * w + 4
        t = np.log(mu ** np.arange(N, -1, -1.0))
        one = np.ones(N)
        lo.append(np.stack([t[:-1], 0 * one, 0 * one], 1))
        hi.append(np.stack([t[1:], 0.5 * np.pi * one, one], 1))
        nb = np.full((N, 6), -1, dtype=np.int64)
        nb[1:, 0] = off + np.arange(N - 1)
        nb[0, 0] = -2 - p
        nb[:-1, 1] = off + 1 + np.arange(N - 1)
        nbr.append(nb)
        W.append(np.full(N, w))
        prob.append(np.full(N, p))
        off += N
    cat = np.concatenate
    K = len(Ws)
    return SimpleNamespace(elem_lo=cat(lo), elem_hi=cat(hi), elem_W=cat(W).astype(np.int32),
                           elem_nbr=cat(nbr).astype(np.int32), elem_problem=cat(prob).astype(np.int32),
                           corner_W=np.asarray(Ws, dtype=np.int32), corner_lo=np.zeros(K), corner_hi=np.ones(K),
                           corner_problem=np.arange(K, dtype=np.int32), n_problem=K, kind="edge")


def _degrees(c):
    """Degrees cycling through wmin..wmax over the problems."""
    return [c["wmin"] + p % (c["wmax"] - c["wmin"] + 1) for p in range(c["problems"])]


def _desc(c):
    if c["family"] == "edge":
        return _edge_desc([w for w in range(c["wmin"], c["wmax"] + 1) for _ in range(c["copies"])])
    if c["family"] in ("residual", "gradient"):
        return _box_desc(c["n"], c["n"], c["n"], _degrees(c))
    general = c.get("kind") == "general"
    d = _box_desc(c["nx"], c["ny"], c["nz"], [c["W"]] * c.get("problems", 1), -1.0 if general else 0.0, 1.0)
    if general:  # Dirichlet on x = +-1 and y = -1, Neumann on y = 1 and z = +-1
        bc = np.zeros_like(d.elem_nbr)
        bc[:, 3:] = d.elem_nbr[:, 3:] == -1
        d.elem_bc = bc
    return d


def _kind(c):
    return {"edge": "laplace"}.get(c["family"], c.get("kind", "scalar"))


# ---------------------------------------------------------------------------
# data at the volume points (made on the GPU from the seed alone)
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, dtype=F64, device=DEV)


def _uniform(g, lo, hi):
    return float(torch.rand(1, generator=g, dtype=F64, device=DEV)) * (hi - lo) + lo


def _legendre(t, K):
    """L_0..L_K at t, last axis K + 1."""
    p = [torch.ones_like(t), t]
    for m in range(1, K):
        p.append(((2 * m + 1) * t * p[m] - m * p[m - 1]) / (m + 1))
    return torch.stack(p[: K + 1], -1)


def _groups(desc):
    """Runs of consecutive elements of one degree: (degree, first element, end)."""
    W = np.asarray(desc.elem_W)
    cut = [0] + [int(i) + 1 for i in np.nonzero(np.diff(W))[0]] + [len(W)]
    return [(int(W[b]), b, e) for b, e in zip(cut[:-1], cut[1:])]


def _points(desc, b, e, W):
    """The coordinates of the (2W+1)-point rules of elements b..e: three [E, Q] tensors."""
    xq = torch.tensor(_gll(2 * W + 1)[0], dtype=F64, device=DEV)
    lo = torch.tensor(desc.elem_lo[b:e], dtype=F64, device=DEV)
    hi = torch.tensor(desc.elem_hi[b:e], dtype=F64, device=DEV)
    return [lo[:, a, None] + 0.5 * (xq + 1) * (hi - lo)[:, a, None] for a in range(3)]


def _make_data(c, desc, seed):
    """f [R, nq] (Legendre coefficients N(0, 1) decaying as 2^-k, other ones in each problem), a and grad a
    (a = 1 + amp sin sin sin) or the ten general coefficients, as set_data takes them."""
    g = _gen(seed)
    R, K = c.get("rhs", 1), 5
    kind = _kind(c)
    coef = _randn(g, R, desc.n_problem, K + 1, K + 1, K + 1)
    d = 2.0 ** -torch.arange(K + 1, dtype=F64, device=DEV)
    coef = coef * d[:, None, None] * d[:, None] * d
    amp, ph = _uniform(g, 0.3, 0.6), [_uniform(g, 0.0, 1.0) for _ in range(3)]
    lo, hi = torch.tensor(desc.elem_lo.min(0), dtype=F64), torch.tensor(desc.elem_hi.max(0), dtype=F64)
    fs, As, Gs, ops = [], [], [], []
    prob = torch.tensor(desc.elem_problem, dtype=torch.int64, device=DEV)
    for W, b, e in _groups(desc):
        X = _points(desc, b, e, W)
        L = [_legendre(2 * (X[a] - lo[a].item()) / (hi[a] - lo[a]).item() - 1, K) for a in range(3)]
        if desc.n_problem == 1:
            t = torch.einsum("rijk,eai->reajk", coef[:, 0], L[0])
        else:
            t = torch.einsum("reijk,eai->reajk", coef[:, prob[b:e]], L[0])
        t = torch.einsum("reajk,ebj->rebak", t, L[1])
        fs.append(torch.einsum("rebak,eck->recba", t, L[2]).reshape(R, -1))
        x, y, z = X[0][:, None, None, :], X[1][:, None, :, None], X[2][:, :, None, None]
        if kind == "scalar":
            w = 2 * math.pi
            s = [torch.sin(w * v + p) for v, p in zip((x, y, z), ph)]
            k = [torch.cos(w * v + p) for v, p in zip((x, y, z), ph)]
            As.append((1 + amp * s[0] * s[1] * s[2]).reshape(-1))
            Gs.append(torch.stack([(amp * w * k[0] * s[1] * s[2]).reshape(-1),
                                   (amp * w * s[0] * k[1] * s[2]).reshape(-1),
                                   (amp * w * s[0] * s[1] * k[2]).reshape(-1)]))
        elif kind == "general":
            one = torch.ones_like(x * y * z)
            t = math.pi * (x + y + z)
            m = -0.001 * torch.sin(t) * 0.5
            v = [-(0.5 + 0.05 * torch.exp(x * y * z)) * (1 + amp), -(1 + 0.015 * torch.cos(x + y)) * one,
                 -(2.5 + 0.02 * torch.exp(y + z)) * one, m, m, m, 0.1 * amp * x * one, 0.2 * y * one, 0.3 * z * one,
                 4.05 + 0.045 * torch.cos(t / 2)]
            ops.append(torch.stack([u.reshape(-1) for u in v]))
    out = dict(f=torch.cat(fs, 1))
    if As:
        out.update(a=torch.cat(As), grad_a=torch.cat(Gs, 1).contiguous())
    if ops:
        out["op"] = torch.cat(ops, 1).contiguous()
    return out


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------
def prepare(case, seed):
    c, fam = case, case["family"]
    desc = _desc(c)
    data = _make_data(c, desc, seed)
    m = api.Mesh(desc, n_rhs=c.get("rhs", 1), coef_kind=KIND[_kind(c)])
    n = m.n_rhs * m.ndof
    g = _gen(seed + 7)
    s = SimpleNamespace(family=fam, mesh=m, case=c)
    prec, dtype = PREC[c.get("prec", "f64")]
    if fam in ("setup", "gradient"):
        s.data = data
        if fam == "gradient":
            m.set_data(**data)
            s.target = _make_data(c, desc, seed + 3)["f"]
            s.weights = torch.empty(m.nquad, dtype=F64, device=DEV)
            m.quad_weights(s.weights)
        else:
            s.r = _randn(g, n)
        return s
    m.set_data(**data)
    if c.get("pre") == "block":
        m.setup_block_preconditioner()
    if fam == "solve":
        s.prec = prec
    elif fam == "residual":
        s.u = _randn(g, n).to(dtype)
        s.gz = _randn(g, m.n_rhs, m.nquad).to(dtype)
    else:
        s.u = _randn(g, n).to(dtype)
    return s


def run(state):
    s, m = state, state.mesh
    if s.family == "solve":
        x = torch.empty(m.n_rhs * m.ndof, dtype=F64, device=DEV)
        m.pcg_solve(x, tol=1e-10, prec=s.prec)
        return x
    if s.family in ("apply", "edge"):
        y = torch.empty_like(s.u)
        m.apply_operator(s.u, y)
        return y
    if s.family == "precond":
        z = torch.empty_like(s.u)
        m.apply_preconditioner(s.u, z)
        return z
    if s.family == "residual":
        u = s.u.detach().requires_grad_(True)
        z = ag.ResidualMap.apply(u, m)
        z.backward(s.gz)
        return [z.detach(), u.grad]
    if s.family == "gradient":
        f, a, ga = (s.data[k].detach().requires_grad_(True) for k in ("f", "a", "grad_a"))
        u = ag.Solve.apply(f, a, ga, m, None, 1e-12, api.FP64, api.FP64, 1e-9)
        v = ag.PointValues.apply(u, m)
        (0.5 * s.weights * (v - s.target) ** 2).sum().backward()
        return [u.detach(), f.grad, a.grad, ga.grad]
    m.set_data(**s.data)
    m.setup_block_preconditioner()
    b, z = torch.empty_like(s.r), torch.empty_like(s.r)
    m.get_rhs(b)
    m.apply_preconditioner(s.r, z)
    return [b, z]


# ---------------------------------------------------------------------------
# work: bytes and operations that no implementation of the path can do without
# ---------------------------------------------------------------------------
def _apply_work(W, kind, nsol, nelem, size):
    """(flops, bytes) of one operator apply: the even-odd folded sum factorisation, forward and transposed, and the
    face forms, for nsol (element, rhs) items; coefficients of nelem elements read once."""
    P, Q = W + 1, 2 * W + 1
    n1, n2, n3 = {"laplace": (2, 3, 2), "scalar": (3, 5, 5), "general": (3, 6, 10)}[kind]
    vol = n1 * Q * P ** 3 + n2 * Q * Q * P * P + n3 * Q ** 3 * P
    nc = {"laplace": 0, "scalar": 4, "general": 11}[kind]
    return (2.0 * vol + 2.0 * 6 * 10 * P ** 3) * nsol, (2.0 * P ** 3 * nsol + nc * Q ** 3 * nelem) * size


def work(case):
    c, fam = case, case["family"]
    size = 4 if c.get("prec") == "f32" else 8
    if fam == "edge":
        fl = by = 0.0
        for w in range(c["wmin"], c["wmax"] + 1):
            n = c["copies"] * (2 * w + 4)
            a, b = _apply_work(w, "laplace", n, 0, size)
            fl, by = fl + a, by + b
        return {"bytes": by, "flops": fl}
    if fam in ("residual", "gradient"):
        fl = by = 0.0
        for w in _degrees(c):
            n, P, Q = c["n"] ** 3, w + 1, 2 * w + 1
            a, b = _apply_work(w, "scalar", n, n, size)
            if fam == "residual":  # u, z, the cotangent, y, coefficients and f once
                fl, by = fl + a, by + b + 3.0 * n * Q ** 3 * size
            else:  # two solves of some 12 W iterations, fields and gradients at the points
                fl, by = fl + 24 * w * a, by + b + 10.0 * n * Q ** 3 * 8
        return {"bytes": by, "flops": fl}
    E, n, R = c["nx"] * c["ny"] * c["nz"], (c["W"] + 1) ** 3, c["rhs"]
    if fam == "apply":
        fl, by = _apply_work(c["W"], c["kind"], E * R, E, size)
        return {"bytes": by, "flops": fl}
    if fam == "precond":
        if c["pre"] == "separable":
            return {"bytes": 2.0 * E * n * R * size, "flops": 12.0 * (c["W"] + 1) * n * E * R}
        return {"bytes": (n * (n + 1) / 2 * E + 2.0 * E * n * R) * size, "flops": 2.0 * n * n * E * R}
    if fam == "solve":
        its = (30 if c["kind"] == "laplace" else 60) * c["W"]
        fl, by = _apply_work(c["W"], c["kind"], E * R * c["problems"], E, size)
        pre = 12.0 * (c["W"] + 1) * n if c["pre"] == "separable" else 2.0 * n * n
        return {"bytes": by, "flops": its * (fl + pre * E * R * c["problems"])}
    # setup: the blocks' columns, factorisation and triangular inverse; the factor written once per precision
    fl, by = _apply_work(c["W"], "scalar", E * n, E, 8)
    return {"bytes": 12.0 * n * (n + 1) / 2 * E, "flops": 0.5 * fl + 2.0 / 3 * n ** 3 * E}


# ---------------------------------------------------------------------------
# the method in plain 64-bit torch
# ---------------------------------------------------------------------------
@lru_cache(maxsize=None)
def _gll(n):
    """Nodes and weights of the n-point Gauss-Lobatto-Legendre rule."""
    N = n - 1
    c = np.zeros(N + 1)
    c[N] = 1.0
    x = np.concatenate([[-1.0], np.sort(np.real(npleg.legroots(npleg.legder(c)))) if N > 1 else [], [1.0]])
    for _ in range(3):  # Newton on L_N'
        d1, d2 = npleg.legval(x[1:-1], npleg.legder(c)), npleg.legval(x[1:-1], npleg.legder(c, 2))
        x[1:-1] -= d1 / d2
    return x, 2.0 / (N * (N + 1) * npleg.legval(x, c) ** 2)


def _interp(xp, x):
    M = np.ones((len(x), len(xp)))
    for j in range(len(xp)):
        for m in range(len(xp)):
            if m != j:
                M[:, j] *= (x - xp[m]) / (xp[j] - xp[m])
    return M


def _diff(x):
    n = len(x)
    w = np.array([1.0 / np.prod([x[j] - x[m] for m in range(n) if m != j]) for j in range(n)])
    D = np.zeros((n, n))
    for i in range(n):
        for j in range(n):
            if i != j:
                D[i, j] = w[j] / w[i] / (x[i] - x[j])
        D[i, i] = -D[i].sum()
    return D


@lru_cache(maxsize=None)
def _tables(W):
    """Interpolation and derivative matrices to the (2W+1)-point grid, the nodal differentiation matrix, the nodal L2
    and H^{1/2} forms of a face line, the Q weights and the separable form's eigenbasis (GPU tensors)."""
    xp, wp = _gll(W + 1)
    xq, wq = _gll(2 * W + 1)
    D = _diff(xp)
    B0 = _interp(xp, xq)
    B1 = B0 @ D
    B2 = B1 @ D
    DQ = _diff(xq)
    dx = xq[:, None] - xq[None, :] + np.eye(len(xq))
    off = -np.outer(wq, wq) / dx ** 2 * 2.0
    np.fill_diagonal(off, 0.0)
    K = off - np.diag(off.sum(1)) + DQ.T @ np.diag(wq * wq) @ DQ
    D2 = D @ D
    E = (D2.T * wp) @ D2 + (D.T * wp) @ D
    ev, V = np.linalg.eigh(E / np.sqrt(np.outer(wp, wp)))
    t = dict(B=[B0, B1, B2], D=D, MP=(B0.T * wq) @ B0, KP=B0.T @ K @ B0, wq=wq, S=V / np.sqrt(wp)[:, None],
             mu=np.maximum(ev, 0.0))
    T = lambda v: torch.tensor(v, dtype=F64, device=DEV)  # noqa: E731
    return SimpleNamespace(**{k: [T(v) for v in vs] if isinstance(vs, list) else T(vs) for k, vs in t.items()})


class _Reference:
    """The least-squares normal operator of a mesh of runs of equal degree."""

    def __init__(self, c, desc, data):
        self.c, self.desc, self.R = c, desc, c.get("rhs", 1)
        self.kind, self.edge = _kind(c), c["family"] == "edge"
        T = lambda v, t=F64: torch.tensor(v, dtype=t, device=DEV)  # noqa: E731
        h = T(desc.elem_hi - desc.elem_lo)
        self.s, self.half, self.jac = 2.0 / h, h / 2, (h / 2).prod(1)
        self.nbr = T(desc.elem_nbr, torch.int64)
        bc = getattr(desc, "elem_bc", None)
        self.bc = T(bc, torch.int64) if bc is not None else torch.zeros_like(self.nbr)
        self.prob = T(desc.elem_problem, torch.int64)
        self.runs, o, oq = [], 0, 0
        for W, b, e in _groups(desc):
            n, q = (e - b) * (W + 1) ** 3, (e - b) * (2 * W + 1) ** 3
            self.runs.append(SimpleNamespace(W=W, b=b, e=e, o=o, n=n, oq=oq, q=q, t=_tables(W)))
            o, oq = o + n, oq + q
        self.nelem_dof, self.nquad = o, oq
        if self.edge:
            cw = np.asarray(desc.corner_W) + 1
            self.coff = np.concatenate([[0], np.cumsum(cw)]) + o
            o = int(self.coff[-1])
            self.hi_tau, self.lo_tau = T(desc.elem_hi[:, 0]), T(desc.elem_lo[:, 0])
        self.ndof = o
        for r in self.runs:
            r.terms = self._terms(r, data)
            E, wq = r.e - r.b, r.t.wq
            r.w = (wq[:, None, None] * wq[:, None] * wq) * self.jac[r.b:r.e, None, None, None]
            r.f = data["f"][:, r.oq:r.oq + r.q].reshape(self.R, E, *r.w.shape[1:]) if "f" in data else None

    def _terms(self, r, data):
        """((x, y, z derivative orders), coefficient [E, Q, Q, Q] or [E, 1, 1, 1]) of L."""
        E, Q = r.e - r.b, 2 * r.W + 1
        s = self.s[r.b:r.e]
        S = lambda v: v.reshape(E, 1, 1, 1)  # noqa: E731
        orders = [(2, 0, 0), (0, 2, 0), (0, 0, 2)]
        if self.kind == "laplace":
            k = [-S(s[:, a] ** 2) for a in range(3)]
            if self.edge:
                k[2] = k[2] * torch.exp(2 * _points(self.desc, r.b, r.e, r.W)[0])[:, None, None, :]
            return list(zip(orders, k))
        cut = lambda v: v[r.oq:r.oq + r.q].reshape(E, Q, Q, Q)  # noqa: E731
        first = [(1, 0, 0), (0, 1, 0), (0, 0, 1)]
        if self.kind == "scalar":
            a, g = cut(data["a"]), [cut(data["grad_a"][k]) for k in range(3)]
            return ([(orders[k], -a * S(s[:, k] ** 2)) for k in range(3)] +
                    [(first[k], -g[k] * S(s[:, k])) for k in range(3)])
        op = [cut(data["op"][k]) for k in range(10)]
        out = [(orders[k], op[k] * S(s[:, k] ** 2)) for k in range(3)]
        for k, (i, j, o) in enumerate([(0, 1, (1, 1, 0)), (1, 2, (0, 1, 1)), (0, 2, (1, 0, 1))]):
            out.append((o, 2 * op[3 + k] * S(s[:, i] * s[:, j])))
        out += [(first[k], op[6 + k] * S(s[:, k])) for k in range(3)]
        return out + [((0, 0, 0), op[9])]

    @staticmethod
    def L(r, u, terms=None):
        """L u at the (2W+1)^3 points; u [R, E, P, P, P] (z, y, x)."""
        B, X, Y, out = r.t.B, {}, {}, None
        for (mx, my, mz), k in terms or r.terms:
            if mx not in X:
                X[mx] = u @ B[mx].T
            if (mx, my) not in Y:
                Y[mx, my] = B[my] @ X[mx]
            v = k * torch.einsum("ck,rekba->recba", B[mz], Y[mx, my])
            out = v if out is None else out + v
        return out

    @staticmethod
    def LT(r, z):
        B, X, Y = r.t.B, {}, {}
        for (mx, my, mz), k in r.terms:
            v = torch.einsum("ck,recba->rekba", B[mz], k * z)
            Y[mx, my] = Y[mx, my] + v if (mx, my) in Y else v
        for (mx, my), v in Y.items():
            v = B[my].T @ v
            X[mx] = X[mx] + v if mx in X else v
        return sum(v @ B[mx] for mx, v in X.items())

    def _face_weights(self, r, axis, side):
        """Per element: the L2 weight of [u] and (L2, t1, t2) weights of the three derivative fields, the same of the
        Dirichlet terms, and the scales of the tangential derivatives there."""
        E = r.e - r.b
        one = torch.ones(E, dtype=F64, device=DEV)
        if not self.edge:
            k = torch.ones(E, 3, 3, dtype=F64, device=DEV)
            return one, k, one, k, torch.ones(E, 3, dtype=F64, device=DEV)
        t1, t2 = [a for a in range(3) if a != axis]
        hh = self.half[r.b:r.e]
        tau = self.lo_tau[r.b:r.e] if (axis, side) == (0, 0) else self.hi_tau[r.b:r.e]
        G = torch.exp(tau)
        cc = torch.stack([hh[:, t1] * hh[:, t2], hh[:, t2] * (G if t1 == 2 else 1), hh[:, t1] * (G if t2 == 2 else 1)],
                         1)
        if axis == 2:
            cc = cc * G[:, None]
        g2 = torch.stack([one, one, G * G], 1)
        l2 = hh[:, t1] * hh[:, t2]
        return l2 * (G if axis == 2 else one), cc[:, None] * g2[:, :, None], l2, cc[:, None] * g2[:, :, None], \
            self.s[r.b:r.e]

    def faces(self, r, u, sel, U=None, yc=None):
        """The face terms' rows of the elements sel of run r (u: their blocks; U: all blocks of the run, or None where
        the neighbours' traces are taken as zero; yc: corner sets' rows, added to)."""
        t, P = r.t, r.W + 1
        y = torch.zeros_like(u)
        D, MP, KP = t.D, t.MP, t.KP
        s = self.s[r.b:r.e][sel]
        col = lambda v: v[:, None, None]  # noqa: E731
        for axis in range(3):
            t1, t2 = [a for a in range(3) if a != axis]
            v, yv = u.movedim(4 - axis, 2), y.movedim(4 - axis, 2)
            for side in range(2):
                end = P - 1 if side else 0
                nb = self.nbr[r.b:r.e, 2 * axis + side][sel]
                neu = (self.bc[r.b:r.e, 2 * axis + side][sel] != 0) & (nb == -1)
                dirichlet, inner = (nb == -1) & ~neu, nb != -1
                w0, wk, d0, dk, ds = (x[sel] for x in self._face_weights(r, axis, side))
                F, N = v[:, :, end], torch.einsum("n,renab->reab", D[end], v)
                Fo, No, so = torch.zeros_like(F), torch.zeros_like(N), s.clone()
                if U is not None:
                    have = nb >= 0
                    if bool(have.any()):
                        loc = nb[have] - r.b
                        o = U[:, loc].movedim(4 - axis, 2)
                        far = 0 if side else P - 1
                        Fo[:, have] = o[:, :, far]
                        No[:, have] = torch.einsum("n,renab->reab", D[far], o)
                        so[have] = self.s[nb[have]]
                    if yc is not None and (axis, side) == (0, 0):
                        have = torch.nonzero(nb <= -2).flatten()
                        rows = torch.tensor(self.coff[(-2 - nb[have]).cpu().numpy()], device=DEV)[:, None] + \
                            torch.arange(P, device=DEV)
                        Fo[:, have] = self._corner[:, rows][..., None].expand(-1, -1, P, P)
                m = lambda k: col(k.to(F64))  # noqa: E731
                # jumps of u and of the derivatives along t1, t2 and the normal
                J = [m(~neu) * (F - Fo)]
                sc1, sc2 = torch.where(inner, s[:, t1], ds[:, t1]), torch.where(inner, s[:, t2], ds[:, t2])
                J.append(m(~neu) * (col(sc1) * (F @ D.T) - col(so[:, t1]) * (Fo @ D.T)))
                J.append(m(~neu) * (col(sc2) * (D @ F) - col(so[:, t2]) * (D @ Fo)))
                sn = torch.where(inner, s[:, axis], torch.where(neu, s[:, axis] * (1 if side else -1), 0 * d0))
                J.append(col(sn) * N - m(inner) * col(so[:, axis]) * No)
                G = [col(torch.where(dirichlet, d0, w0)) * (MP @ J[0] @ MP)]
                for k, a in ((1, t1), (2, t2), (3, axis)):
                    w = torch.where(dirichlet[:, None], dk[:, a], wk[:, a])
                    A, Bk = J[k] @ MP, J[k] @ KP
                    G.append(col(w[:, 0]) * (MP @ A) + col(w[:, 1]) * (MP @ Bk) + col(w[:, 2]) * (KP @ A))
                yv[:, :, end] += G[0] + col(sc1) * (G[1] @ D) + col(sc2) * (D.T @ G[2])
                yv += D[end][None, None, :, None, None] * (col(sn) * G[3])[:, :, None]
                if U is not None and yc is not None and (axis, side) == (0, 0) and len(have):
                    back = -(G[0][:, have].sum(-1) + s[have, t2][None, :, None] *
                             torch.einsum("mk,rem->rek", D, G[2][:, have].sum(-1)))
                    yc.index_add_(1, rows.flatten(), back.reshape(back.shape[0], -1))
        return y

    def apply(self, u):
        """A u for u [R, ndof] (right-hand sides in pieces that fit)."""
        big = max((r.e - r.b) * (2 * r.W + 1) ** 3 for r in self.runs)
        step = max(1, int(1.5e8 // big))
        return torch.cat([self._apply(u[i:i + step]) for i in range(0, u.shape[0], step)])

    def _apply(self, u):
        y = torch.zeros_like(u)
        if self.edge:
            self._corner = u
        for r in self.runs:
            P = r.W + 1
            b = u[:, r.o:r.o + r.n].reshape(u.shape[0], -1, P, P, P)
            v = self.LT(r, r.w * self.L(r, b))
            sel = torch.arange(r.e - r.b, device=DEV)
            v = v + self.faces(r, b, sel, b, y if self.edge else None)
            y[:, r.o:r.o + r.n] = v.reshape(u.shape[0], -1)
        return y

    def rhs(self):
        """b for the sampled f and homogeneous boundary data."""
        return torch.cat([self.LT(r, r.w * r.f).reshape(self.R, -1) for r in self.runs], 1)

    def blocks(self):
        """The element's own blocks A_ee, per run [E, n, n]."""
        out = []
        for r in self.runs:
            P, E = r.W + 1, r.e - r.b
            n = P ** 3
            eye = torch.eye(n, dtype=F64, device=DEV).reshape(n, 1, P, P, P)
            step = max(1, int(1.0e8 // (n * (2 * r.W + 1) ** 3)))
            got = torch.empty(E, n, n, dtype=F64, device=DEV)
            for i in range(0, E, step):
                sel = torch.arange(i, min(E, i + step), device=DEV)
                u = eye.expand(n, len(sel), P, P, P)
                part = SimpleNamespace(t=r.t, terms=[(o, k[sel]) for o, k in r.terms])
                v = self.LT(part, r.w[sel] * self.L(part, u)) + self.faces(r, u, sel)
                got[sel] = v.reshape(n, len(sel), n).permute(1, 0, 2)
            out.append(got)
        return out

    def block_solve(self, chol, v):
        y = torch.empty_like(v)
        for r, k in zip(self.runs, chol):
            P = r.W + 1
            b = v[:, r.o:r.o + r.n].reshape(v.shape[0], -1, P ** 3).permute(1, 2, 0)
            y[:, r.o:r.o + r.n] = torch.cholesky_solve(b, k).permute(2, 0, 1).reshape(v.shape[0], -1)
        return y

    def separable(self, v):
        y = torch.empty_like(v)
        for r in self.runs:
            P, t = r.W + 1, r.t
            b = v[:, r.o:r.o + r.n].reshape(v.shape[0], -1, P, P, P)
            b = torch.einsum("kc,jb,ia,rekji->recba", t.S, t.S, t.S, b)
            b = b / (t.mu[:, None, None] + t.mu[:, None] + t.mu + 1)
            y[:, r.o:r.o + r.n] = torch.einsum("kc,jb,ia,recba->rekji", t.S, t.S, t.S, b).reshape(v.shape[0], -1)
        return y

    def solve(self, b):
        """A x = b by CG with the inverted element blocks, restarted on the true residual until that stops falling."""
        inv = [torch.cholesky_inverse(torch.linalg.cholesky(k)) for k in self.blocks()]
        dofprob = torch.cat([self.prob[r.b:r.e].repeat_interleave((r.W + 1) ** 3) for r in self.runs])
        n = self.desc.n_problem

        def pre(v):
            y = torch.empty_like(v)
            for r, k in zip(self.runs, inv):
                w = v[:, r.o:r.o + r.n].reshape(v.shape[0], r.e - r.b, -1).permute(1, 2, 0)
                y[:, r.o:r.o + r.n] = (k @ w).permute(2, 0, 1).reshape(v.shape[0], -1)
            return y

        def dot(p, q):
            return torch.zeros(p.shape[0], n, dtype=F64, device=DEV).index_add_(1, dofprob, p * q)

        spread = lambda k: k[:, dofprob]  # noqa: E731
        x, bb = torch.zeros_like(b), dot(b, b)
        best = math.inf
        for sweep in range(4):
            r = b - self.apply(x)
            level = float((dot(r, r) / bb).max().sqrt())
            if level < 1e-14 or level > 0.3 * best:
                break
            best, d = level, torch.zeros_like(x)
            z = pre(r)
            p, rz, r0 = z, dot(r, z), dot(r, r)
            for it in range(4000):
                q = self.apply(p)
                al = rz / dot(p, q).clamp_min(1e-300)
                d += spread(al) * p
                r = r - spread(al) * q
                if it % 10 == 9 and float((dot(r, r) / r0).max()) < 1e-24 * max(1.0, 1e-22 / level ** 2):
                    break
                z = pre(r)
                new = dot(r, z)
                p = z + spread(new / rz.clamp_min(1e-300)) * p
                rz = new
            x = x + d
        return x


def exact(case, seed):
    c, fam = case, case["family"]
    if fam == "solve" and _dofs(c) * c["rhs"] * c["problems"] * c["W"] > 8_000_000:
        return None  # minutes of CG in 64 bits
    desc = _desc(c)
    data = _make_data(c, desc, seed)
    ref = _Reference(c, desc, data)
    R, n = ref.R, ref.R * ref.ndof
    g = _gen(seed + 7)
    dtype = PREC[c.get("prec", "f64")][1]
    if fam == "solve":
        return ref.solve(ref.rhs()).reshape(-1)
    if fam in ("apply", "edge"):
        u = _randn(g, n).to(dtype).double().reshape(R, -1)
        return ref.apply(u).reshape(-1)
    if fam == "precond":
        u = _randn(g, n).to(dtype).double().reshape(R, -1)
        if c["pre"] == "separable":
            return ref.separable(u).reshape(-1)
        return ref.block_solve([torch.linalg.cholesky(k) for k in ref.blocks()], u).reshape(-1)
    if fam == "setup":
        r = _randn(g, n).reshape(R, -1)
        z = ref.block_solve([torch.linalg.cholesky(k) for k in ref.blocks()], r)
        return [ref.rhs().reshape(-1), z.reshape(-1)]
    if fam == "residual":
        u = _randn(g, n).to(dtype).double().reshape(R, -1)
        gz = _randn(g, R, ref.nquad).to(dtype).double()
        z, y = [], []
        for r in ref.runs:
            P, Q = r.W + 1, 2 * r.W + 1
            v = ref.L(r, u[:, r.o:r.o + r.n].reshape(R, -1, P, P, P)) - r.f
            z.append((r.w.sqrt() * v).reshape(R, -1))
            y.append(ref.LT(r, r.w.sqrt() * gz[:, r.oq:r.oq + r.q].reshape(R, -1, Q, Q, Q)).reshape(R, -1))
        return [torch.cat(z, 1), torch.cat(y, 1).reshape(-1)]
    # gradient of J = 1/2 sum w (u - target)^2 with respect to f, a, grad a at the points: the derivative of
    # -lambda^T (A u - b) for fixed u and lambda, A lambda = dJ/du
    target = _make_data(c, desc, seed + 3)["f"]
    u = ref.solve(ref.rhs())
    blk = lambda r, v: v[:, r.o:r.o + r.n].reshape(1, -1, *(3 * (r.W + 1,)))  # noqa: E731
    value, j = [((0, 0, 0), torch.ones(1, 1, 1, 1, dtype=F64, device=DEV))], []
    for r in ref.runs:
        v = ref.L(r, blk(r, u), value) - target[:, r.oq:r.oq + r.q].reshape(1, *r.w.shape)
        part = SimpleNamespace(t=r.t, terms=value)
        j.append(ref.LT(part, r.w * v).reshape(1, -1))
    lam = ref.solve(torch.cat(j, 1))
    leaves = {k: data[k].detach().requires_grad_(True) for k in ("f", "a", "grad_a")}
    tot = 0.0
    for r in ref.runs:
        terms = ref._terms(r, leaves)
        f = leaves["f"][:, r.oq:r.oq + r.q].reshape(1, *r.w.shape)
        tot = tot - (r.w * ref.L(r, blk(r, lam), terms) * (ref.L(r, blk(r, u), terms) - f)).sum()
    tot.backward()
    return [u.reshape(-1), leaves["f"].grad, leaves["a"].grad, leaves["grad_a"].grad]
