"""The work that users have this library do, as cases that can be timed and compared.

An interior-point ACOPF code analyses the KKT pattern of its grid once and then, for every Newton iteration, evaluates
the values of K, refactors, solves and refines; batches of scenarios do the same for many instances of one pattern.
Kinds of cases, each through the package's public entry points:

* ``step``: ``KKTSolver.refactor_refine`` of one fresh K (``count`` > 1: of that many scenarios of one grid at once),
  the linear algebra of a Newton iteration.
* ``solve``: ``KKTSolver.solve``, triangular solves with the factors at hand (predictor-corrector right-hand sides).
* ``residual``: ``KKTSolver.residual``, the backward error of a given x.
* ``model``: ``KKTModel.assemble``, the values of K at an iterate.
* ``ipm``: ``KKTModel.ipm_solve``, a whole ACOPF solve.

Grids are the seeded synthetic ones of ``kktgen`` with the repository's proportions (1.28 lines and 0.2 generators per
bus where nothing else is said); an iterate's multipliers, barrier diagonal (log-uniform on [1e-8, 1e8]) and
regularization (1e-8, 1e-10) are those of its benchmark. On these matrices (condition numbers of 1e13 and more at 60
buses) FP64 factors give x to 3 to 6 digits on small grids, which are compared with a dense 64-bit solve; FP32 factors
meet the backward error asked for with an x that differs from it by its own size, so those cases are compared with each
other alone.
"""
import functools
import math

import numpy as np
import torch

import paper_2302_08656_gb300 as K
from kktgen import flat_start, make_grid, opf_data

DEV = "cuda"
DW, DC = 1e-8, 1e-10
TOL = 1e-10
DENSE_BUSES = 400       # FP64 steps up to this size are compared with a dense solve
MAX_BUSES = 70_000


def _step(n_bus, precision, count=1, **sizes):
    return dict(kind="step", n_bus=n_bus, precision=precision, count=count, **sizes)


def listed():
    return [
        # a small grid: launches and the host path of one Newton iteration (the tests' 200-bus system)
        dict(_step(200, "fp64", n_branch=300, n_gen=40), name="step-200-fp64"),
        # a mid-sized grid with FP32 factors, an odd size
        dict(_step(2_003, "fp32"), name="step-2003-fp32"),
        # a regional grid in plain FP64, an odd size
        dict(_step(9_973, "fp64"), name="step-9973-fp64"),
        # the paper's Northeast sizes, both factor precisions
        dict(_step(25_000, "fp32", n_branch=32_000, n_gen=5_000), name="step-25k-fp32"),
        dict(_step(25_000, "fp64", n_branch=32_000, n_gen=5_000), name="step-25k-fp64"),
        # the paper's Eastern sizes, the benchmark's headline, both factor precisions
        dict(_step(70_000, "fp32", n_branch=88_000, n_gen=10_000), name="step-70k-fp32"),
        dict(_step(70_000, "fp64", n_branch=88_000, n_gen=10_000), name="step-70k-fp64"),
        # 64 scenarios of one 2,000-bus grid
        dict(_step(2_000, "fp32", count=64), name="batch-64x2k-fp32"),
        # one more right-hand side with the factors at hand
        dict(kind="solve", n_bus=25_000, n_branch=32_000, n_gen=5_000, precision="fp64", name="solve-25k-fp64"),
        # the accuracy check of a given x
        dict(kind="residual", n_bus=25_000, n_branch=32_000, n_gen=5_000, name="residual-25k"),
        # the values of K at an iterate of the largest grid
        dict(kind="model", n_bus=70_000, n_branch=88_000, n_gen=10_000, name="model-70k"),
        # a whole ACOPF solve, about 25 Newton iterations
        dict(kind="ipm", n_bus=2_000, name="ipm-2k"),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["step"] * 10 + ["batch"] * 3 + ["solve"] * 3 + ["residual"] + ["model"] * 2 + ["ipm"])
    if kind == "step":
        return _step(size(60, MAX_BUSES), rng.choice(["fp64", "fp32"]))
    if kind == "batch":
        n = size(100, 10_000)
        return _step(n, "fp32", count=min(size(2, 64), max(2, 128_000 // n)))
    if kind == "solve":
        return dict(kind=kind, n_bus=size(200, 25_000), precision=rng.choice(["fp64", "fp32"]))
    if kind == "ipm":
        return dict(kind=kind, n_bus=size(60, 1_900))
    return dict(kind=kind, n_bus=size(200, 25_000 if kind == "residual" else MAX_BUSES))


# ------------------------------------------------------------------ inputs

def _sizes(case):
    B = case["n_bus"]
    return B, case.get("n_branch", int(round(1.28 * B))), case.get("n_gen", max(1, int(round(0.2 * B))))


@functools.lru_cache(maxsize=4)
def _grid(n_bus, n_branch, n_gen):
    return make_grid(1, n_bus, n_branch, n_gen)


def _iterate(g, rng):
    """One interior-point iterate (V, theta, lambda, Sigma)."""
    V = rng.uniform(0.95, 1.05, g.n_bus)
    dth = rng.normal(0.0, 0.1, g.n_bus).tolist()
    parent, theta = g.tree_parent.tolist(), [0.0] * g.n_bus
    for v in g.tree_order[1:].tolist():
        theta[v] = theta[parent[v]] + dth[v]
    lam = rng.normal(0.0, 1.0, 2 * g.n_bus + 2 * g.n_branch)
    sigma = np.exp(rng.uniform(math.log(1e-8), math.log(1e8), 2 * g.n_bus + 2 * g.n_gen))
    sigma[g.n_bus:2 * g.n_bus] = 0.0
    return V, np.array(theta), lam, sigma


def _draws(case, seed):
    """The grid, `count` iterates and as many right-hand sides; the x of a residual case."""
    g = _grid(*_sizes(case))
    rng = np.random.default_rng([int(seed), 0x6b6b74])
    its = [_iterate(g, rng) for _ in range(case.get("count", 1))]
    n = 4 * g.n_bus + 2 * g.n_gen + 2 * g.n_branch
    b = rng.normal(0.0, 1.0, (len(its), n))
    return g, its, b, rng.normal(0.0, 1.0, n)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def prepare(case, seed):
    if case["kind"] == "ipm":
        g = _grid(*_sizes(case))
        data = opf_data(g, seed)
        model = K.KKTModel.from_grid(g)
        model.set_limits(data)
        solver = K.KKTSolver(model.rowptr, model.colidx, model.n_primal)
        return dict(case=case, model=model, solver=solver, x0=_dev(flat_start(g, data)))
    g, its, b, x = _draws(case, seed)
    model = K.KKTModel.from_grid(g)
    dev = [tuple(_dev(a) for a in it) for it in its]
    if case["kind"] == "model":
        vals = torch.empty(model.nnz, dtype=torch.float64, device=DEV)
        return dict(case=case, model=model, it=dev[0], vals=vals)
    vals = torch.empty(len(its), model.nnz, dtype=torch.float64, device=DEV)
    for v, it in zip(vals, dev):
        model.assemble(*it, DW, DC, out=v)
    count = len(its)
    solver = K.KKTSolver(model.rowptr, model.colidx, model.n_primal, count=count,
                         precision=case.get("precision", "fp64"))
    rhs = _dev(b.reshape(-1))
    state = dict(case=case, solver=solver, vals=vals.reshape(-1), rhs=rhs, out=torch.empty_like(rhs))
    if case["kind"] in ("solve", "residual"):
        solver.refactor(state["vals"])
        state["x"] = _dev(x)
    torch.cuda.synchronize()
    return state


def run(s):
    kind = s["case"]["kind"]
    if kind == "step":
        x, info = s["solver"].refactor_refine(s["vals"], s["rhs"], out=s["out"], tol=TOL)
        infos = info if isinstance(info, list) else [info]
        return dict(x=x, perturbed=np.array([i.n_perturbed for i in infos]),
                    iterations=np.array([i.iters for i in infos]))
    if kind == "solve":
        return dict(x=s["solver"].solve(s["rhs"], out=s["out"]))
    if kind == "residual":
        r, omega = s["solver"].residual(s["rhs"], s["x"], out=s["out"])
        return dict(r=r, omega=omega)
    if kind == "model":
        return dict(vals=s["model"].assemble(*s["it"], DW, DC, out=s["vals"]))
    x, lam, info = s["model"].ipm_solve(s["solver"], s["x0"].clone())
    return dict(x=x, lam=lam, iterations=info.iters, objective=info.objective)


# -------------------------------------------------------------------- work

def work(case):
    """Compulsory bytes and operations. Per instance: K's values and the right-hand side read, x written, the factors
    written by the refactorization and read by the solve (nonzeros of L + U: 1.65 times K's on these grids, flops
    growing as buses^1.25, both measured on the 25,000- and 70,000-bus grids)."""
    B, L, G = _sizes(case)
    n = 4 * B + 2 * G + 2 * L
    nnz = n + 10 * B + 40 * L + 4 * G
    lu = 1.65 * nnz * (4 if case.get("precision") == "fp32" else 8)
    flops = 75e6 * (B / 25_000) ** 1.25
    if case["kind"] == "step":
        c = case["count"]
        return dict(bytes=c * (8 * nnz + 16 * n + 2 * lu), flops=c * (flops + 2 * 1.65 * nnz))
    if case["kind"] == "solve":
        return dict(bytes=16 * n + lu, flops=2 * 1.65 * nnz)
    if case["kind"] == "residual":
        return dict(bytes=12 * nnz + 24 * n, flops=2 * nnz)
    if case["kind"] == "model":
        return dict(bytes=8 * nnz + 8 * (2 * B + 2 * B + 2 * L + 2 * B + 2 * G) + 32 * L, flops=600 * L)
    return dict(bytes=25 * (8 * nnz + 16 * n + 2 * lu), flops=25 * (flops + 2 * 1.65 * nnz))


# ------------------------------------------------------------------- exact

def _line_flow(Vi, Vj, ti, tj, gg, bb):
    t = ti - tj
    P = gg * Vi * Vi - Vi * Vj * (gg * torch.cos(t) + bb * torch.sin(t))
    Q = -bb * Vi * Vi - Vi * Vj * (gg * torch.sin(t) - bb * torch.cos(t))
    return P, Q


def _exact_K(g, it):
    """(rows, columns, values) of K in CSR order: the ACOPF Lagrangian differentiated line by line, in 64 bits."""
    V, theta, lam, sigma = it
    B, L, G = g.n_bus, g.n_branch, g.n_gen
    n, m = 2 * B + 2 * G, 2 * B + 2 * L
    f, t = torch.from_numpy(g.f), torch.from_numpy(g.t)
    Vt, th, lm = (torch.from_numpy(a) for a in (V, theta, lam))
    u = [a.clone().requires_grad_() for a in (Vt[f], Vt[t], th[f], th[t])]
    gg, bb = torch.from_numpy(g.g), torch.from_numpy(g.b)
    Pf, Qf = _line_flow(u[0], u[1], u[2], u[3], gg, bb)
    Pt, Qt = _line_flow(u[1], u[0], u[3], u[2], gg, bb)
    cons = [(f, -Pf), (t, -Pt), (B + f, -Qf), (B + t, -Qt), (2 * B + torch.arange(L), Pf * Pf + Qf * Qf),
            (2 * B + L + torch.arange(L), Pt * Pt + Qt * Qt)]
    loc = [f, t, B + f, B + t]
    rows, cols, vals = [], [], []

    def put(r, c, v):
        rows.append(r), cols.append(c), vals.append(v)

    for r, c in cons:
        for k, d in enumerate(torch.autograd.grad(c.sum(), u, create_graph=True)):
            put(n + r, loc[k], d.detach())
            put(loc[k], n + r, d.detach())
    lag = sum((lm[r] * c).sum() for r, c in cons)
    for a, d in enumerate(torch.autograd.grad(lag, u, create_graph=True)):
        for k, h in enumerate(torch.autograd.grad(d.sum(), u, retain_graph=True)):
            put(loc[a], loc[k], h)
    gen = torch.from_numpy(g.gen_bus)
    for o, r in ((0, n + gen), (G, n + B + gen)):
        put(r, 2 * B + o + torch.arange(G), torch.ones(G, dtype=torch.float64))
        put(2 * B + o + torch.arange(G), r, torch.ones(G, dtype=torch.float64))
    diag = sigma + DW
    diag[2 * B:2 * B + G] += 2.0 * g.c2
    diag = np.concatenate([diag, np.full(m, -DC)])
    put(torch.arange(n + m), torch.arange(n + m), torch.from_numpy(diag))
    keys, inv = np.unique((torch.cat(rows) * (n + m) + torch.cat(cols)).numpy(), return_inverse=True)
    v = np.bincount(inv.reshape(-1), weights=torch.cat(vals).detach().numpy(), minlength=keys.size)
    return keys // (n + m), keys % (n + m), v


def exact(case, seed):
    if case["kind"] == "model":
        g, its, _, _ = _draws(case, seed)
        return dict(vals=_exact_K(g, its[0])[2])
    if case["kind"] == "residual":
        g, its, b, x = _draws(case, seed)
        i, j, v = _exact_K(g, its[0])
        r = b[0] - np.bincount(i, weights=v * x[j], minlength=x.size)
        knorm = np.bincount(i, weights=np.abs(v)).max()
        return dict(r=r, omega=float(np.abs(r).max() / (knorm * np.abs(x).max() + np.abs(b).max())))
    if case["kind"] == "step" and case["precision"] == "fp64" and case["count"] == 1 and case["n_bus"] <= DENSE_BUSES:
        # a dense solve, equilibrated by powers of two so that the scaling is exact, refined twice
        g, its, b, _ = _draws(case, seed)
        i, j, v = _exact_K(g, its[0])
        A = np.zeros((b.shape[1], b.shape[1]))
        A[i, j] = v
        d = 2.0 ** np.round(-0.5 * np.log2(np.abs(A).max(axis=1)))
        S = torch.from_numpy(d[:, None] * A * d[None, :])
        lu, piv = torch.linalg.lu_factor(S)
        c = torch.from_numpy(d * b[0])[:, None]
        y = torch.linalg.lu_solve(lu, piv, c)
        for _ in range(2):
            y = y + torch.linalg.lu_solve(lu, piv, c - S @ y)
        return dict(x=d * y[:, 0].numpy(), perturbed=None, iterations=None)
    # a dense solve of these sizes, or of every Newton step of an interior-point run, takes minutes; FP32 factors: above
    return None
