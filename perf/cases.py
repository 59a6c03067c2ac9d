"""Performance cases of the GLRM library: what its users run, through the public
Python entry points (`paper_1410_0342_gb300.glrm`, `.autograd`).

`listed()` gives the fixed cases, `draw(rng)` more of the same ranges,
`prepare(case, seed)` the inputs and the model a program has in hand before the
call, `run(state)` one pass, `work(case)` the bytes and flops a pass cannot do
without, `exact(case, seed)` the same results in 64 bits by plain torch.

Forms (a case's "form"):
  sweep   a short fit: factors and step sizes set, a few alternating
          proximal-gradient sweeps with their objectives, factors read back
  grad    one differentiable objective, forward and backward
  als     one alternating-least-squares sweep
  batch   one sweep of many independent small models
  host    a fit from host arrays: observed set in, one sweep, factors out
Tables (a case's "table"):
  mixed     real (Huber), Boolean (hinge) and ordinal columns, each cell
            observed with probability p; "grouped": the kinds in contiguous
            blocks, else cycling column by column
  dense     the same with every cell present, given as a matrix
  qpca      quadratic loss, every cell observed
  logistic  Boolean columns with logistic loss, cells observed with
            probability p
  completion  quadratic loss on a sparse table of about per_row entries a
            row; skew > 1 makes low-numbered columns popular
"""
import math
import types

import numpy as np
import torch

from paper_1410_0342_gb300 import autograd as AG
from paper_1410_0342_gb300 import glrm as G

QUAD, HUBER, HINGE, LOGISTIC, ORDINAL = range(5)
RQUAD, RL1, RNONNEG = 1, 2, 3
LEVELS = 7
DEV = "cuda"


def listed():
    return [
        # a small experiment in double precision (the qPCA convergence table): latency
        dict(name="qpca_f64_200", form="sweep", table="qpca", m=200, n=100, k=5, prec="f64", sweeps=20),
        # a data frame of a thousand rows whose column types alternate, ragged sizes
        dict(name="frame_1303", form="sweep", table="mixed", grouped=False, m=1303, n=150, k=12, p=0.5, prec="f32",
             sweeps=5),
        # the benchmark: a large mixed-type table, 60% observed
        dict(name="mixed_100k", form="sweep", table="mixed", grouped=True, m=100_000, n=1000, k=20, p=0.6, prec="f32",
             sweeps=1),
        # a mixed table observed too thinly to be stored densely, odd sizes
        dict(name="mixed_thin_50k", form="sweep", table="mixed", grouped=True, m=50_021, n=701, k=18, p=0.25,
             prec="f32", sweeps=1),
        # a complete table with a rank between the padded widths
        dict(name="dense_30k_k33", form="sweep", table="dense", grouped=True, m=30_011, n=777, k=33, prec="f32",
             sweeps=1),
        # large matrix completion, 1% observed
        dict(name="completion_1m", form="sweep", table="completion", m=1_000_000, n=20_000, k=64, per_row=200,
             skew=1.0, prec="f32", sweeps=1),
        # the BF16 precision form of the same problem, a fifth of the rows
        dict(name="completion_bf16", form="sweep", table="completion", m=200_000, n=20_000, k=64, per_row=200,
             skew=1.0, prec="bf16", sweeps=1),
        # a training step of the differentiable form on a mostly observed Boolean table
        dict(name="grad_logistic_50k", form="grad", table="logistic", m=50_000, n=2000, k=32, p=0.8, prec="f32"),
        # a training step on ratings with popular columns, a rank that is no multiple of 4
        dict(name="grad_ratings_60k", form="grad", table="completion", m=60_013, n=5003, k=10, per_row=60, skew=2.0,
             prec="f32"),
        # alternating least squares on a completion table
        dict(name="als_100k", form="als", table="completion", m=100_000, n=20_000, k=32, per_row=200, skew=1.0,
             prec="f32"),
        # hundreds of small models of uneven size, half ALS (quadratic), half prox-grad (Huber)
        dict(name="batch_512", form="batch", count=512, mmax=5000, nmax=500, p=0.7),
        # end to end: host arrays in, one sweep, factors and objective out
        dict(name="host_100k", form="host", table="mixed", grouped=True, m=100_000, n=1000, k=20, p=0.6, prec="f32",
             sweeps=1),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    form = rng.choice(["tiny64", "frame", "mixed", "mixed", "dense", "completion", "completion", "grad", "grad", "als",
                       "batch", "host"])
    if form == "tiny64":
        return dict(form="sweep", table="qpca", m=_log(rng, 40, 1500), n=_log(rng, 20, 300), k=rng.randint(2, 12),
                    prec="f64", sweeps=rng.randint(5, 20))
    if form == "frame":
        return dict(form="sweep", table="mixed", grouped=rng.random() < 0.3, m=_log(rng, 200, 5000),
                    n=_log(rng, 30, 300), k=rng.randint(3, 24), p=round(rng.uniform(0.15, 0.9), 3), prec="f32",
                    sweeps=rng.randint(1, 5))
    if form == "mixed":
        return dict(form="sweep", table="mixed", grouped=rng.random() < 0.8, m=_log(rng, 5000, 100_000),
                    n=_log(rng, 100, 1000), k=rng.randint(4, 32), p=round(rng.uniform(0.12, 0.9), 3),
                    prec=rng.choice(["f32", "f32", "f32", "bf16"]), sweeps=1)
    if form == "dense":
        return dict(form="sweep", table="dense", grouped=rng.random() < 0.8, m=_log(rng, 500, 60_000),
                    n=_log(rng, 60, 1000), k=rng.randint(4, 48), prec=rng.choice(["f32", "f32", "bf16"]), sweeps=1)
    if form in ("completion", "grad", "als"):
        if form == "grad" and rng.random() < 0.5:
            return dict(form="grad", table="logistic", m=_log(rng, 500, 50_000), n=_log(rng, 50, 2000),
                        k=rng.randint(4, 40), p=round(rng.uniform(0.1, 0.9), 3), prec="f32")
        m, per_row = _log(rng, 3000, 400_000 if form == "completion" else 100_000), _log(rng, 10, 200)
        c = dict(form="sweep" if form == "completion" else form, table="completion", m=m,
                 n=_log(rng, 1000, 20_000), k=rng.randint(4, 64) if form != "als" else rng.randint(3, 32),
                 per_row=per_row, skew=rng.choice([1.0, 1.5, 2.0]),
                 prec=rng.choice(["f32", "f32", "bf16"]) if form == "completion" else "f32")
        return dict(c, sweeps=1) if form == "completion" else c
    if form == "batch":
        return dict(form="batch", count=_log(rng, 12, 400), mmax=_log(rng, 200, 5000), nmax=_log(rng, 60, 500),
                    p=round(rng.uniform(0.5, 0.9), 3))
    return dict(form="host", table="mixed", grouped=True, m=_log(rng, 2000, 100_000), n=_log(rng, 100, 1000),
                k=rng.randint(4, 32), p=round(rng.uniform(0.2, 0.8), 3), prec="f32", sweeps=1)


# ----------------------------------------------------------------- inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV)


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV)


def _dtype(case):
    return torch.float64 if case["prec"] == "f64" else torch.float32


def _losses(case):
    """(kind, param, levels) per column."""
    n, t = case["n"], case["table"]
    if t in ("mixed", "dense"):
        j = np.arange(n)
        kind = np.where(j < n // 2, HUBER, np.where(j < n * 4 // 5, HINGE, ORDINAL)) if case["grouped"] else j % 5
    else:
        kind = np.full(n, LOGISTIC if t == "logistic" else QUAD)
    return kind, np.where(kind == HUBER, 1.0, 0.0), np.where(kind == ORDINAL, LEVELS, 0)


def _regs(case):
    t = case["table"]
    if t in ("mixed", "dense"):
        return (RL1, 0.01), (RNONNEG, 0.0)
    w = 0.05 if t == "completion" else 0.1
    return (RQUAD, w), (RQUAD, w)


def _matrix(case, g):
    """(A, observed): the m x n values and which of them are seen (None: all)."""
    m, n, k = case["m"], case["n"], case["k"]
    X, Y = _randn(g, m, k), _randn(g, n, k)
    U = X @ Y.T
    if case["table"] == "qpca":
        return U + 0.1 * _randn(g, m, n), None
    if case["table"] == "logistic":
        A = torch.where(_rand(g, m, n) < torch.sigmoid(U), 1.0, -1.0)
        return A, _rand(g, m, n) < case["p"]
    kind = torch.as_tensor(_losses(case)[0], device=DEV)
    A = U + 0.1 * _randn(g, m, n)                                        # quadratic columns
    s = (kind == HUBER).nonzero()[:, 0]
    if s.numel():                                                        # Laplace(0, 0.5), 1% of entries x 20
        v = _rand(g, m, s.numel()) - 0.5
        e = -0.5 * torch.sign(v) * torch.log1p(-2 * v.abs().clamp(max=0.49999))
        A[:, s] = U[:, s] + torch.where(_rand(g, m, s.numel()) < 0.01, 20 * e, e)
    for q in (HINGE, LOGISTIC):
        s = (kind == q).nonzero()[:, 0]
        if s.numel():
            A[:, s] = torch.where(U[:, s] + 0.5 * _randn(g, m, s.numel()) >= 0, 1.0, -1.0)
    s = (kind == ORDINAL).nonzero()[:, 0]
    if s.numel():                                                        # binned at the septiles of x . y_j
        z = math.sqrt(2) * torch.erfinv(2 * torch.arange(1, LEVELS, device=DEV) / LEVELS - 1)
        u = U[:, s] / Y[s].norm(dim=1)
        A[:, s] = 1.0 + sum((u > z[q]).float() for q in range(LEVELS - 1))
    return A, (None if case["table"] == "dense" else _rand(g, m, n) < case["p"])


def _sparse(case, g):
    """(rows, cols, values) of a completion table in row order, columns ascending."""
    m, n, k, r = case["m"], case["n"], case["k"], case["per_row"]
    sd = k ** -0.25
    X, Y = _randn(g, m, k) * sd, _randn(g, n, k) * sd
    uniform = case["skew"] == 1.0
    slots = min(r if uniform else 2 * r, n // 2)                         # skewed tables have rows of uneven length
    u = _rand(g, m, slots)
    c = ((n - slots + 1) * (u if uniform else u ** case["skew"])).to(torch.int32).clamp_(max=n - slots)
    del u
    c = torch.sort(c, dim=1).values + torch.arange(slots, dtype=torch.int32, device=DEV)
    if uniform:
        rows = torch.arange(m, dtype=torch.int32, device=DEV).repeat_interleave(slots)
        cols = c.reshape(-1)
    else:
        keep = _rand(g, m, slots) < 0.5
        rows = keep.nonzero()[:, 0].to(torch.int32)
        cols = c[keep]
    val = 0.1 * _randn(g, cols.numel())
    for a in range(0, cols.numel(), 1 << 23):
        s = slice(a, a + (1 << 23))
        val[s] += (X[rows[s]] * Y[cols[s]]).sum(1)
    return rows, cols, val


def _pointers(idx, n):
    p = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    p[1:] = torch.cumsum(torch.bincount(idx, minlength=n), 0)
    return p.to(torch.int32)


def _entries(case, g):
    """(rows, cols, values) of the observed set in row order."""
    if case["table"] == "completion":
        return _sparse(case, g)
    A, seen = _matrix(case, g)
    nz = (torch.ones_like(A, dtype=torch.bool) if seen is None else seen).nonzero()
    return nz[:, 0].to(torch.int32), nz[:, 1].to(torch.int32), A[nz[:, 0], nz[:, 1]]


def _csc(rows, cols, val):
    order = torch.sort(cols, stable=True).indices
    return rows[order], val[order]


def _start(case, g):
    """Initial factors: small, as a fit begins (nonnegative where Y has to be)."""
    m, n, k, t = case["m"], case["n"], case["k"], case["table"]
    sd = {"qpca": 1.0, "logistic": 1.0, "completion": k ** -0.25}.get(t, 0.1)
    X, Y = sd * _randn(g, m, k), sd * _randn(g, n, k)
    return X.to(_dtype(case)), (Y.abs() if _regs(case)[1][0] == RNONNEG else Y).to(_dtype(case))


def _batch(case, seed):
    """Concatenated instances: m in [50, mmax], n in [20, nmax], k of 4, 8, 16;
    even ones quadratic, odd ones Huber; A = X0 Y0 + N(0, 0.2^2)."""
    host = np.random.default_rng(case["count"])  # the sizes; the values come from the seed
    g = _gen(seed)
    b = types.SimpleNamespace(count=case["count"], m=[], n=[], k=[], kind=[], nnz=[])
    parts = {q: [] for q in ("rowptr", "colidx", "val", "colptr", "rowidx", "cval", "X0", "Yt0")}
    for s in range(case["count"]):
        m, n = int(host.integers(50, case["mmax"] + 1)), int(host.integers(20, case["nmax"] + 1))
        k = int(host.choice([4, 8, 16]))
        A = _randn(g, m, k) @ _randn(g, n, k).T + 0.2 * _randn(g, m, n)
        seen = _rand(g, m, n) < case["p"]
        nz, tz = seen.nonzero(), seen.T.nonzero()
        for q, v in (("rowptr", _pointers(nz[:, 0], m)), ("colidx", nz[:, 1]), ("val", A[nz[:, 0], nz[:, 1]]),
                     ("colptr", _pointers(tz[:, 0], n)), ("rowidx", tz[:, 1]), ("cval", A[tz[:, 1], tz[:, 0]]),
                     ("X0", _randn(g, m * k)), ("Yt0", _randn(g, n * k))):
            parts[q].append(v if v.is_floating_point() else v.to(torch.int32))
        for q, v in (("m", m), ("n", n), ("k", k), ("kind", s % 2), ("nnz", nz.shape[0])):
            getattr(b, q).append(v)
    for q in ("m", "n", "k", "kind", "nnz"):
        setattr(b, q, np.array(getattr(b, q), np.int64))
    for q, v in parts.items():
        setattr(b, q, torch.cat(v))
    return b


def prepare(case, seed):
    if case["form"] == "batch":
        b = _batch(case, seed)
        methods = np.where(b.kind == QUAD, G.GLRM_BATCH_ALS, G.GLRM_BATCH_PROXGRAD)
        return dict(form="batch", batch=G.Batch(b, methods, rx=(RQUAD, 0.1), ry=(RQUAD, 0.1)), X0=b.X0, Yt0=b.Yt0)
    g = _gen(seed)
    prec = {"f64": G.GLRM_FP64, "f32": G.GLRM_FP32, "bf16": G.GLRM_BF16}[case["prec"]]
    rx, ry = _regs(case)
    model = G.GLRM(case["m"], case["n"], case["k"], _losses(case), rx, ry, prec)
    state = dict(form=case["form"], model=model, sweeps=case.get("sweeps", 1))
    dt = _dtype(case)
    if case["table"] == "dense":
        model.set_dense(_matrix(case, g)[0])
    else:
        rows, cols, val = _entries(case, g)
        rowptr, val = _pointers(rows, case["m"]), val.to(dt)
        if case["form"] == "host":
            state["csr"] = [torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for t in (rowptr, cols, val)]
        else:
            rowidx, cval = _csc(rows, cols, val)
            G.glrm_set_observed(model.h, int(cols.numel()), rowptr, cols.contiguous(), val,
                                _pointers(cols, case["n"]), rowidx, cval)
    X0, Yt0 = _start(case, g)
    if case["form"] == "grad":
        X0, Yt0 = X0.requires_grad_(), Yt0.requires_grad_()
    if case["form"] == "host":
        X0, Yt0 = ([torch.empty(t.shape, dtype=t.dtype, pin_memory=True).copy_(t) for t in (X0, Yt0)])
        state["X"], state["Yt"] = torch.empty_like(X0).pin_memory(), torch.empty_like(Yt0).pin_memory()
    state["X0"], state["Yt0"] = X0, Yt0
    return state


# ------------------------------------------------------------------- a pass

def run(state):
    if state["form"] == "batch":
        b = state["batch"]
        b.set_factors(state["X0"], state["Yt0"])
        objective = b.sweep(1)
        X, Yt = b.factors()
        return dict(X=X, Yt=Yt, objective=objective.astype(np.float32))
    model, X0, Yt0 = state["model"], state["X0"], state["Yt0"]
    if state["form"] == "grad":
        X0.grad = Yt0.grad = None
        F = AG.glrm_objective(X0, Yt0, model)
        F.backward()
        return dict(X=X0.grad, Yt=Yt0.grad, objective=F.detach().to(X0.dtype))
    if state["form"] == "host":
        rowptr, cols, val = state["csr"]
        G.glrm_set_observed_csr_host(model.h, cols.numel(), rowptr, cols, val)
        G.glrm_set_factors_host(model.h, X0, Yt0)
        objective = model.sweep(state["sweeps"])
        G.glrm_get_factors_host(model.h, state["X"], state["Yt"])
        return dict(X=state["X"], Yt=state["Yt"], objective=objective.astype(np.float32))
    model.set_factors(X0, Yt0)
    if state["form"] == "als":
        objective = model.als_sweep(1)
    else:
        G.glrm_reset_steps(model.h)
        objective = model.sweep(state["sweeps"])
    X, Yt = model.factors()
    # the objective is a sum of terms in the model's element type
    return dict(X=X, Yt=Yt, objective=objective.astype(np.float64 if X.dtype == torch.float64 else np.float32))


def work(case):
    """Every observed entry's index and value once per half-step, every factor
    row read and written; per entry and half-step a dot product, the gradient
    update and the new candidate's dot product (2 k each; the gradient form
    has no candidate; a Gram update takes k (k + 1))."""
    if case["form"] == "batch":
        host = np.random.default_rng(case["count"])
        nnz = fl = rows = 0
        for _ in range(case["count"]):
            m, n = int(host.integers(50, case["mmax"] + 1)), int(host.integers(20, case["nmax"] + 1))
            k = int(host.choice([4, 8, 16]))
            e = case["p"] * m * n
            nnz, rows, fl = nnz + e, rows + (m + n) * k, fl + e * (6 * k * k + 12 * k) / 2
        return dict(bytes=16 * nnz + 16 * rows, flops=fl)
    m, n, k = case["m"], case["n"], case["k"]
    es = 8 if case["prec"] == "f64" else 4
    nnz = m * min(case["per_row"], n // 2) if case["table"] == "completion" else m * n * case.get("p", 1.0)
    entry = es if case["table"] == "dense" else es + 4
    factors = (m + n) * k * es
    if case["form"] == "grad":
        return dict(bytes=2 * nnz * entry + 2 * factors, flops=10 * k * nnz)
    if case["form"] == "als":
        return dict(bytes=2 * nnz * entry + 2 * factors, flops=2 * nnz * (k * (k + 1) + 2 * k) + 2 * k * nnz)
    T = case["sweeps"]
    host = nnz * entry if case["form"] == "host" else 0
    return dict(bytes=host + T * (2 * nnz * entry + 2 * factors), flops=12 * k * nnz * T)


# --------------------------------------------- the same results in 64 bits

def _loss(kind, u, a):
    """(L, dL/du) of one kind; Huber threshold 1, ordinal levels 1 .. LEVELS."""
    if kind == QUAD:
        return (u - a) ** 2, 2 * (u - a)
    if kind == HUBER:
        x = u - a
        c = x.clamp(-1, 1)
        return c * (x - 0.5 * c), c
    if kind == HINGE:
        z = 1 - a * u
        return z.clamp(min=0), torch.where(z > 0, -a, torch.zeros_like(a))
    if kind == LOGISTIC:
        z = -a * u
        return torch.nn.functional.softplus(z, threshold=700), -a * torch.sigmoid(z)
    L, d = torch.zeros_like(u), torch.zeros_like(u)
    for q in range(1, LEVELS + 1):
        below, above = (q < a) & (1 - u + q > 0), (q > a) & (1 + u - q > 0)
        L += torch.where(below, 1 - u + q, 0.0) + torch.where(above, 1 + u - q, 0.0)
        d += above.double() - below.double()
    return L, d


def _reg(reg, x):
    kind, w = reg
    if kind == RQUAD:
        return w * (x * x).sum(1)
    if kind == RL1:
        return w * x.abs().sum(1)
    return torch.where((x < 0).any(1), math.inf, 0.0).double()


def _prox(reg, al, z):
    kind, w = reg
    al = al[:, None]
    if kind == RQUAD:
        return z / (1 + 2 * al * w)
    if kind == RL1:
        return torch.sign(z) * (z.abs() - al * w).clamp(min=0)
    return z.clamp(min=0)


class _Exact:
    """The table in 64 bits: a matrix with its mask, or entry lists."""

    def __init__(self, case, g):
        self.m, self.n, self.kind = case["m"], case["n"], _losses(case)[0]
        self.entries = None
        if case["table"] == "completion":
            self.entries = _sparse(case, g)
            self.counts = [torch.bincount(e, minlength=s).double() for e, s in zip(self.entries, (self.m, self.n))]
        else:
            self.A, seen = _matrix(case, g)
            self.seen = torch.ones_like(self.A, dtype=torch.bool) if seen is None else seen
            self.counts = [self.seen.sum(1).double(), self.seen.sum(0).double()]

    def half(self, rowside, X, Y, grad):
        """(loss per segment, gradient) of the rows' or the columns' side."""
        F, W = (X, Y) if rowside else (Y, X)
        f = torch.zeros(F.shape[0], dtype=torch.float64, device=DEV)
        gr = torch.zeros_like(F) if grad else None
        if self.entries is not None:
            rows, cols, val = self.entries
            for a in range(0, cols.numel(), 1 << 22):
                s = slice(a, a + (1 << 22))
                i, j = (rows[s], cols[s]) if rowside else (cols[s], rows[s])
                w = W[j]
                L, d = _loss(QUAD, (F[i] * w).sum(1), val[s].double())
                f.index_add_(0, i, L)
                if grad:
                    gr.index_add_(0, i, d[:, None] * w)
            return f, gr
        for kd in np.unique(self.kind):
            c = torch.as_tensor(np.nonzero(self.kind == kd)[0], device=DEV)
            for a in range(0, self.m, 1 << 14):
                r = slice(a, a + (1 << 14))
                see = self.seen[r][:, c].double()
                L, d = _loss(kd, X[r] @ Y[c].T, self.A[r][:, c].double())
                L, d = L * see, d * see
                if rowside:
                    f[r] += L.sum(1)
                    if grad:
                        gr[r] += d @ Y[c]
                else:
                    f[c] += L.sum(0)
                    if grad:
                        gr[c] += d.T @ X[r]
        return f, gr


def _exact_sweeps(T, X, Y, regs, sweeps):
    F = [X, Y]
    al = [1 / c.clamp(min=1) for c in T.counts]
    hist = []
    for _ in range(sweeps):
        for q in (0, 1):
            f0, gr = T.half(q == 0, F[0], F[1], True)
            cand = _prox(regs[q], al[q], F[q] - al[q][:, None] * gr)
            new = (cand, F[1]) if q == 0 else (F[0], cand)
            f1, _ = T.half(q == 0, *new, False)
            ok = f1 + _reg(regs[q], cand) <= f0 + _reg(regs[q], F[q])
            F[q] = torch.where(ok[:, None], cand, F[q])
            al[q] = al[q] * (0.7 + 0.35 * ok.double())
            kept = torch.where(ok, f1, f0)
        hist.append(float(kept.sum() + _reg(regs[0], F[0]).sum() + _reg(regs[1], F[1]).sum()))
    return dict(X=F[0], Yt=F[1], objective=np.array(hist))


def _exact_als(rows, cols, val, m, n, X, Y, w):
    out = []
    for nseg, seg, oth, W in ((m, rows, cols, lambda: Y), (n, cols, rows, lambda: out[0])):
        order = torch.sort(seg, stable=True).indices
        ptr = _pointers(seg, nseg).long()
        o, v, V = oth[order], val[order].double(), W()
        k = V.shape[1]
        F = torch.zeros(nseg, k, dtype=torch.float64, device=DEV)
        for a in range(0, nseg, 128):
            z = min(a + 128, nseg)
            p, e = ptr[a:z], ptr[a + 1:z + 1]
            at = p[:, None] + torch.arange(max(1, int((e - p).max())), device=DEV)
            in_ = at < e[:, None]
            at = torch.where(in_, at, 0)
            w_ = V[o[at]] * in_[:, :, None]
            b = (w_ * (v[at] * in_)[:, :, None]).sum(1)
            F[a:z] = torch.linalg.solve(w_.transpose(1, 2) @ w_ + w * torch.eye(k, device=DEV).double(), b)
        out.append(F)
    loss = sum(float((((out[0][rows[a:a + (1 << 22)]] * out[1][cols[a:a + (1 << 22)]]).sum(1)
                       - val[a:a + (1 << 22)].double()) ** 2).sum()) for a in range(0, cols.numel(), 1 << 22))
    return dict(X=out[0], Yt=out[1],
                objective=np.array([loss + w * float((out[0] ** 2).sum() + (out[1] ** 2).sum())]))


def _exact_batch(case, seed):
    b = _batch(case, seed)
    X, Y, obj = [], [], []
    e = xo = yo = rp = 0
    regs = ((RQUAD, 0.1), (RQUAD, 0.1))
    for s in range(b.count):
        m, n, k, nnz = (int(v[s]) for v in (b.m, b.n, b.k, b.nnz))
        X0, Y0 = b.X0[xo:xo + m * k].reshape(m, k).double(), b.Yt0[yo:yo + n * k].reshape(n, k).double()
        cols, val = b.colidx[e:e + nnz].long(), b.val[e:e + nnz]
        rows = torch.arange(m, device=DEV).repeat_interleave(torch.diff(b.rowptr[rp:rp + m + 1].long()))
        A = torch.zeros(m, n, device=DEV)
        A[rows, cols] = val
        T = _Exact.__new__(_Exact)
        T.m, T.n, T.kind, T.entries, T.A = m, n, np.full(n, b.kind[s]), None, A
        T.seen = torch.zeros(m, n, dtype=torch.bool, device=DEV)
        T.seen[rows, cols] = True
        T.counts = [T.seen.sum(1).double(), T.seen.sum(0).double()]
        if b.kind[s] == QUAD:
            M, eye = T.seen.double(), 0.1 * torch.eye(k, device=DEV).double()
            for q in (0, 1):
                V, Mq = (Y0, M) if q == 0 else (X0, M.T)
                gram = (Mq @ (V[:, :, None] * V[:, None, :]).reshape(-1, k * k)).reshape(-1, k, k)
                F = torch.linalg.solve(gram + eye, (A.double() if q == 0 else A.double().T) @ V)
                X0, Y0 = (F, Y0) if q == 0 else (X0, F)
            f = float((M * (X0 @ Y0.T - A) ** 2).sum() + 0.1 * ((X0 ** 2).sum() + (Y0 ** 2).sum()))
            r = dict(X=X0, Yt=Y0, objective=[f])
        else:
            r = _exact_sweeps(T, X0, Y0, regs, 1)
        X.append(r["X"].reshape(-1))
        Y.append(r["Yt"].reshape(-1))
        obj.append(r["objective"][0])
        e, xo, yo, rp = e + nnz, xo + m * k, yo + n * k, rp + m + 1
    return dict(X=torch.cat(X), Yt=torch.cat(Y), objective=np.array([obj]))


def exact(case, seed):
    if case["form"] == "batch":
        return _exact_batch(case, seed)
    g = _gen(seed)
    regs = _regs(case)
    if case["form"] == "als":
        rows, cols, val = _sparse(case, g)
        X, Y = (v.double() for v in _start(case, g))
        return _exact_als(rows, cols, val, case["m"], case["n"], X, Y, regs[0][1])
    T = _Exact(case, g)
    X, Y = (v.double() for v in _start(case, g))
    if case["form"] == "grad":
        f, gx = T.half(True, X, Y, True)
        _, gy = T.half(False, X, Y, True)
        w = regs[0][1]
        return dict(X=gx + 2 * w * X, Yt=gy + 2 * w * Y,
                    objective=f.sum() + w * ((X ** 2).sum() + (Y ** 2).sum()))
    return _exact_sweeps(T, X, Y, regs, case["sweeps"])
