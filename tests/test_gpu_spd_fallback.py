"""Alternating minimisation on systems that the FP32 factorisation cannot
precondition: the FP64 factorisation has to solve them, in the single-model and
the batched form.  All Gram matrices and right-hand sides are sums of small
integers, exact in FP32, so the stored solution may differ from the exact one by
the FP64 solve's error (some 8 k 2^-53 times the condition number) and one
rounding to FP32.  Systems that the refined FP32 solve settles and systems that
it does not alternate, so both kinds share a warp."""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_1410_0342_gb300 import workloads as W

pytestmark = pytest.mark.gpu

GAMMA = 2.0 ** -12  # above the rounding of the columns' FP32 Gram matrices (1e-6), below the rows' second pivots (0.008)
COUNT = 44


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1410_0342_gb300 import build
    build.build()
    from paper_1410_0342_gb300 import glrm
    return glrm


def pair_entry(s):
    """The s-th p for which rows (p, p - 64), (p + 1, p - 63) (determinant 64,
    condition number about 2^27) leave a second pivot in FP32 that is negative
    or off by more than a quarter: too far for corrections that have to shrink
    by 2^30 in six rounds, a factor of 1/32 each."""
    f = np.float32
    found = []
    for p in range(500, 300, -1):
        g11, g12, g22 = f(p * p + (p + 1) ** 2), f(p * (p - 64) + (p + 1) * (p - 63)), f((p - 64) ** 2 + (p - 63) ** 2)
        d = f(float(g22) - float(g12 * (f(1) / g11)) * float(g12))
        if d <= 0 or abs(1 - (4096.0 / float(g11) + 2 * GAMMA) / float(d)) > 0.25:
            found.append(p)
    return found[s]


def system(k, s):
    """The k rows of system s (k x k whole numbers) and its solution; odd
    systems hold two almost parallel rows."""
    rng = W.rng_for(7000 + 100 * k + s)
    j = s % (k - 1)
    pair = [j, j + 1] if s % 2 else []
    rest = [c for c in range(k) if c not in pair]
    w = np.zeros((k, k))
    for i, c in enumerate(rest):
        w[c, c] = 2
        if i + 1 < len(rest):
            w[c, rest[i + 1]] = 1
    if pair:
        p = pair_entry(s)
        w[j, pair] = p, p - 64
        w[j + 1, pair] = p + 1, p - 63
    return w, rng.integers(-4, 5, k).astype(np.float64)


def table(k):
    """Row i of the table is system i; its entries lie in columns of its own."""
    sys_ = [system(k, s) for s in range(COUNT)]
    Yt = np.concatenate([w for w, _ in sys_])
    val = np.concatenate([w @ x for w, x in sys_])
    m, n = COUNT, COUNT * k
    rowptr = np.arange(m + 1) * k
    colidx = np.arange(n, dtype=np.int32)
    t = W._finish("spd", m, n, k, rowptr, colidx, val, np.zeros(n, np.int32), np.zeros(n), np.zeros(n),
                  (1, GAMMA), (1, GAMMA), W.rng_for(k))
    t.X0, t.Yt0 = np.zeros((m, k)), Yt
    return t, sys_


def solve_exact(w, x):
    """(w^T w + gamma I)^-1 w^T w x in rational arithmetic."""
    k = len(x)
    gram = (w.T @ w).astype(int)
    a = [[Fraction(int(gram[i, j])) + (Fraction(GAMMA) if i == j else 0) for j in range(k)]
         + [Fraction(int(gram[i] @ x.astype(int)))] for i in range(k)]
    for c in range(k):
        for r in range(c + 1, k):
            if a[r][c]:
                f = a[r][c] / a[c][c]
                a[r] = [u - f * v if v else u for u, v in zip(a[r], a[c])]
    out = [Fraction(0)] * k
    for c in reversed(range(k)):
        out[c] = (a[c][k] - sum(a[c][q] * out[q] for q in range(c + 1, k))) / a[c][c]
    return np.array([float(v) for v in out])


def check(X, sys_, k):
    for s, (w, x) in enumerate(sys_):
        want = solve_exact(w, x)
        cond = np.linalg.cond(w.T @ w + GAMMA * np.eye(k))
        bound = (2.0 ** -24 + 2.0 ** -30 + 8 * k * 2.0 ** -53 * cond) * np.abs(want).max()
        assert np.abs(X[s] - want).max() <= bound, (s, X[s], want, bound)


@pytest.mark.parametrize("k", [4, 8, 16, 32])
def test_single_model(G, k):
    t, sys_ = table(k)
    g = G.GLRM.from_table(t)
    G.glrm_set_path(g.h, 1, 1)
    g.als_sweep(1)
    check(g.factors()[0].double().cpu().numpy(), sys_, k)


@pytest.mark.parametrize("k", [4, 8, 16])
def test_batched_form(G, k):
    t, sys_ = table(k)
    dev = lambda v, dt: torch.as_tensor(np.asarray(v), dtype=dt, device="cuda")
    wb = W.Batch(m=np.array([t.m]), n=np.array([t.n]), k=np.array([k], np.int32), kind=np.array([0], np.int32),
                 nnz=np.array([t.n]), rowptr=dev(t.rowptr, torch.int32), colidx=dev(t.colidx, torch.int32),
                 val=dev(t.val, torch.float32), colptr=dev(t.colptr, torch.int32),
                 rowidx=dev(t.rowidx, torch.int32), cval=dev(t.cval, torch.float32),
                 X0=dev(t.X0.reshape(-1), torch.float32), Yt0=dev(t.Yt0.reshape(-1), torch.float32))
    B = G.Batch(wb, [G.GLRM_BATCH_ALS], rx=(1, GAMMA), ry=(1, GAMMA))
    B.sweep(1)
    check(B.factors()[0].reshape(t.m, k).double().cpu().numpy(), sys_, k)
