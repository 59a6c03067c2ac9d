"""Chunked passes of large ranks (k > 32) against the oracle: segments of 0, 1,
7..9, 1,023 and 1,024 entries and one of 1,025, long columns, weights and
offset, gradients; and the BF16 form's half-step by hand, at a rank its
gradient pass streams through shared memory (56, 64) and one it does not."""
import numpy as np
import pytest
import torch

from paper_1410_0342_gb300 import workloads as W

from gpu_parity import assert_grad_close, grad_bounds, oracle_problem, synced_sweeps

pytestmark = pytest.mark.gpu

RQ, RL1 = 1, 2


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1410_0342_gb300 import build
    build.build()
    from paper_1410_0342_gb300 import glrm
    return glrm


def table(k, longest, seed, nkinds=4):
    rng = W.rng_for(seed)
    lens = [0, 1, 7, 8, 9, 63, 64, 65, 1023, longest] + [int(v) for v in rng.integers(0, 70, 80)]
    m, n = len(lens), 1100
    rowptr = np.concatenate([[0], np.cumsum(lens)])
    colidx = np.concatenate([np.sort(rng.choice(n, c, replace=False)) for c in lens]).astype(np.int32)
    sd = k ** -0.25
    u = W.sampled_products(rng.standard_normal((m, k)) * sd, rng.standard_normal((n, k)) * sd, rowptr, colidx)
    kinds = np.arange(n) % nkinds
    val = np.where(kinds[colidx] >= 2, np.where(u >= 0, 1.0, -1.0), u + 0.1 * rng.standard_normal(u.size))
    t = W._finish("staged", m, n, k, rowptr, colidx, val, kinds, np.where(kinds == 1, 1.0, 0.0), np.zeros(n),
                  (RQ, 0.05), (RL1, 0.02), rng, init_std=sd)
    t.X0, t.Yt0 = (np.asarray(a, np.float32).astype(np.float64) for a in (t.X0, t.Yt0))
    return t


@pytest.mark.parametrize("longest", [1024, 1025])
@pytest.mark.parametrize("k,nkinds", [(35, 4), (36, 4), (44, 1), (48, 4), (52, 1), (64, 4)])
def test_short_segments(G, oracle_mod, k, nkinds, longest):
    t = table(k, longest, 6100 + k, nkinds)
    g = G.GLRM.from_table(t)
    G.glrm_set_path(g.h, 1, 1)
    synced_sweeps(g, oracle_mod, t, 3)


@pytest.mark.parametrize("k", [40, 64])
def test_long_columns_and_gradients(G, oracle_mod, k):
    t = W.completion(m=3001, n=40, k=k, per_row=21, seed=6200 + k)
    g = G.GLRM.from_table(t)
    G.glrm_set_path(g.h, 1, 1)
    p = oracle_problem(oracle_mod, t)
    X, Yt = (np.asarray(a, np.float32).astype(np.float64) for a in (t.X0, t.Yt0))
    gx, gy = p.gradient(X, Yt)
    sx, sy, vx, vy = grad_bounds(p, X, Yt)
    GX, GYt = g.grad()
    assert_grad_close(GX.cpu().numpy(), gx, sx, vx, what="dF/dX")
    assert_grad_close(GYt.cpu().numpy(), gy, sy, vy, what="dF/dYt")
    assert abs(g.objective() - p.objective(X, Yt)) <= 1e-5 * p.objective(X, Yt)
    synced_sweeps(g, oracle_mod, t, 3)


def test_weights_and_offset(G, oracle_mod):
    t = table(40, 1024, 6300)
    w = np.linspace(0.5, 2.0, t.n).astype(np.float32).astype(np.float64)
    g = G.GLRM.from_table(t)
    G.glrm_set_path(g.h, 1, 1)
    g.set_offset(True)
    g.set_column_scale(w)
    synced_sweeps(g, oracle_mod, t, 3, offset=True, col_scale=w)


@pytest.mark.parametrize("k", [44, 56, 64])
def test_bf16_half_step(G, k):
    """One BF16 X-step by hand in FP64: gradients from the rows of Y rounded to
    BF16, candidate and decision on the FP32 rows.  X within the FP32 rounding
    of the gradient's sum (16 units of 2^-24 of its terms' magnitudes, times the
    step) and of the stored result; no row's objectives are near a tie."""
    t = W.completion(m=1501, n=400, k=k, per_row=60, seed=6400 + k)
    g = G.GLRM.from_table(t, precision=G.GLRM_BF16)
    G.glrm_set_path(g.h, 1, 1)
    X0, Y0 = (torch.as_tensor(a, dtype=torch.float32) for a in (t.X0, t.Yt0))
    g.set_factors(X0.cuda(), Y0.cuda())
    g.sweep(1)
    X1 = g.factors()[0].double().cpu().numpy()
    Xd, Yd, Yr = X0.double().numpy(), Y0.double().numpy(), Y0.bfloat16().double().numpy()
    w, al = t.rx[1], 1 / 60
    vals = np.asarray(t.val, np.float32).astype(np.float64)
    for i in range(t.m):
        s = slice(t.rowptr[i], t.rowptr[i + 1])
        j, a = t.colidx[s], vals[s]
        r = Xd[i] @ Yr[j].T - a
        cand = (Xd[i] - al * 2 * r @ Yr[j]) / (1 + 2 * al * w)
        f = lambda x: ((x @ Yd[j].T - a) ** 2).sum() + w * (x ** 2).sum()
        assert abs(f(cand) - f(Xd[i])) > 1e-5 * f(Xd[i])
        want = cand if f(cand) <= f(Xd[i]) else Xd[i]
        bound = al * 2 * 16 * 2.0 ** -24 * (np.abs(r) + np.abs(Xd[i]) @ np.abs(Yr[j]).T) @ np.abs(Yr[j]) + 2.0 ** -22 * np.abs(want)
        assert (np.abs(X1[i] - want) <= bound).all(), i
