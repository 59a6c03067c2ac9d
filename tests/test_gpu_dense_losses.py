"""The dense form's loss blocks, kind by kind: tables whose columns share one
loss kind, at sizes that leave partial 16-column groups, 32-column blocks,
64-wide chunks and 128-row tiles, fully observed and with missing cells, at
factors that reach the logistic loss's tails and ordinal levels beyond the
whole numbers BF16 holds.  Objective and gradient against the FP64 oracle
within the FP32 summation bounds of gpu_parity."""
import numpy as np
import pytest
import torch

from paper_1410_0342_gb300 import workloads as W

from gpu_parity import assert_grad_close, grad_bounds, oracle_problem

pytestmark = pytest.mark.gpu

RQ = 1


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1410_0342_gb300 import build
    build.build()
    from paper_1410_0342_gb300 import glrm
    return glrm


def one_kind_table(kind, m, n, k, p_obs, levels, scale, seed):
    rng = W.rng_for(seed)
    X0, Y0t = rng.standard_normal((m, k)), rng.standard_normal((n, k))
    rowptr, colidx = W.omega_bernoulli(m, n, p_obs, rng)
    u = W.sampled_products(X0, Y0t, rowptr, colidx)
    if kind in (W.LOSS_HINGE, W.LOSS_LOGISTIC):
        val = np.where(u + 0.5 * rng.standard_normal(u.size) >= 0, 1.0, -1.0)
    elif kind == W.LOSS_ORDINAL:
        val = np.clip(np.round(u * levels / 8 + (levels + 1) / 2), 1, levels)
    else:
        val = u + rng.laplace(0.0, 0.5, u.size)
    t = W._finish("one_kind", m, n, k, rowptr, colidx, val, np.full(n, kind),
                  np.full(n, 1.0 if kind == W.LOSS_HUBER else 0.0), np.full(n, levels if kind == W.LOSS_ORDINAL else 0),
                  (RQ, 0.1), (RQ, 0.1), rng)
    t.X0 = np.asarray(scale * t.X0, np.float32).astype(np.float64)
    t.Yt0 = np.asarray(t.Yt0, np.float32).astype(np.float64)
    t.val = t.val.astype(np.float32).astype(np.float64)
    t.cval = t.cval.astype(np.float32).astype(np.float64)
    return t


@pytest.mark.parametrize("p_obs", [0.6, 1.0])
@pytest.mark.parametrize("m,n", [(197, 83), (129, 64), (64, 17)])
@pytest.mark.parametrize("kind,levels,scale", [(0, 0, 1.0), (1, 0, 1.0), (2, 0, 1.0), (3, 0, 1.0), (3, 0, 40.0),
                                               (4, 7, 2.0), (4, 600, 90.0)])
def test_loss_blocks_of_one_kind(G, oracle_mod, kind, levels, scale, m, n, p_obs):
    t = one_kind_table(kind, m, n, 6, p_obs, levels, scale, seed=900 + kind + m)
    g = G.GLRM.from_dense_table(t) if p_obs == 1.0 else G.GLRM.from_table(t)
    assert G.glrm_get_path(g.h) == (G.GLRM_PATH_DENSE, G.GLRM_PATH_DENSE)
    p = oracle_problem(oracle_mod, t)
    F = p.objective(t.X0, t.Yt0)
    assert abs(g.objective() - F) <= 1e-5 * abs(F)
    gx, gy = p.gradient(t.X0, t.Yt0)
    sx, sy, vx, vy = grad_bounds(p, t.X0, t.Yt0)
    GX, GYt = g.grad()
    assert_grad_close(GX.cpu().numpy(), gx, sx, vx, what="dF/dX")
    assert_grad_close(GYt.cpu().numpy(), gy, sy, vy, what="dF/dYt")
