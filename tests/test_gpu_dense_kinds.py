"""The dense form's l1 and quantile blocks (the loss kinds that
test_gpu_dense_losses leaves out), as tables of one kind and in uniform groups of
32 columns beside other kinds.  Objective and gradient against the FP64 oracle
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


def table(kinds, m, k, p_obs, seed):
    """Columns of the given kinds; Huber threshold 1, quantile 0.3."""
    rng = W.rng_for(seed)
    n = kinds.size
    rowptr, colidx = W.omega_bernoulli(m, n, p_obs, rng)
    u = W.sampled_products(rng.standard_normal((m, k)), rng.standard_normal((n, k)), rowptr, colidx)
    val = (u + rng.laplace(0.0, 0.5, u.size)).astype(np.float32).astype(np.float64)
    val = np.where(kinds[colidx] == W.LOSS_HINGE, np.where(u >= 0, 1.0, -1.0), val)
    param = np.select([kinds == W.LOSS_HUBER, kinds == W.LOSS_QUANTILE], [1.0, 0.3], 0.0)
    t = W._finish("kinds", m, n, k, rowptr, colidx, val, kinds, param, np.zeros(n), (RQ, 0.1), (RQ, 0.1), rng)
    t.X0, t.Yt0 = (np.asarray(a, np.float32).astype(np.float64) for a in (t.X0, t.Yt0))
    return t


def check(G, oracle_mod, t, full):
    g = G.GLRM.from_dense_table(t) if full else G.GLRM.from_table(t)
    assert G.glrm_get_path(g.h) == (G.GLRM_PATH_DENSE, G.GLRM_PATH_DENSE)
    p = oracle_problem(oracle_mod, t)
    F = p.objective(t.X0, t.Yt0)
    assert abs(g.objective() - F) <= 1e-5 * abs(F)
    gx, gy = p.gradient(t.X0, t.Yt0)
    sx, sy, vx, vy = grad_bounds(p, t.X0, t.Yt0)
    GX, GYt = g.grad()
    assert_grad_close(GX.cpu().numpy(), gx, sx, vx, what="dF/dX")
    assert_grad_close(GYt.cpu().numpy(), gy, sy, vy, what="dF/dYt")


@pytest.mark.parametrize("p_obs", [0.6, 1.0])
@pytest.mark.parametrize("m,n", [(197, 83), (128, 64), (64, 17)])
@pytest.mark.parametrize("kind", [W.LOSS_L1, W.LOSS_QUANTILE])
def test_one_kind(G, oracle_mod, kind, m, n, p_obs):
    check(G, oracle_mod, table(np.full(n, kind), m, 6, p_obs, 8100 + kind + m), p_obs == 1.0)


@pytest.mark.parametrize("p_obs", [0.6, 1.0])
def test_groups_beside_other_kinds(G, oracle_mod, p_obs):
    kinds = np.repeat([W.LOSS_L1, W.LOSS_HUBER, W.LOSS_QUANTILE, W.LOSS_HINGE, W.LOSS_L1], 32)[:150]
    check(G, oracle_mod, table(kinds, 150, 20, p_obs, 8200), p_obs == 1.0)
