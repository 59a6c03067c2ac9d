"""Segments of many partials (a CTA each from 16 on average): columns of 15,
16, 17 and 66 chunks in the chunked form, in FP32 and FP64, at ranks whose
partials fit one shared-memory batch and ranks that take several; the dense
form's columns of 33 items; sweeps and gradients against the oracle."""
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


def check_gradients(g, p, t):
    X, Yt = (np.asarray(a, np.float32).astype(np.float64) for a in (t.X0, t.Yt0))
    gx, gy = p.gradient(X, Yt)
    sx, sy, vx, vy = grad_bounds(p, X, Yt)
    GX, GYt = g.grad()
    assert_grad_close(GX.cpu().numpy(), gx, sx, vx, what="dF/dX")
    assert_grad_close(GYt.cpu().numpy(), gy, sy, vy, what="dF/dYt")


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("chunks,k", [(15, 7), (16, 7), (17, 33), (66, 64)])
def test_chunked_columns(G, oracle_mod, chunks, k, prec):
    t = W.small_mixed(m=chunks * 1024, n=6, k=k, p_obs=1.0, seed=7200 + k, rx=(RQ, 0.1), ry=(RL1, 0.1))
    t.X0, t.Yt0 = (np.asarray(a, np.float32).astype(np.float64) for a in (t.X0, t.Yt0))
    g = G.GLRM.from_table(t, precision=G.GLRM_FP64 if prec else G.GLRM_FP32)
    G.glrm_set_path(g.h, 1, 1)
    check_gradients(g, oracle_problem(oracle_mod, t), t)
    if not prec:
        synced_sweeps(g, oracle_mod, t, 2)


@pytest.mark.parametrize("k", [5, 64])
def test_dense_columns(G, oracle_mod, k):
    t = W.small_mixed(m=2100, n=100, k=k, p_obs=0.9, seed=7300 + k, rx=(RQ, 0.1), ry=(RQ, 0.1))
    t.X0, t.Yt0 = (np.asarray(a, np.float32).astype(np.float64) for a in (t.X0, t.Yt0))
    g = G.GLRM.from_table(t)
    assert G.glrm_get_path(g.h) == (G.GLRM_PATH_DENSE, G.GLRM_PATH_DENSE)
    check_gradients(g, oracle_problem(oracle_mod, t), t)
    synced_sweeps(g, oracle_mod, t, 2)
