"""The one-launch chunked half-step (a warp per segment, taken where no
segment is longer than one chunk of 1,024 entries) at its edges: segments of
0, 1, 31..33, 1,023 and 1,024 entries, one longer segment switching that
orientation to the four launches, every lane layout, the offset and column
weights, and the automatic choice on a small fully observed FP64 table."""
import numpy as np
import pytest
import torch

from paper_1410_0342_gb300 import workloads as W

from gpu_parity import synced_sweeps

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


def table(k, longest, seed):
    rng = W.rng_for(seed)
    lens = [0, 1, 31, 32, 33, 1023, longest] + [int(v) for v in rng.integers(0, 70, 90)]
    m, n = len(lens), 1100
    rowptr = np.concatenate([[0], np.cumsum(lens)])
    colidx = np.concatenate([np.sort(rng.choice(n, c, replace=False)) for c in lens]).astype(np.int32)
    X0, Y0 = rng.standard_normal((m, k)), rng.standard_normal((n, k))
    u = W.sampled_products(X0, Y0, rowptr, colidx)
    kinds = np.arange(n) % 4
    val = np.where(kinds[colidx] >= 2, np.where(u >= 0, 1.0, -1.0), u + 0.1 * rng.standard_normal(u.size))
    return W._finish("seg", m, n, k, rowptr, colidx, val, kinds, np.where(kinds == 1, 1.0, 0.0), np.zeros(n),
                     (RQ, 0.05), (RL1, 0.02), rng, init_std=0.5)


@pytest.mark.parametrize("longest", [1024, 1025])
@pytest.mark.parametrize("k", [1, 4, 7, 20, 33, 64])
def test_segments_match_oracle(G, oracle_mod, k, longest):
    t = table(k, longest, 5200 + k)
    g = G.GLRM.from_table(t)
    G.glrm_set_path(g.h, 1, 1)
    G.glrm_timing_enable(g.h, True)
    synced_sweeps(g, oracle_mod, t, 3)
    names = set(G.glrm_timing_read(g.h))
    assert ("seg_x" in names) == (longest <= 1024) and ("pass_grad_x" in names) == (longest > 1024)
    assert "seg_y" in names


def test_segments_with_offset_and_weights(G, oracle_mod):
    t = table(9, 1024, 5300)
    w = np.linspace(0.5, 2.0, t.n).astype(np.float32).astype(np.float64)
    g = G.GLRM.from_table(t)
    G.glrm_set_path(g.h, 1, 1)
    g.set_offset(True)
    g.set_column_scale(w)
    synced_sweeps(g, oracle_mod, t, 3, offset=True, col_scale=w)


def test_small_fp64_table_takes_it(G, oracle_mod):
    t = W.qpca_dense()
    g = G.GLRM.from_table(t, precision=G.GLRM_FP64)
    assert G.glrm_get_path(g.h) == (G.GLRM_PATH_CHUNKED, G.GLRM_PATH_CHUNKED)
    hist = g.sweep(20)
    p = oracle_mod.Problem.from_csr(t.m, t.n, t.k, t.rowptr, t.colidx, t.val, loss_kind=t.loss_kind,
                                    loss_param=t.loss_param, loss_levels=t.loss_levels, rx=t.rx, ry=t.ry)
    ohist = p.proxgrad(t.X0, t.Yt0, 20)[4]
    assert (np.abs(hist - ohist) / np.abs(ohist)).max() < 1e-9
