"""Row loads and sums of the chunked passes at their edges: odd ranks (scalar
loads), even ranks (pairs), multiples of 4 (16-byte units), factors at
addresses that allow neither; one loss for all columns and several; chunk
counts that leave a block's last warps idle; segments of 0, 1, 31..33, 64 and
1,025 entries; FP64 at the ranks without padding."""
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


def table(k, longest, seed, nkinds):
    rng = W.rng_for(seed)
    lens = [0, 1, 31, 32, 33, 63, 64, 65, longest] + [int(v) for v in rng.integers(0, 70, 84)]
    m, n = len(lens), 1100
    rowptr = np.concatenate([[0], np.cumsum(lens)])
    colidx = np.concatenate([np.sort(rng.choice(n, c, replace=False)) for c in lens]).astype(np.int32)
    sd = k ** -0.25
    u = W.sampled_products(rng.standard_normal((m, k)) * sd, rng.standard_normal((n, k)) * sd, rowptr, colidx)
    kinds = np.arange(n) % nkinds
    val = np.where(kinds[colidx] >= 2, np.where(u >= 0, 1.0, -1.0), u + 0.1 * rng.standard_normal(u.size))
    t = W._finish("rows", m, n, k, rowptr, colidx, val, kinds, np.where(kinds == 1, 1.0, 0.0), np.zeros(n),
                  (RQ, 0.05), (RL1, 0.02), rng, init_std=sd)
    t.X0, t.Yt0 = (np.asarray(a, np.float32).astype(np.float64) for a in (t.X0, t.Yt0))
    return t


def shifted(a):
    """A contiguous copy 4 bytes beyond a 16-byte boundary."""
    b = torch.empty(a.numel() + 1, dtype=a.dtype, device=a.device)[1:].view(a.shape)
    b.copy_(a)
    return b


@pytest.mark.parametrize("longest,nkinds", [(64, 4), (1025, 1), (1025, 4)])
@pytest.mark.parametrize("k", [1, 2, 4, 6, 7, 10, 18, 20, 30, 32])
def test_sweeps_and_gradients(G, oracle_mod, k, longest, nkinds):
    t = table(k, longest, 7400 + k, nkinds)
    g = G.GLRM.from_table(t)
    G.glrm_set_path(g.h, 1, 1)
    p = oracle_problem(oracle_mod, t)
    gx, gy = p.gradient(t.X0, t.Yt0)
    sx, sy, vx, vy = grad_bounds(p, t.X0, t.Yt0)
    X, Yt = (torch.tensor(a, dtype=torch.float32, device="cuda") for a in (t.X0, t.Yt0))
    for at in (lambda a: a, shifted):
        GX, GYt = torch.empty_like(X), torch.empty_like(Yt)
        G.glrm_grad_at(g.h, at(X), at(Yt), GX, GYt, False)
        assert_grad_close(GX.cpu().numpy(), gx, sx, vx, what="dF/dX")
        assert_grad_close(GYt.cpu().numpy(), gy, sy, vy, what="dF/dYt")
    synced_sweeps(g, oracle_mod, t, 2)


@pytest.mark.parametrize("k", [3, 4, 5, 6, 7, 8])
def test_fp64_small_ranks(G, oracle_mod, k):
    t = table(k, 64, 7500 + k, 4)
    g = G.GLRM.from_table(t, precision=G.GLRM_FP64)
    G.glrm_set_path(g.h, 1, 1)
    p = oracle_problem(oracle_mod, t)
    X, Yt = p.proxgrad(t.X0, t.Yt0, 3)[:2]
    g.sweep(3)
    for got, want in zip(g.factors(), (X, Yt)):
        assert np.linalg.norm(got.cpu().numpy() - want) <= 1e-10 * np.linalg.norm(want)
