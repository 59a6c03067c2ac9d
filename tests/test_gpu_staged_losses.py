"""The BF16 form's streamed gradient passes (k = 56 and 64) with losses that
differ from column to column, for segments of 0, 1, 7..9, 57, 63..65, 1,023 and
1,024 or 1,025 entries as rows and as columns: both gradients against the
oracle's at the rounded rows of the other factor."""
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


def table(k, longest, as_columns, seed):
    rng = W.rng_for(seed)
    lens = [0, 1, 7, 8, 9, 57, 63, 64, 65, 1023, longest] + [int(v) for v in rng.integers(0, 70, 80)]
    nseg, nother = len(lens), 1100
    seg = np.repeat(np.arange(nseg), lens)
    oth = np.concatenate([np.sort(rng.choice(nother, c, replace=False)) for c in lens])
    m, n = (nother, nseg) if as_columns else (nseg, nother)
    rows, cols = (oth, seg) if as_columns else (seg, oth)
    order = np.lexsort((cols, rows))
    rows, cols = rows[order], cols[order].astype(np.int32)
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(rows, minlength=m))])
    sd = k ** -0.25
    u = W.sampled_products(rng.standard_normal((m, k)) * sd, rng.standard_normal((n, k)) * sd, rowptr, cols)
    kinds = np.arange(n) % 4
    val = np.where(kinds[cols] >= 2, np.where(u >= 0, 1.0, -1.0), u + 0.1 * rng.standard_normal(u.size))
    val = val.astype(np.float32).astype(np.float64)
    t = W._finish("staged", m, n, k, rowptr, cols, val, kinds, np.where(kinds == 1, 1.0, 0.0), np.zeros(n),
                  (RQ, 0.05), (RQ, 0.05), rng, init_std=sd)
    t.X0, t.Yt0 = (np.asarray(a, np.float32).astype(np.float64) for a in (t.X0, t.Yt0))
    return t


@pytest.mark.parametrize("as_columns", [False, True])
@pytest.mark.parametrize("longest", [1024, 1025])
@pytest.mark.parametrize("k", [56, 64])
def test_gradients(G, oracle_mod, k, longest, as_columns):
    t = table(k, longest, as_columns, 8300 + k)
    g = G.GLRM.from_table(t, precision=G.GLRM_BF16)
    G.glrm_set_path(g.h, 1, 1)
    GX, GYt = g.grad()
    p = oracle_problem(oracle_mod, t)
    Xr, Yr = (torch.as_tensor(a).float().bfloat16().double().numpy() for a in (t.X0, t.Yt0))
    for X, Yt, got, q, what in ((t.X0, Yr, GX, 0, "dF/dX"), (Xr, t.Yt0, GYt, 1, "dF/dYt")):
        want, bounds = p.gradient(X, Yt)[q], grad_bounds(p, X, Yt)
        assert_grad_close(got.cpu().numpy(), want, bounds[q], bounds[2 + q], what=what)
