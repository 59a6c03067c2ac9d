"""The Gram kernel and the refined solve of an FP32 ALS half-step, row by row
against FP64 solves of the same systems: every padded width, rows without
entries, with one, around a batch of 32 and beyond one chunk of 1,024, and
systems too ill-conditioned for the FP32 preconditioner (they go to the FP64
factorisation).  The Gram matrix accumulates in FP32, so a row's solution may
move by its condition number times the rounding of that sum, c 2^-24 relative
for c entries, plus the FP32 rounding of the stored result."""
import numpy as np
import pytest
import torch

from paper_1410_0342_gb300 import workloads as W

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


@pytest.mark.parametrize("k,gamma,decay", [(1, 0.1, 1.0), (3, 0.1, 1.0), (4, 0.1, 1.0), (7, 0.1, 1.0), (8, 0.1, 1.0),
                                           (13, 0.1, 1.0), (16, 0.1, 1.0), (20, 0.1, 1.0), (32, 0.1, 1.0),
                                           (8, 1e-4, 0.05), (32, 1e-4, 0.5)])
def test_rows_match_fp64_solves(G, k, gamma, decay):
    rng = W.rng_for(4100 + k)
    lens = [0, 1, 31, 32, 33, 64, 200, 1023, 1024, 1025, 1500] + [int(v) for v in rng.integers(0, 90, 60)]
    m, n = len(lens), 1600
    rowptr = np.concatenate([[0], np.cumsum(lens)])
    colidx = np.concatenate([np.sort(rng.choice(n, c, replace=False)) for c in lens]).astype(np.int32)
    val = rng.standard_normal(colidx.size).astype(np.float32).astype(np.float64)
    t = W._finish("als", m, n, k, rowptr, colidx, val, np.zeros(n, np.int32), np.zeros(n), np.zeros(n),
                  (RQ, gamma), (RQ, gamma), rng)
    # decay < 1: the columns of Y shrink, the Gram matrices grow ill-conditioned
    Yt = (rng.standard_normal((n, k)) * decay ** np.arange(k)).astype(np.float32)
    g = G.GLRM.from_table(t, factors=False)
    G.glrm_set_path(g.h, 1, 1)
    g.set_factors(torch.zeros(m, k, device="cuda"), torch.as_tensor(Yt, device="cuda"))
    if k == 32 and gamma < 1e-3:
        # rounding the 32 x 32 Gram matrix to FP32 outweighs gamma here: the
        # call reports the systems that are not positive definite
        with pytest.raises(G.GLRMError):
            g.als_sweep(1)
        return
    g.als_sweep(1)
    X = g.factors()[0].double().cpu().numpy()
    Y = Yt.astype(np.float64)
    for i in range(m):
        s = slice(rowptr[i], rowptr[i + 1])
        w, a = Y[colidx[s]], val[s]
        gram = w.T @ w + gamma * np.eye(k)
        x = np.linalg.solve(gram, w.T @ a)
        # the rounding of both FP32 sums, in the norms that perturb the solution
        c = len(a) + 2
        db = c * 2.0 ** -24 * np.linalg.norm(np.abs(w).T @ np.abs(a))
        dg = c * 2.0 ** -24 * np.linalg.norm(np.abs(w).T @ np.abs(w))
        bound = np.linalg.norm(np.linalg.inv(gram), 2) * (db + dg * np.linalg.norm(x)) * 2 + 2.0 ** -23 * np.linalg.norm(x)
        assert np.linalg.norm(X[i] - x) <= bound, (i, len(a), np.linalg.norm(X[i] - x), bound)
