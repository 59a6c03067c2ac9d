"""FP32 tables below the dense form's density that the automatic choice takes
to the chunked half-steps: long columns before masked tiles, rows and columns
of 8 entries or more before the fused and blocked forms; those it leaves (short
rows, rows of a larger odd rank, shorter columns of a masked table); all
against the oracle."""
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


@pytest.mark.parametrize("m,n,k,p,paths", [
    (14_000, 70, 6, 0.33, "MC"),   # columns of 4,620 entries
    (12_000, 64, 8, 0.33, "MS"),   # of 3,960
    (12_000, 70, 6, 0.33, "MC"),   # too long a factor to stage, no rank to gather by
    (4_000, 220, 12, 0.18, "CC"),  # rows of 40, columns of 720
    (4_000, 220, 16, 0.04, "CC"),  # rows of 9
    (4_000, 220, 16, 0.03, "FC"),  # rows of 7
    (4_000, 220, 15, 0.18, "CC"),
    (4_000, 220, 17, 0.18, "FC"),
    (260, 4_000, 10, 0.2, "CC")])  # rows of 800 over a factor in panels
def test_choice_and_parity(G, oracle_mod, m, n, k, p, paths):
    t = W.small_mixed(m=m, n=n, k=k, p_obs=p, seed=7600 + k, rx=(RQ, 0.05), ry=(RL1, 0.02))
    g = G.GLRM.from_table(t)
    names = {"M": G.GLRM_PATH_MASKED, "S": G.GLRM_PATH_MASKED_SPLIT, "C": G.GLRM_PATH_CHUNKED, "F": G.GLRM_PATH_FUSED}
    want = [names[c] for c in paths]
    got = G.glrm_get_path(g.h)
    assert all(a == b or (b == names["M"] and a == names["S"]) for a, b in zip(got, want))
    synced_sweeps(g, oracle_mod, t, 2)
