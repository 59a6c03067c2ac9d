"""The work items of the batched form: many sweeps in one persistent launch,
where every factor row is written and read again by other SMs of the same
launch, give the bits of one launch per sweep; systems that cannot be factorised
are reported as such and leave the other instances alone."""
import numpy as np
import pytest
import torch

from paper_1410_0342_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1410_0342_gb300 import build
    build.build()
    from paper_1410_0342_gb300 import glrm
    return glrm


@pytest.mark.parametrize("count,m_range,n_range", [(2, (4000, 5000), (400, 500)), (48, (50, 2500), (20, 400))])
def test_sweeps_of_one_launch_are_those_of_many(G, count, m_range, n_range):
    wb = W.batch_torch(count, device="cuda", m_range=m_range, n_range=n_range)
    meth = [G.GLRM_BATCH_ALS if s % 2 == 0 else G.GLRM_BATCH_PROXGRAD for s in range(count)]
    T = 16
    one, many = G.Batch(wb, meth), G.Batch(wb, meth)
    h1 = one.sweep(T, mode=G.GLRM_BATCH_STREAM)
    h2 = np.concatenate([many.sweep(1, mode=G.GLRM_BATCH_STREAM) for _ in range(T)])
    np.testing.assert_array_equal(h1, h2)
    for a, b in zip(one.factors() + one.steps(), many.factors() + many.steps()):
        assert torch.equal(a, b)


def test_failed_systems_leave_the_others(G):
    """One ALS instance whose factors are not finite among others, several sweeps
    in one launch: GLRM_ERR_NONFINITE, and every other instance as without it."""
    wb = W.batch_torch(24, device="cuda", m_range=(50, 1500), n_range=(20, 300))
    meth = [G.GLRM_BATCH_ALS if s % 2 == 0 else G.GLRM_BATCH_PROXGRAD for s in range(wb.count)]
    good = G.Batch(wb, meth)
    good.sweep(6, mode=G.GLRM_BATCH_STREAM)
    want = good.factors()
    bad = 4
    x0, y0 = int((wb.m * wb.k)[:bad].sum()), int((wb.n * wb.k)[:bad].sum())
    x1, y1 = x0 + int(wb.m[bad] * wb.k[bad]), y0 + int(wb.n[bad] * wb.k[bad])
    Yt = wb.Yt0.clone()
    Yt[y0:y1] = float("inf")
    B = G.Batch(wb, meth)
    B.set_factors(wb.X0, Yt)
    with pytest.raises(G.GLRMError) as e:
        B.sweep(6, mode=G.GLRM_BATCH_STREAM)
    assert e.value.code == G.GLRM_ERR_NONFINITE
    X, Yt = B.factors()
    for got, ref, a, b in ((X, want[0], x0, x1), (Yt, want[1], y0, y1)):
        got, ref = got.clone(), ref.clone()
        got[a:b] = ref[a:b] = 0.0
        assert torch.equal(got, ref)
