"""The work items of the batched form: many sweeps in one persistent launch,
where every factor row is written and read again by other SMs of the same
launch, give the bits of one launch per sweep."""
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
