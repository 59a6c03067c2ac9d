"""Rounding of the dense form's gradient sums on the tensor core.  With A = 0,
quadratic loss and positive factors every term of dF/dX = 2 X (Y^T Y) is positive:
each addition to the accumulator may lose one unit, 2^-23, of a sum that only
grows, on average half a unit of half of the final sum.  608 tiles of 128 rows are
one work item each, 32 chunks of 64 columns, and the products of the high parts
take 4 additions a chunk: 128 in all.  The products of the lower parts, 2^-8 of
the sum, and the products U add less than 8 units more.  (One accumulator for all
six products takes 768 additions.)"""
import pytest
import torch

pytestmark = pytest.mark.gpu

M, N = 128 * 608, 2048


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1410_0342_gb300 import build
    build.build()
    from paper_1410_0342_gb300 import glrm
    return glrm


@pytest.mark.parametrize("k", [12, 16, 20, 32, 33, 48])
def test_sums_of_positive_terms(G, k):
    gen = torch.Generator(device="cuda").manual_seed(k)
    X = torch.rand(M, k, generator=gen, device="cuda") + 0.5
    Yt = torch.rand(N, k, generator=gen, device="cuda") + 0.5
    zero = torch.zeros(N).numpy()
    g = G.GLRM(M, N, k, (zero, zero, zero), (0, 0.0), (0, 0.0))
    g.set_dense(torch.zeros(M, N, device="cuda"))
    g.set_factors(X, Yt)
    got = g.grad()[0].double()
    want = 2 * X.double() @ (Yt.double().T @ Yt.double())
    err = ((got - want).abs() / want) * 2.0 ** 23
    assert err.max().item() <= 4 * 32 + 8
    assert err.mean().item() <= 4 * 32 / 4 + 8
