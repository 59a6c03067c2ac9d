"""The dense form's logistic block cell by cell against 64 bits.  One cell of the
table has the product z (a BF16 value, so the tensor-core product is exact), all
others lie at z = -200, where loss and derivative are 0 in FP32: the objective is
that cell's loss, and a gradient coordinate its derivative times 1.

Bounds, in units of 2^-24: loss log(1 + e^z): an exponential and a logarithm good to
one unit in the last place (2 each), 4 in all.  Derivative: the exponential (2),
1 + e and the quotient (1 each), its split in three BF16 parts and their
FP32 accumulation on the tensor core (2 per addition), 8 in all.  Over many points
the errors of single operations add like independent ones: a rounding leaves
0.425 units in the root mean square (uniform over half a unit in the last place,
mantissas spread over their logarithm), three of them (exponential, logarithm,
sum) 0.74 in the loss, four (exponential, sum, quotient, accumulation) 0.85 in the
derivative."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

LOGISTIC = 3
M, N = 128, 16


@pytest.fixture(scope="module")
def G():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1410_0342_gb300 import build
    build.build()
    from paper_1410_0342_gb300 import glrm
    return glrm


def model(G, full, m, n):
    g = G.GLRM(m, n, 2, (np.full(n, LOGISTIC), np.zeros(n), np.zeros(n)), (0, 0.0), (0, 0.0))
    if full:
        g.set_dense(torch.ones(m, n, device="cuda"))
        return g
    # the last cell missing: the block that tests for missing values
    rowptr = np.arange(m + 1) * n
    rowptr[m] -= 1
    colptr = np.arange(n + 1) * m
    colptr[n] -= 1
    i32 = lambda v: torch.as_tensor(np.asarray(v), dtype=torch.int32, device="cuda")
    e = m * n - 1
    G.glrm_set_observed(g.h, e, i32(rowptr), i32(np.tile(np.arange(n), m)[:e]), torch.ones(e, device="cuda"),
                        i32(colptr), i32(np.tile(np.arange(m), n)[:e]), torch.ones(e, device="cuda"))
    assert G.glrm_get_path(g.h) == (G.GLRM_PATH_DENSE, G.GLRM_PATH_DENSE)
    return g


def points():
    """BF16 values of z from 2^-12 to 80, both signs."""
    rng = np.random.default_rng(3)
    v = np.ldexp(1 + rng.integers(0, 128, 400) / 128, rng.integers(-12, 7, 400))
    v = np.concatenate([v[v < 80], [0.34375, 0.34765625, 0.6875, 0.69140625, 1.0, 2.0]])
    return np.concatenate([v, -v])


def rel(got, want):
    return np.abs(np.asarray(got, np.float64) / want - 1)


@pytest.mark.parametrize("full", [True, False])
def test_losses(G, full):
    g = model(G, full, M, N)
    X = torch.tensor([200.0, 1.0], device="cuda").repeat(M, 1)
    Yt = torch.tensor([0.0, 200.0], device="cuda").repeat(N, 1)
    Yt[0] = torch.tensor([1.0, 0.0])
    z = points()
    got = []
    for v in z:
        X[0, 0] = -v  # a = 1: z = -u
        g.set_factors(X, Yt)
        got.append(g.objective())
    want = np.maximum(z, 0) + np.log1p(np.exp(-np.abs(z)))
    err = rel(got, want)
    assert err.max() <= 4 * 2.0 ** -24, (z[err.argmax()], err.max() * 2 ** 24)


@pytest.mark.parametrize("full", [True, False])
def test_derivatives(G, full):
    z = points()
    g = model(G, full, z.size, N)
    X = torch.ones(z.size, 2, device="cuda")
    X[:, 0] = torch.as_tensor(-z)
    Yt = torch.tensor([0.0, 200.0], device="cuda").repeat(N, 1)
    Yt[0] = torch.tensor([1.0, 0.0])
    g.set_factors(X, Yt)
    got = g.grad()[0][:, 0].double().cpu().numpy()
    want = -1 / (1 + np.exp(-z))
    err = rel(got, want)
    assert err.max() <= 8 * 2.0 ** -24, (z[err.argmax()], err.max() * 2 ** 24)


def test_root_mean_square(G):
    rng = np.random.default_rng(11)
    z = rng.uniform(-8, 8, 1 << 15).astype(np.float32)
    z = (z.view(np.uint32) & 0xffffff00).view(np.float32).astype(np.float64)  # two BF16 parts hold it
    Yt = torch.tensor([0.0, 200.0], device="cuda").repeat(N, 1)
    Yt[0] = torch.tensor([1.0, 0.0])
    g = model(G, True, z.size, N)
    X = torch.ones(z.size, 2, device="cuda")
    X[:, 0] = torch.as_tensor(-z)
    g.set_factors(X, Yt)
    err = rel(g.grad()[0][:, 0].double().cpu().numpy(), -1 / (1 + np.exp(-z)))
    assert np.sqrt((err ** 2).mean()) <= 0.85 * 2.0 ** -24
    z = z[:2000]
    g = model(G, True, M, N)
    X = torch.tensor([200.0, 1.0], device="cuda").repeat(M, 1)
    got = []
    for v in z:
        X[0, 0] = -v
        g.set_factors(X, Yt)
        got.append(g.objective())
    err = rel(got, np.maximum(z, 0) + np.log1p(np.exp(-np.abs(z))))
    assert np.sqrt((err ** 2).mean()) <= 0.74 * 2.0 ** -24


def test_far_tails_and_undefined_products(G):
    """exp(-|z|) below FP32: loss 0 or z, derivative 0 or -1; an undefined
    product gives an undefined objective."""
    z = np.array([-1e30, -1000.0, -100.0, 100.0, 1000.0, 1e30])
    g = model(G, True, z.size, N)
    X = torch.ones(z.size, 2, device="cuda")
    X[:, 0] = torch.as_tensor(-z)
    Yt = torch.tensor([0.0, 200.0], device="cuda").repeat(N, 1)
    Yt[0] = torch.tensor([1.0, 0.0])
    g.set_factors(X, Yt)
    got = g.grad()[0][:, 0].cpu().numpy()
    np.testing.assert_array_equal(got, np.where(z > 0, -1.0, 0.0))
    want = float(np.maximum(z, 0).astype(np.float32).astype(np.float64).sum())
    assert abs(g.objective() - want) <= 2.0 ** -23 * want
    X[0, 0] = float("nan")
    g.set_factors(X, Yt)
    assert np.isnan(g.objective())
