"""The covariance through exact integer products on the tensor cores, against
quad- or extended-precision sums of the same centred values, at the edges of its
tiles (128 x 64 columns), mock chunks (32) and drain groups (512), and on
columns that it multiplies directly (not finite, denormal, out of range).

Tolerance per entry: half a unit of the last place for the single rounding and
one for the reciprocal of M - 1 (2^-52 |C|), and per mock 2^-53 of the product
of the columns' largest magnitudes: the digits dropped are at most 7 x 2^12 of
2^54 (their scale is at most twice the magnitude, squared), and each value's
rounding to 55 bits 2^-56 twice."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_05303_gb300 import build

    build.build()
    return torch


@pytest.mark.parametrize("m,d", [(700, 256), (512, 321), (513, 300), (31, 1153), (33, 1152), (2, 4500), (1100, 257)])
def test_covariance_digits(torch_cuda, m, d):
    from paper_1708_05303_gb300 import bsp

    rng = np.random.Generator(np.random.PCG64(m * 7 + d))
    X = rng.standard_normal((m, d)) * np.exp(8 * rng.standard_normal(d)) + 3.0
    X[:, 1] = 0.25                       # no scatter at all
    X[:, 2] *= 1e-200                    # out of the digits' range: direct
    X[:, 3] = rng.standard_normal(m) * 1e150
    X[m - 1, 4] = 1e6 * X[0, 4]          # one outlying mock
    X[:, d - 1] = -X[:, 0]
    mean, cov = bsp.Batch.covariance(torch_cuda.from_numpy(X).cuda())
    mean, cov = mean.cpu().numpy(), cov.cpu().numpy()
    assert np.allclose(mean, X.mean(axis=0), rtol=1e-13, atol=1e-13 * np.abs(X).max(axis=0))
    assert np.array_equal(cov, cov.T)
    y = X - mean
    cols = np.unique(np.concatenate([[0, 1, 2, 3, 4, 63, 64, 127, 128, 255, d - 1], rng.integers(0, d, 20)]))
    yl = y[:, cols].astype(np.longdouble)
    top = np.abs(y[:, cols]).max(axis=0)
    ref = np.array([[np.sum(yl[:, a] * yl[:, b]) / (m - 1) for b in range(len(cols))] for a in range(len(cols))])
    tol = 2.0 ** -52 * np.abs(ref) + 2.0 ** -53 * m / (m - 1) * np.outer(top, top) + 1e-300
    assert np.all(np.abs(cov[np.ix_(cols, cols)] - ref) <= tol)


def test_covariance_not_finite(torch_cuda):
    from paper_1708_05303_gb300 import bsp

    m, d = 600, 300
    rng = np.random.Generator(np.random.PCG64(5))
    X = rng.standard_normal((m, d))
    X[3, 7] = np.nan
    X[4, 9] = np.inf
    X[:, 11] = 5e-324 * rng.integers(0, 9, m)
    _, cov = bsp.Batch.covariance(torch_cuda.from_numpy(X).cuda())
    cov = cov.cpu().numpy()
    bad = np.zeros(d, bool)
    bad[[7, 9]] = True
    assert np.isnan(cov[bad]).all() and np.isnan(cov[:, bad]).all()
    rest = np.ix_(~bad, ~bad)
    assert np.allclose(cov[rest], np.cov(X[:, ~bad], rowvar=False), rtol=1e-9, atol=1e-12)
