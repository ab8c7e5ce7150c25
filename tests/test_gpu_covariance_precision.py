"""What the covariance's digit products keep, entry by entry against exact sums (extended
or quad precision) of the same centred values.

Outlying mocks in different columns must not cost the other mocks their bits: every
entry within the bound of an FP64 sum of its products, (m + 1) 2^-53 of the sum of
their magnitudes (m - 1 fused additions, the division, the entry's own rounding).
Columns of one magnitude, signs alternating, whose digits lose the most: every mock's
loss has the same sign, and the sum is within the stated bound: 9.1 x 2^-64 of
2^(e_i + e_j) per mock (digit products left out, at most 7 x 2^14 x 2^48 of 2^126 on
the first level left out, 6 x 2^14 x 2^40 on the second, ...: 7.03 x 2^-64; half a unit of 2^-63
for each value's rounding times the other value: 2 x 2^-64) and one rounding, 2^-53 of
the entry and 2^-10 of that."""
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


def covariance(torch, X):
    from paper_1708_05303_gb300 import bsp

    mean, cov = bsp.Batch.covariance(torch.from_numpy(X).cuda())
    return mean.cpu().numpy(), cov.cpu().numpy()


@pytest.mark.parametrize("m", [100, 200, 640])
@pytest.mark.parametrize("size", [30.0, 1e3, 1e6, 1e12])
@pytest.mark.parametrize("opposite", [False, True])
def test_outlying_mocks(torch_cuda, m, size, opposite):
    d = 130
    rng = np.random.Generator(np.random.PCG64(int(size) % 1000 + m))
    X = rng.standard_normal((m, d))
    out = [1, 2, 40, 63, 64, 100, 129]
    for k, j in enumerate(out):          # every column another mock (and its mirror image)
        X[3 * k, j] += size
        if opposite:
            X[3 * k + 1, j] -= size
    X[:, 7] = X[:, 8] * X[:, 9] * X[:, 10]   # heavy tails of its own
    mean, cov = covariance(torch_cuda, X)
    y = (X - mean).astype(np.longdouble)
    for a in out + [0, 7, 65]:
        p = y[:, a, None] * y
        ref, tol = p.sum(axis=0) / (m - 1), (m + 1) * 2.0 ** -53 * np.abs(p).sum(axis=0) / (m - 1)
        assert np.all(np.abs(cov[a] - ref) <= tol)


def value(digits, bits):
    v = 0
    for g in digits:
        v = (v << bits) + g
    return v


def test_digits_that_lose_the_most(torch_cuda):
    m = 512
    sign = np.where(np.arange(m) % 2, -1.0, 1.0)
    v = [value([64] + [-128] * 6 + [0], 8), value([127] + [-128] * 5 + [0, 0], 8), value([33] + [-64] * 7, 7) << 8,
         value([65] + [127] * 5 + [0, 0], 8), (1 << 62) + (1 << 10), (1 << 63) - (1 << 10), value([100] + [-128, 127] * 2 + [-128, 0, 0], 8)]
    assert all(int(float(q)) == q for q in v)   # 53 bits
    X = sign[:, None] * np.array([float(q) for q in v])[None, :] * 2.0 ** np.arange(-3, 4)[None, :]
    X = np.concatenate([X, X[:, ::-1]], axis=1)
    mean, cov = covariance(torch_cuda, X)
    assert np.all(mean == 0)
    e = np.frexp(np.abs(X[0]))[1].astype(float)
    for a in range(X.shape[1]):
        ref = X[0, a].astype(np.longdouble) * X[0] * m / (m - 1)
        tol = 2.0 ** -53 * (1 + 2.0 ** -10) * np.abs(ref) + 9.1 * 2.0 ** -64 * m / (m - 1) * 2.0 ** (e[a] + e)
        assert np.all(np.abs(cov[a] - ref) <= tol)


@pytest.mark.parametrize("m", [128, 129, 512, 1500])
def test_no_further_off_than_the_direct_path(torch_cuda, m):
    from paper_1708_05303_gb300 import bsp

    torch, d = torch_cuda, 96
    rng = np.random.Generator(np.random.PCG64(m))
    X = rng.standard_normal((m, d)) * np.exp(3 * rng.standard_normal(d))
    X[:, ::4] *= rng.standard_normal((m, d // 4)) * rng.standard_normal((m, d // 4))
    X[:, 1::4] = X[:, 1::4] ** 2
    x = torch.from_numpy(X).cuda()
    mean, direct = torch.empty(d, dtype=torch.float64, device="cuda"), torch.empty((d, d), dtype=torch.float64, device="cuda")
    assert bsp.load().bsp_covariance(m, d, x.data_ptr(), mean.data_ptr(), direct.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream) == 0
    worst = []
    for mu, cov in ((mean.cpu().numpy(), direct.cpu().numpy()), covariance(torch, X)):
        y = (X - mu).astype(np.longdouble)
        w = 0.0
        for a in range(0, d, 5):
            p = y[:, a, None] * y
            w = max(w, float(np.max(np.abs(cov[a] * np.longdouble(m - 1) - p.sum(axis=0)) / np.abs(p).sum(axis=0))))
        worst.append(w)
    print(m, worst)
    assert worst[1] <= worst[0]
