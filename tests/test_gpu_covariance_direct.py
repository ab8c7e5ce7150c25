"""Columns that the covariance multiplies directly beside the digit products: a few
scattered ones (gathered, 32 to a tile), and all of them, where the call must cost
what the direct path alone costs.

Tolerance per entry: an FP64 sum of m products is within m 2^-53 of the sum of their
magnitudes (m - 1 additions, each fused with its product), and the division by m - 1
adds one rounding; two units of m 2^-53 cover both."""
import ctypes

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


@pytest.mark.parametrize("m,d,count", [(120, 33, 1), (130, 200, 5), (200, 1153, 40), (200, 300, 150), (200, 300, 151), (150, 97, 97)])
def test_direct_columns(torch_cuda, m, d, count):
    from paper_1708_05303_gb300 import bsp

    rng = np.random.Generator(np.random.PCG64(m + d + count))
    X = rng.standard_normal((m, d)) + 1.0
    direct = np.sort(rng.choice(d, count, replace=False))
    X[:, direct] *= np.where(np.arange(count) % 2, 1e-140, 1e140)   # out of the digits' range
    mean, cov = bsp.Batch.covariance(torch_cuda.from_numpy(X).cuda())
    mean, cov = mean.cpu().numpy(), cov.cpu().numpy()
    assert np.array_equal(cov, cov.T)
    y = (X - mean).astype(np.longdouble)
    cols = np.unique(np.concatenate([direct[:3], direct[-3:], rng.integers(0, d, 12)]))
    rows = np.unique(np.concatenate([direct[:40], direct[-3:]]))
    for a in rows:
        ref = (y[:, a, None] * y[:, cols]).sum(axis=0) / (m - 1)
        tol = 2 * m * 2.0 ** -53 * np.abs(y[:, a, None] * y[:, cols]).sum(axis=0) / (m - 1)
        assert np.all(np.abs(cov[a, cols] - ref) <= tol)


def test_all_direct_costs_the_direct_path(torch_cuda):
    from paper_1708_05303_gb300 import bsp

    torch = torch_cuda
    m, d = 600, 2000
    X = np.random.Generator(np.random.PCG64(1)).standard_normal((m, d))
    X[5] = np.nan                        # one mock that is not finite: no column is the digits'
    x = torch.from_numpy(X).cuda()
    lib = bsp.load()
    mean, cov = torch.empty(d, dtype=torch.float64, device="cuda"), torch.empty((d, d), dtype=torch.float64, device="cuda")
    nb = ctypes.c_size_t()
    assert lib.bsp_covariance_workspace_size(m, d, ctypes.byref(nb)) == 0 and nb.value > 0
    ws = torch.empty(nb.value, dtype=torch.uint8, device="cuda")
    st = torch.cuda.current_stream().cuda_stream

    def time(call):
        best = 1e9
        for _ in range(4):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record()
            assert call() == 0
            e[1].record()
            torch.cuda.synchronize()
            best = min(best, e[0].elapsed_time(e[1]))
        return best

    direct = time(lambda: lib.bsp_covariance(m, d, x.data_ptr(), mean.data_ptr(), cov.data_ptr(), st))
    both = time(lambda: lib.bsp_covariance_ws(m, d, x.data_ptr(), mean.data_ptr(), cov.data_ptr(), ws.data_ptr(), nb.value, st))
    print("direct %.3f ms, with a workspace %.3f ms" % (direct, both))
    assert torch.isnan(cov).all()
    assert both <= 1.5 * direct
