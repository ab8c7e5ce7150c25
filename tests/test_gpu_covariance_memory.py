"""A covariance whose digit workspace does not fit beside the matrix is still computed:
under an allocation limit that lets the results through and not the workspace, the call
must give what the direct path gives, bit for bit."""
import pytest

pytestmark = pytest.mark.gpu


def test_falls_back_to_the_direct_path():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_05303_gb300 import build, bsp

    build.build()
    m, d = 6000, 1500
    rows = torch.randn((m, d), dtype=torch.float64, device="cuda")
    mean, cov = torch.empty(d, dtype=torch.float64, device="cuda"), torch.empty((d, d), dtype=torch.float64, device="cuda")
    assert bsp.load().bsp_covariance(m, d, rows.data_ptr(), mean.data_ptr(), cov.data_ptr(),
                                     torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    try:
        # room for the 18 MB of results, not for the 147 MB of digits
        torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + 64 * 2 ** 20) / total)
        got = bsp.Batch.covariance(rows)
    finally:
        torch.cuda.set_per_process_memory_fraction(1.0)
    assert torch.equal(got[0], mean) and torch.equal(got[1], cov)
