"""A covariance on a side stream must not write memory that work queued on the current
stream still reads: blocks of its buffers' sizes are released while a copy of them
waits behind a long kernel, and the copy must see what was in them."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


def test_buffers_come_from_the_stream_that_writes_them():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_05303_gb300 import build, bsp

    build.build()
    m, d = 600, 1000
    rows = torch.randn((m, d), dtype=torch.float64, device="cuda")
    side = torch.cuda.Stream()
    want = bsp.Batch.covariance(rows)[1]
    nb = ctypes.c_size_t()
    assert bsp.load().bsp_covariance_workspace_size(m, d, ctypes.byref(nb)) == 0 and nb.value > 0
    victims = [torch.full((k,), 7, dtype=torch.uint8, device="cuda") for k in (nb.value, 8 * d * d, 8 * d)]
    copies = [torch.empty_like(v) for v in victims]
    torch.cuda.synchronize()
    torch.cuda._sleep(400_000_000)       # about 0.2 s
    for c, v in zip(copies, victims):
        c.copy_(v)
    del victims, v
    mean, cov = bsp.Batch.covariance(rows, stream=side)
    side.synchronize()
    assert torch.equal(cov, want)
    torch.cuda.synchronize()
    assert all(bool((c == 7).all()) for c in copies)
