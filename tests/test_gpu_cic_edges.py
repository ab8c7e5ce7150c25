"""The particle deposit at its edges, against the FP64 oracle at the density tests'
gate (1e-4 of the modes' rms): rows whose length is no multiple of the 16-byte
reductions, cell and half-cell boundaries and their neighbours in FP32, the wrap
on every axis, and positions outside the box (the FP64 path)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
BOX = 1000.0


@pytest.fixture(scope="module")
def torch_cuda():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_05303_gb300 import build

    build.build()
    return torch


@pytest.mark.parametrize("n", [10, 18, 24, 50])
@pytest.mark.parametrize("outside", [False, True])
def test_cic_edges(torch_cuda, ora, n, outside):
    from paper_1708_05303_gb300 import bsp

    rng = np.random.default_rng(n)
    half = np.arange(2 * n) * (BOX / (2 * n))
    edge = np.concatenate([half, np.nextafter(half.astype(np.float32), np.float32(BOX)),
                           np.nextafter(half.astype(np.float32)[1:], np.float32(0)), [np.nextafter(np.float32(BOX), 0)]])
    pos = np.concatenate([rng.choice(edge, (4000, 3)), rng.random((4000, 3)) * BOX]).astype(np.float32)
    pos = np.minimum(pos, np.nextafter(np.float32(BOX), np.float32(0)))
    if outside:
        pos[::3, 0] += np.float32(BOX)
        pos[1::3, 1] -= np.float32(2 * BOX)
        pos[::5, 2] = -pos[::5, 2]
    d, _ = bsp.density_from_particles(torch_cuda.from_numpy(pos).cuda(), n, BOX)
    ref, _ = ora.density_from_particles(pos.astype(np.float64), n, BOX)
    assert np.max(np.abs(d.cpu().numpy() - ref)) <= 1e-4 * np.sqrt(np.mean(np.abs(ref) ** 2))
