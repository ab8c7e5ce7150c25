"""Particles a hair below 0 (the wrap rounds them to the far edge of the box, which is cell
0), against the FP64 oracle at the density tests' gate (1e-4 of the modes' rms)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
BOX = 1000.0


@pytest.mark.parametrize("n", [10, 64])
def test_tiny_negative_positions(ora, n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_05303_gb300 import build, bsp

    build.build()
    rng = np.random.default_rng(n)
    pos = (rng.random((2000, 3)) * BOX).astype(np.float32)
    pos = np.minimum(pos, np.nextafter(np.float32(BOX), np.float32(0)))
    tiny = np.array([-1e-15, -1e-20, -1e-30, -1e-40, -1e-12, -1e-6, -0.0], dtype=np.float32)
    for a in range(3):
        pos[a * 200:(a + 1) * 200, a] = rng.choice(tiny, 200)
    pos[600:620] = rng.choice(tiny, (20, 3))
    d, _ = bsp.density_from_particles(torch.from_numpy(pos).cuda(), n, BOX)
    ref, _ = ora.density_from_particles(pos.astype(np.float64), n, BOX)
    assert np.max(np.abs(d.cpu().numpy() - ref)) <= 1e-4 * np.sqrt(np.mean(np.abs(ref) ** 2))
