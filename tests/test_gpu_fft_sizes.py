"""The inverse transform over the radix lists its kernels meet (one stage to five,
radices 2 to 16, odd half lengths, lines that leave the last CTA partly filled)
through the skew spectrum and, pruned, through the bispectrum, against the FP64
oracle.  Gate: 1e-5 of the l = 0 values' rms times 2 l + 1, the size of the terms
that an l > 0 sum of few modes cancels (its own rms can be a hundredth of them)."""
import numpy as np
import pytest

from paper_1708_05303_gb300.synth import FieldModel, linear_edges, make_field

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


def gate(a, b):
    scale = np.sqrt(np.mean(b[0] ** 2)) * np.array([[1.0], [5.0], [9.0]])
    return np.max(np.abs(a - b) / np.maximum(np.abs(b), scale))


# n and n/2: 8 = 8, 4; 10 = 2 5, 5; 18 = 2 3 3, 9; 30, 15; 48, 24; 50, 25; 54, 27; 64 = 16 4, 8 4; 72; 96; 120 = 8 3 5
@pytest.mark.parametrize("n", [8, 10, 16, 18, 30, 48, 50, 54, 64, 72, 96, 120])
def test_inverse_transform_sizes(torch_cuda, ora, n):
    from paper_1708_05303_gb300 import bsp

    dk, _ = make_field(FieldModel(n=n, box=BOX, sigma_g=0.3), 300 + n)
    d = torch_cuda.from_numpy(dk).cuda()
    edges = linear_edges(2, n / 6)
    S, _ = bsp.Spectra(n, BOX, edges).skew(d)
    r = ora.skew_spectrum(dk.astype(np.complex128), n, BOX, edges)
    assert gate(S.cpu().numpy(), r["S"]) <= 1e-5
    for prec in ("fp32", "split_f16"):
        est = bsp.Bispectrum(n, BOX, edges, (0, 2, 4), prec=prec)
        B = est.compute(d).cpu().numpy()
        bins = [tuple(t) for t in est.bins]
        est.close()
        assert gate(B, ora.bispectrum(dk.astype(np.complex128), n, BOX, edges, bins=bins)["B"]) <= 1e-5


# large and small run-time sizes through the three users of the forward passes in turn: one
# kernel serves them all, and a small size must not take a large one's shared memory away
def test_run_time_sizes_in_turn(torch_cuda):
    from paper_1708_05303_gb300 import bsp

    torch = torch_cuda
    gen = torch.Generator(device="cuda").manual_seed(5)
    d = torch.randn(400, 400, 201, dtype=torch.complex64, device="cuda", generator=gen)
    spec = bsp.Spectra(400, BOX, linear_edges(4, 20.0))
    first = spec.skew(d)[0].cpu()
    pos = torch.rand(1000, 3, device="cuda", generator=gen) * BOX
    bsp.density_from_particles(pos, 216, BOX)
    spec.integrated(d, 2)
    assert torch.equal(spec.skew(d)[0].cpu(), first)
