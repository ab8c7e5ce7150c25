"""The FP32 contraction's schedule at its edges, against the FP64 oracle: shells
that leave octets and works partly filled, row lists of one block and of more
than one work's rows, point counts that leave the last 64-point block ragged,
and the number of segments.

Tolerance: a sum's FP32 error is at most (64 + 1) 2^-24 (its 64-point chains and
the product) plus 3 x 2^-20 (three fields from five-stage FP32 transforms, a few
2^-24 a stage) of the sum of its terms' magnitudes, together 6.8e-6; that sum is
at most sqrt(points x the sum of the squared terms), which the oracle returns.
A shell on which L_l vanishes (n^2 = 3 alone, l = 2) has no terms of its own: the
FP32 weight's rounding is relative to 2 l + 1, so the magnitudes are those of
the l = 0 terms times 2 l + 1."""
import ctypes

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


# n: 18^3 and 10^3 are no multiples of 64 points; shells 1, 8, 9, 17, 20: around the
# octets of shells; the full tensor with 20 shells has row lists longer than 56
@pytest.mark.parametrize("n,shells,width,ells,full", [(10, 1, 2.0, (0,), False), (18, 8, 1.0, (0, 2, 4), False),
                                                      (18, 9, 0.8, (2, 4), False), (24, 17, 0.6, (0, 2), False),
                                                      (24, 20, 0.5, (0, 2, 4), True)])
def test_fp32_edges(torch_cuda, ora, n, shells, width, ells, full):
    from paper_1708_05303_gb300 import bsp

    edges = linear_edges(shells, width)
    dk, _ = make_field(FieldModel(n=n, box=BOX, sigma_g=0.3), 31 + n)
    est = bsp.Bispectrum(n, BOX, edges, ells, full_tensor=full)
    d = torch_cuda.from_numpy(dk).cuda()
    est.compute(d)
    T = est.raw().cpu().numpy()
    r = ora.bispectrum(dk.astype(np.complex128), n, BOX, edges, ells, bins=[tuple(t) for t in est.bins])
    r0 = ora.bispectrum(dk.astype(np.complex128), n, BOX, edges, (0,), bins=[tuple(t) for t in est.bins])
    scale = np.sqrt(float(n) ** 3 * r0["sumsq"]) * (2 * np.array(ells)[:, None] + 1)
    assert np.max(np.abs(T - r["T"]) / scale) <= 6.8e-6
    # another number of segments sums the same 64-point blocks, each folded into a
    # compensated pair: 2^-46 of the magnitudes at most
    assert bsp.load().bsp_plan_tune(ctypes.c_void_p(est.plan), 3, 0) == 0
    est.compute(d)
    assert np.max(np.abs(est.raw().cpu().numpy() - T) / scale) <= 2.0 ** -46
    est.close()
