"""A tensor-core call whose waits run out must not return numbers: its partial sums may be
an earlier call's.  With a wait limit of 200 cycles every output is NaN, and with the
default limit the plan gives its bits again."""
import numpy as np
import pytest

from paper_1708_05303_gb300.synth import FieldModel, linear_edges, make_field

pytestmark = pytest.mark.gpu
BOX = 1000.0


@pytest.mark.parametrize("kind", ["bispectrum", "modal"])
def test_outputs_are_nan(kind):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1708_05303_gb300 import build, bsp

    build.build()
    n, kf = 32, 2 * np.pi / BOX
    dk, amp = make_field(FieldModel(n=n, box=BOX, sigma_g=0.3), 11)
    d = torch.from_numpy(dk).cuda()
    if kind == "bispectrum":
        est = bsp.Bispectrum(n, BOX, linear_edges(8), (0, 2, 4), prec="split_f16")
    else:
        est = bsp.Modal(n, BOX, bsp.bsp_modal_radial_powerlaw(n, BOX, 6, kf, 14 * kf, amp, -1.5, True), (0, 2, 4), prec="split_f16")
    before = est.compute(d).clone()
    assert torch.isfinite(before).all()
    bsp.bsp_set_wait_limit(est.plan, 200)
    after = est.compute(d).clone()
    torch.cuda.synchronize()
    assert bsp.bsp_device_status(est.plan) != 0
    assert torch.isnan(after).all()
    bsp.bsp_set_wait_limit(est.plan, 0)
    assert torch.equal(est.compute(d), before)
    est.close()
