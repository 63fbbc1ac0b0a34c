"""The one-lane staggered kernels keep nine CTAs per SM, whatever the links' form."""
import pytest

from helpers import F16, F32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [F32, F16])
def test_time_follows_the_bytes(dirac, prec):
    """18-real long links instead of 12-real ones are 1.2 times the bytes; on 24^4, near the size
    of L2, they took 1.7 (FP32) and 1.4 (FP16) times as long with seven and fewer CTAs per SM."""
    import torch
    from paper_1109_2935_gb300 import synth
    dims = (24, 24, 24, 24)
    fat, lng = synth.asqtad_links(dims, 1, 2, device="cuda")
    psi = synth.staggered_spinor(dims, 3, device="cuda")
    us = []
    for recon in (12, 18):
        lat = dirac.Lattice(dims, dirac.ASQTAD, mass=0.1, recon=(recon,) * 3, prec_mask=1 << prec)
        lat.load_gauge(fat, 1)
        lat.load_gauge(lng, 2)
        x, y = lat.to_device(psi, prec, 0), lat.new_field(prec, 0)
        start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        best = float("inf")
        for _ in range(8):
            start.record()
            for _ in range(50):
                lat.apply_normal(y, x, dirac.PARITY_EVEN, prec)
            end.record()
            torch.cuda.synchronize()
            best = min(best, start.elapsed_time(end) * 20)
        us.append(best)
    assert us[1] < 1.33 * us[0], us
