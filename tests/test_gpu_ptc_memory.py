"""What training keeps allocated between calls is bounded."""
import pytest

from helpers import F32

pytestmark = pytest.mark.gpu


def test_long_loss_history_is_given_back(dirac):
    import torch
    from paper_1109_2935_gb300 import synth
    dims = (4, 4, 4, 4)
    lat = dirac.Lattice(dims, dirac.WILSON_CLOVER, kappa=0.12, csw=0.0, prec_mask=2)
    lat.load_gauge(synth.wilson_gauge(dims, 0.5, 0, 5, device="cuda"))
    v = [lat.to_device(synth.wilson_spinor(dims, 9, device="cuda"), F32)]
    net = dirac.Ptc(lat, (1, 1))
    net.train(v, steps=3, batch=1)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    assert len(net.train(v, steps=140_000, batch=1, lr=1e-6)) == 140_000  # 1.1 MB of losses
    torch.cuda.synchronize()
    assert torch.cuda.mem_get_info()[0] >= free


def test_large_sources_are_given_back(dirac):
    import torch
    from paper_1109_2935_gb300 import synth
    dims = (16, 16, 16, 16)
    lat = dirac.Lattice(dims, dirac.WILSON_CLOVER, kappa=0.12, csw=0.0, prec_mask=2)
    lat.load_gauge(synth.wilson_gauge(dims, 0.5, 0, 5, device="cuda"))
    v = [lat.to_device(synth.wilson_spinor(dims, 9, device="cuda"), F32)] * 50  # 50 sources of 6.3 MB
    net = dirac.Ptc(lat, (1, 1))
    net.train(v[:1], steps=1, batch=1)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    net.train(v, steps=1, batch=1)
    torch.cuda.synchronize()
    # the 6.3 MB of the first call went with the large buffer
    assert torch.cuda.mem_get_info()[0] >= free
