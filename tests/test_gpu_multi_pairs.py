"""Two right-hand sides per thread give the bits of one application each: even and odd counts,
half-volumes that are and are not a multiple of a warp, planned and unplanned launches."""
import pytest

from helpers import F16, F32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(12, 12, 12, 20), (10, 10, 14, 18), (2, 6, 18, 50)])
@pytest.mark.parametrize("prec,nrhs", [(F32, 7), (F32, 12), (F16, 9), (F16, 14), (F16, 16)])
@pytest.mark.parametrize("csw", [1.0, 0.0])
def test_multi_equals_single(dirac, dims, prec, nrhs, csw):
    import torch
    from paper_1109_2935_gb300 import synth
    lat = dirac.Lattice(dims, dirac.WILSON_CLOVER, kappa=0.124, csw=csw, prec_mask=1 << prec)
    lat.load_gauge(synth.wilson_gauge(dims, 0.5, 0, 81, device="cuda"))
    n = lat.field_bytes(prec)
    x = torch.cat([lat.to_device(synth.wilson_spinor(dims, 90 + r, device="cuda"), prec) for r in range(nrhs)])
    ref, y, z = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x)
    for r in range(nrhs):
        lat.apply(ref[r * n:(r + 1) * n], x[r * n:(r + 1) * n], dirac.PARITY_FULL, prec)
    lat.apply_multi(y, x, nrhs, prec)
    plan = dirac.Batch([lat], [z], [x], [nrhs], prec)
    if prec == F16:
        plan.set_tensor_cores(False)
    z.zero_()
    plan.apply()
    torch.cuda.synchronize()
    assert torch.equal(y, ref)
    assert torch.equal(z, ref)
