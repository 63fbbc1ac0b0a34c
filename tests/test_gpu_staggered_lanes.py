"""The staggered stencil with four lanes per site (small half-volumes) gives the bits of one
lane per site: a lattice of two copies along periodic t has twice the sites and runs the other
form, and repeats the small lattice's result."""
import pytest

from helpers import F16, F32, F64

pytestmark = pytest.mark.gpu


# the last half-volumes of four lanes (8192 FP64, 16384 FP32 / FP16) and ragged ones below
@pytest.mark.parametrize("prec,dims", [(F64, (8, 8, 16, 16)), (F64, (6, 10, 14, 18)), (F32, (16, 16, 16, 8)),
                                       (F32, (10, 14, 14, 14)), (F16, (16, 16, 8, 16)), (F16, (14, 10, 14, 16))])
@pytest.mark.parametrize("recon", [18, 12, 8])
def test_lanes_equal_one(dirac, prec, dims, recon):
    import torch
    from paper_1109_2935_gb300 import synth
    fat, lng = synth.asqtad_links(dims, 1, 2, device="cuda")
    psi = synth.staggered_spinor(dims, 3, device="cuda")
    out = []
    for n in (1, 2):
        lat = dirac.Lattice(dims[:3] + (n * dims[3],), dirac.ASQTAD, mass=0.01, t_antiperiodic=False,
                            recon=(recon,) * 3, prec_mask=1 << prec)
        lat.load_gauge(torch.cat([fat] * n), 1)
        lat.load_gauge(torch.cat([lng] * n), 2)
        x = lat.to_device(torch.cat([psi] * n), prec)
        y = lat.new_field(prec)
        lat.apply(y, x, dirac.PARITY_FULL, prec)
        out.append(lat.to_natural(y, prec))
    assert torch.equal(torch.cat([out[0]] * 2), out[1])
