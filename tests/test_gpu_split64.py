"""The split-site FP64 stencil (lattices of at most 8192 output sites) gives the bits of the
one-thread-per-site stencil, which the multi-right-hand-side kernel runs at every size."""
import pytest

from helpers import F64

pytestmark = pytest.mark.gpu


# 16 sites; an odd half-volume; the largest lattice of the split form; the next one
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 2, 2, 6), (6, 6, 6, 10), (8, 8, 8, 16), (8, 8, 8, 18)])
@pytest.mark.parametrize("recon,csw", [(18, 1.0), (18, 0.0), (12, 1.0), (8, 1.0)])
def test_split_equals_one_thread_per_site(dirac, dims, recon, csw):
    import torch
    from paper_1109_2935_gb300 import synth
    lat = dirac.Lattice(dims, dirac.WILSON_CLOVER, kappa=0.124, csw=csw, recon=(recon, 12, 12), prec_mask=1)
    lat.load_gauge(synth.wilson_gauge(dims, 0.5, 0, 71, device="cuda"))
    x = lat.to_device(synth.wilson_spinor(dims, 72, device="cuda"), F64)
    y, z = lat.new_field(F64), lat.new_field(F64)
    lat.apply(y, x, dirac.PARITY_FULL, F64)
    lat.apply_multi(z, x, 1, F64)
    torch.cuda.synchronize()
    assert torch.equal(y, z)
    # without the clover term M = 1 - kappa D: the hopping blocks of both parities give M too
    if csw == 0.0:
        n = lat.field_bytes(F64, 0)
        d = torch.cat([lat.new_field(F64, 0) for _ in range(2)])
        lat.apply(d[:n], x[n:], dirac.PARITY_EVEN, F64)
        lat.apply(d[n:], x[:n], dirac.PARITY_ODD, F64)
        ref = x.view(torch.float64) - 0.124 * d.view(torch.float64)
        err = (y.view(torch.float64) - ref).norm() / ref.norm()
        assert err < 1e-15
