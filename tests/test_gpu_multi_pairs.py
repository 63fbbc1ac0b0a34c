"""Two right-hand sides per thread give the bits of one application each: even and odd counts,
half-volumes that are and are not a multiple of a warp, planned and unplanned launches."""
import pytest

from helpers import F16, F32, F64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(12, 12, 12, 20), (10, 10, 14, 18), (2, 6, 18, 50)])
@pytest.mark.parametrize("prec,nrhs,recon", [(F32, 7, 12), (F32, 12, 12), (F16, 9, 12), (F16, 14, 12), (F16, 16, 12),
                                             (F16, 14, 18), (F16, 14, 8)])
@pytest.mark.parametrize("csw", [1.0, 0.0])
def test_multi_equals_single(dirac, dims, prec, nrhs, recon, csw):
    import torch
    from paper_1109_2935_gb300 import synth
    lat = dirac.Lattice(dims, dirac.WILSON_CLOVER, kappa=0.124, csw=csw, recon=(18, recon, recon),
                        prec_mask=1 << prec)
    lat.load_gauge(synth.wilson_gauge(dims, 0.5, 0, 81, device="cuda"))
    n = lat.field_bytes(prec)
    x = torch.cat([lat.to_device(synth.wilson_spinor(dims, 90 + r, device="cuda"), prec) for r in range(nrhs)])
    ref, y, z = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x)
    for r in range(nrhs):
        lat.apply(ref[r * n:(r + 1) * n], x[r * n:(r + 1) * n], dirac.PARITY_FULL, prec)
    lat.apply_multi(y, x, nrhs, prec)
    plan = dirac.Batch([lat], [z], [x], [nrhs], prec)
    if prec == F16 and recon != 8:
        plan.set_tensor_cores(False)
    z.zero_()
    plan.apply()
    torch.cuda.synchronize()
    assert torch.equal(y, ref)
    assert torch.equal(z, ref)


@pytest.mark.parametrize("sloppy", [F16, F32])
def test_masked_pairs(dirac, sloppy):
    """Systems that stop at different times (one has a zero source) leave pairs with one
    member: every system still returns the bytes of being solved alone."""
    import torch
    from paper_1109_2935_gb300 import synth
    lats, xs, bs = [], [], []
    for dims, kappa in (((12, 12, 12, 16), 0.12), ((16, 16, 8, 10), 0.125)):
        lat = dirac.Lattice(dims, dirac.WILSON_CLOVER, kappa=kappa, csw=1.0, prec_mask=1 | 1 << sloppy)
        lat.load_gauge(synth.wilson_gauge(dims, 0.5, 0, 83, device="cuda"))
        b = [lat.to_device(synth.wilson_spinor(dims, 110 + r, device="cuda"), F64) for r in range(8)]
        b[2].zero_()
        lats.append(lat)
        bs.append(torch.cat(b))
        xs.append(torch.zeros_like(bs[-1]))
    dirac.solve_many(lats, xs, bs, [8, 8], tol=1e-10, prec_sloppy=sloppy)
    for lat, x, b in zip(lats, xs, bs):
        n = lat.field_bytes(F64)
        for r in (0, 2, 3, 7):
            x1 = torch.zeros(n, dtype=torch.uint8, device="cuda")
            dirac.solve_many([lat], [x1], [b[r * n:(r + 1) * n].clone()], [1], tol=1e-10, prec_sloppy=sloppy)
            assert torch.equal(x1, x[r * n:(r + 1) * n])
