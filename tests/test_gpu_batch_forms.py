"""Batched plans take the form that is fastest for them."""
import pytest

from helpers import F16, F32, F64

pytestmark = pytest.mark.gpu


def best_us(fn):
    import torch
    start, end = (torch.cuda.Event(enable_timing=True) for _ in range(2))
    best = float("inf")
    for _ in range(8):
        start.record()
        for _ in range(20):
            fn()
        end.record()
        torch.cuda.synchronize()
        best = min(best, start.elapsed_time(end) * 50)
    return best


# one warp per SM scheduler or fewer: 40 us each way where it is spread over the chip
@pytest.mark.parametrize("dims,nrhs", [((8, 8, 8, 16), 1), ((12, 12, 12, 20), 1), ((10, 10, 14, 18), 3)])
def test_fp64_plan_is_as_fast_as_the_unplanned_call(dirac, dims, nrhs):
    import torch
    from paper_1109_2935_gb300 import synth
    lat = dirac.Lattice(dims, dirac.WILSON_CLOVER, kappa=0.12, csw=1.0, prec_mask=1)
    lat.load_gauge(synth.wilson_gauge(dims, 0.5, 0, 5, device="cuda"))
    x = torch.cat([lat.to_device(synth.wilson_spinor(dims, 9 + r, device="cuda"), F64) for r in range(nrhs)])
    y, z = torch.zeros_like(x), torch.zeros_like(x)
    plan = dirac.Batch([lat], [z], [x], [nrhs], F64)
    plan.apply()
    lat.apply_multi(y, x, nrhs, F64)
    assert torch.equal(y, z)
    # the same arithmetic in the same number of warps: 1.00 to 1.04 measured
    assert best_us(plan.apply) < 1.15 * best_us(lambda: lat.apply_multi(y, x, nrhs, F64))


def _plan(dirac, dims, prec, nrhs, recon=12, csw=1.0):
    import torch
    from paper_1109_2935_gb300 import synth
    lat = dirac.Lattice(dims, dirac.WILSON_CLOVER, kappa=0.12, csw=csw, recon=(18, recon, recon), prec_mask=1 << prec)
    lat.load_gauge(synth.wilson_gauge(dims, 0.5, 0, 5, device="cuda"))
    x = torch.cat([lat.to_device(synth.wilson_spinor(dims, 9 + r, device="cuda"), prec) for r in range(nrhs)])
    y = torch.zeros_like(x)
    plan = dirac.Batch([lat], [y], [x], [nrhs], prec)
    if prec == F16 and recon != 8:
        plan.set_tensor_cores(False)
    return lat, x, y, plan


# links and clover from L2 (one per thread is faster) and from DRAM (two are)
@pytest.mark.parametrize("prec,dims,nrhs", [(F16, (10, 10, 14, 18), 10), (F16, (12, 12, 12, 20), 8),
                                            (F32, (24, 24, 24, 32), 9)])
def test_plan_is_as_fast_as_either_kind(dirac, prec, dims, nrhs):
    _, _, _, plan = _plan(dirac, dims, prec, nrhs)
    tuned = best_us(plan.apply)
    for n in (1, 2):
        plan.set_rhs_per_thread(n)
        assert plan.info()["rhs_per_thread"] == n
        assert tuned < 1.06 * best_us(plan.apply), n


# half-volumes of a warp and less, ragged ones, a whole number of warps; odd and even counts,
# one right-hand side (no pair at all) and more than a CTA's four
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 6, 2, 6), (6, 6, 6, 10), (8, 8, 4, 4)])
@pytest.mark.parametrize("prec,recon", [(F32, 12), (F32, 18), (F32, 8), (F16, 12), (F16, 18), (F16, 8)])
@pytest.mark.parametrize("csw", [1.0, 0.0])
def test_two_per_thread_on_small_lattices(dirac, dims, prec, recon, csw):
    import torch
    for nrhs in (1, 2, 3, 7, 8):
        lat, x, y, plan = _plan(dirac, dims, prec, nrhs, recon, csw)
        n = lat.field_bytes(prec)
        plan.set_rhs_per_thread(2)
        assert plan.info()["rhs_per_thread"] == 2
        y.zero_()
        plan.apply()
        ref = torch.zeros_like(x)
        for r in range(nrhs):
            lat.apply(ref[r * n:(r + 1) * n], x[r * n:(r + 1) * n], dirac.PARITY_FULL, prec)
        assert torch.equal(y, ref)


def test_two_per_thread_is_refused_in_fp64(dirac):
    _, _, _, plan = _plan(dirac, (4, 4, 4, 4), F64, 2)
    with pytest.raises(dirac.DiracError):
        plan.set_rhs_per_thread(2)
    with pytest.raises(dirac.DiracError):
        plan.set_rhs_per_thread(3)
    assert plan.info()["rhs_per_thread"] == 1


@pytest.mark.parametrize("sloppy", [F16, F32])
def test_masked_pairs_on_lattices_that_take_pairs(dirac, sloppy):
    """The batched solves run two right-hand sides per thread where all lattices have more than
    two waves of warps; systems that stop at different times leave pairs with one member."""
    import torch
    from paper_1109_2935_gb300 import synth
    lats, xs, bs = [], [], []
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    for dims, kappa in (((12, 12, 12, 16), 0.12), ((16, 16, 16, 16), 0.125)):
        assert dims[0] * dims[1] * dims[2] * dims[3] // 32 * 8 > 32 * sms
        lat = dirac.Lattice(dims, dirac.WILSON_CLOVER, kappa=kappa, csw=1.0, prec_mask=1 | 1 << sloppy)
        lat.load_gauge(synth.wilson_gauge(dims, 0.5, 0, 83, device="cuda"))
        b = [lat.to_device(synth.wilson_spinor(dims, 110 + r, device="cuda"), F64) for r in range(8)]
        b[5].zero_()
        lats.append(lat)
        bs.append(torch.cat(b))
        xs.append(torch.zeros_like(bs[-1]))
    dirac.solve_many(lats, xs, bs, [8, 8], tol=1e-10, prec_sloppy=sloppy)
    for lat, x, b in zip(lats, xs, bs):
        n = lat.field_bytes(F64)
        for r in (0, 4, 5):
            x1 = torch.zeros(n, dtype=torch.uint8, device="cuda")
            dirac.solve_many([lat], [x1], [b[r * n:(r + 1) * n].clone()], [1], tol=1e-10, prec_sloppy=sloppy)
            assert torch.equal(x1, x[r * n:(r + 1) * n])


@pytest.mark.parametrize("dims,nrhs", [((8, 8, 8, 16), 11), ((16, 16, 16, 16), 3)])
def test_plan_launches_follow_as_closely_as_unplanned_ones(dirac, dims, nrhs):
    """Both are dependent launches of the same stencil; a plain one would add 2 us to 9."""
    import torch
    lat, x, _, plan = _plan(dirac, dims, F32, nrhs)
    z = torch.zeros_like(x)
    assert best_us(plan.apply) < 1.1 * best_us(lambda: lat.apply_multi(z, x, nrhs, F32))


def test_unplanned_odd_counts_take_pairs_in_fp32(dirac):
    """Links and clover from DRAM: with one right-hand side per thread they are read once per
    right-hand side (154 us against 130 of the timed plan)."""
    import torch
    lat, x, _, plan = _plan(dirac, (24, 24, 24, 32), F32, 3)
    z = torch.zeros_like(x)
    assert best_us(lambda: lat.apply_multi(z, x, 3, F32)) < 1.08 * best_us(plan.apply)
