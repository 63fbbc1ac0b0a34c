"""FP64 operations on fields run chunk by chunk on few sites and site by site on more: both
sides of the threshold against torch in FP64, and the time of the large reductions."""
import pytest

from helpers import F64

pytestmark = pytest.mark.gpu


# 16,384 sites (the last of the chunk form), as a full and as a half field, and the next ones
@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("dims,parity", [((8, 8, 16, 16), -1), ((8, 8, 16, 18), -1), ((16, 16, 8, 16), 1),
                                         ((2, 6, 38, 36), -1), ((2, 6, 38, 38), -1), ((16, 16, 8, 18), 0)])
def test_both_forms(dirac, kind, dims, parity):
    import torch
    from paper_1109_2935_gb300 import synth
    lat = dirac.Lattice(dims, kind, prec_mask=1)
    gen = synth.wilson_spinor if kind == 0 else synth.staggered_spinor
    x, y = (lat.to_device(gen(dims, s, device="cuda"), F64, parity) for s in (1, 2))
    a, b = (lat.to_natural(f, F64, parity).reshape(-1) for f in (x, y))
    # sums of up to 24 x 17,328 products of numbers of order 1: a few 1e-16 sqrt(n) relative
    n2 = torch.vdot(a, a).real.item()
    assert abs(lat.norm2(x, F64, parity) - n2) <= 1e-13 * n2
    assert abs(lat.cdot(x, y, F64, parity) - torch.vdot(a, b).item()) <= 1e-13 * n2
    r = lat.caxpy_norm(0.3 - 0.7j, x, y, F64, parity)
    got, want = lat.to_natural(y, F64, parity).reshape(-1), b + (0.3 - 0.7j) * a
    assert (got - want).abs().max() <= 4e-15  # two roundings each of numbers below 8
    assert abs(r - torch.vdot(got, got).real.item()) <= 1e-13 * r


def test_reading_two_fields_is_cheaper_than_updating_one(dirac):
    """(x, y) of large FP64 fields moves two thirds of the bytes of y += a x with its norm:
    142 against 206 us at 24^3x64 (207 against 217 where both run chunk by chunk)."""
    import time

    import torch
    lat = dirac.Lattice((24, 24, 24, 64), 0, prec_mask=1)
    x, y = (lat.new_field(F64) for _ in range(2))
    best = []
    for call in (lambda: lat.cdot(x, y, F64), lambda: lat.caxpy_norm(0.5, x, y, F64)):
        t = []
        for _ in range(30):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            call()
            t.append(time.perf_counter() - t0)
        best.append(min(t))
    assert best[0] < 0.85 * best[1], best
