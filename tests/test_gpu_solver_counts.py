"""dslash_calls of the batched solves: every operator application of a system, and no other."""
import pytest

from helpers import F16, F64

pytestmark = pytest.mark.gpu


def _system(dirac, nrhs, ds=False):
    import torch
    from paper_1109_2935_gb300 import synth
    dims = (6, 6, 6, 10)
    lat = dirac.Lattice(dims, dirac.WILSON_CLOVER, kappa=0.12, csw=1.0, prec_mask=1 | 1 << F16)
    lat.load_gauge(synth.wilson_gauge(dims, 0.5, 0, 5, device="cuda"))
    lat.set_ds_residual(ds)
    b = torch.cat([lat.to_device(synth.wilson_spinor(dims, 9 + r, device="cuda"), F64) for r in range(nrhs)])
    return lat, torch.zeros_like(b), b


def test_converged(dirac):
    """Two a Krylov iteration and one a reliable update; the last of these is the final residual."""
    lat, x, b = _system(dirac, 3)
    for st in dirac.solve_many([lat], [x], [b], [3], tol=1e-10)["rhs"]:
        assert st["iters"] > 0 and st["reliable_updates"] > 0
        assert st["dslash_calls"] == 2 * st["iters"] + st["reliable_updates"]


def test_budget_exhausted(dirac):
    """The final residual is one more."""
    lat, x, b = _system(dirac, 2)
    res = dirac.solve_many([lat], [x], [b], [2], tol=1e-12, max_iter=7, raise_on_error=False)
    assert res["status"] == "ERR_NOT_CONVERGED"
    for st in res["rhs"]:
        assert st["dslash_calls"] == 2 * st["iters"] + st["reliable_updates"] + 1


def test_initial_guess(dirac):
    """The starting residual is one more."""
    lat, x, b = _system(dirac, 2)
    dirac.solve_many([lat], [x], [b], [2], tol=1e-4)
    for st in dirac.solve_many([lat], [x], [b], [2], tol=1e-10, use_x0=True)["rhs"]:
        assert st["dslash_calls"] == 2 * st["iters"] + st["reliable_updates"] + 1


def test_double_single_residuals(dirac):
    """A residual that the double-single operator puts below the target is taken again in FP64."""
    lat, x, b = _system(dirac, 1, ds=True)
    st = dirac.solve_many([lat], [x], [b], [1], tol=1e-10)["rhs"][0]
    again = st["dslash_calls"] - 2 * st["iters"] - st["reliable_updates"]
    assert 1 <= again <= st["reliable_updates"]
