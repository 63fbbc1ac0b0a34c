"""Dependent launches on fields, links and clover written just before them: a stream of
calls without any synchronisation returns the bytes of the same calls with one after each,
also where the links are loaded again in between, and under stream capture with a branch."""
import pytest

from helpers import F16, F32, F64

pytestmark = pytest.mark.gpu


def _calls(dirac, op, prec):
    """A lattice, two gauge fields, a source in FP64 storage and the chained call on it."""
    import torch
    from paper_1109_2935_gb300 import synth
    dims = (8, 8, 8, 12)
    if op == "asqtad":
        links = [[(t, w) for t, w in zip(synth.asqtad_links(dims, s, s + 1, device="cuda"), (1, 2))] for s in (3, 5)]
        lat = dirac.Lattice(dims, dirac.ASQTAD, mass=0.05, prec_mask=1 | 1 << prec)
        psi = synth.staggered_spinor(dims, 7, device="cuda")
    else:
        links = [[(synth.wilson_gauge(dims, 0.5, 0, s, device="cuda"), 0)] for s in (3, 5)]
        lat = dirac.Lattice(dims, dirac.WILSON_CLOVER, kappa=0.12, csw=1.0, mr_steps=4, prec_mask=1 | 1 << prec)
        psi = synth.wilson_spinor(dims, 7, device="cuda")
    parity = {"eo": dirac.PARITY_EVEN, "asqtad": dirac.PARITY_FULL}.get(op, dirac.PARITY_FULL)
    call = {"m": lambda y, x: lat.apply(y, x, parity, prec), "eo": lambda y, x: lat.apply_eo(y, x, prec),
            "asqtad": lambda y, x: lat.apply_normal(y, x, parity, prec), "schwarz": lambda y, x: lat.schwarz(y, x, prec),
            "multi": lambda y, x: lat.apply_multi(y, x, 1, prec)}.get(op)
    if op == "ptc":
        net = dirac.Ptc(lat, (1, 2, 2, 1))
        g = torch.Generator().manual_seed(1)
        net.set_weights([0.3 * torch.randn((9, b, a, 4, 4), generator=g, dtype=torch.complex64).numpy()
                         for a, b in ((1, 2), (2, 2), (2, 1))])
        call = net.apply
    src = lat.new_field(F64, parity)
    lat.import_spinor(src, F64, parity, psi)
    return lat, links, src, parity, call


@pytest.mark.parametrize("op,prec", [("m", F64), ("m", F32), ("m", F16), ("eo", F64), ("eo", F16), ("asqtad", F64),
                                     ("asqtad", F32), ("asqtad", F16), ("schwarz", F16), ("schwarz", F32),
                                     ("multi", F32), ("ptc", F32)])
def test_unsynchronised_stream_equals_synchronised(dirac, op, prec):
    import torch
    lat, links, src, parity, call = _calls(dirac, op, prec)
    fields = [lat.new_field(prec, parity) for _ in range(7)]

    def run(wait):
        done = torch.cuda.synchronize if wait else (lambda: None)
        for k in range(2):  # load, convert the source, apply three times in a row; then other links
            for t, which in links[k]:
                lat.load_gauge(t, which)
                done()
            x = fields[0]
            lat.convert(x, prec, src, F64, parity)
            done()
            for y in fields[1 + 3 * k:4 + 3 * k]:
                call(y, x)
                done()
                x = y
        torch.cuda.synchronize()
        return [f.clone() for f in fields[1:]]

    want = run(True)
    assert not torch.equal(want[0], want[3])
    for _ in range(5):
        for f in fields[1:]:
            f.zero_()
        assert all(torch.equal(a, b) for a, b in zip(run(False), want))


@pytest.mark.parametrize("op,prec", [("m", F32), ("eo", F16), ("asqtad", F64)])
def test_capture_with_a_branch(dirac, op, prec):
    """A captured graph whose two branches both feed the last call."""
    import torch
    lat, links, src, parity, call = _calls(dirac, op, prec)
    for t, which in links[0]:
        lat.load_gauge(t, which)
    x, a, b, c = (lat.new_field(prec, parity) for _ in range(4))
    lat.convert(x, prec, src, F64, parity)

    def work(side):
        main = torch.cuda.current_stream()
        side.wait_stream(main)
        call(a, x)
        main.wait_stream(side)
        with torch.cuda.stream(side):
            side.wait_stream(main)
            b.copy_(a)
        main.wait_stream(side)
        call(c, b)

    side = torch.cuda.Stream()
    work(side)
    torch.cuda.synchronize()
    want = c.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        work(side)
    for _ in range(3):
        for f in (a, b, c):
            f.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(c, want)
