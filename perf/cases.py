"""The work of this library, as cases that can be timed and checked.

Each case is one call (or the few calls) that a lattice QCD program makes through
``paper_1109_2935_gb300.dirac``: the operators and the preconditioner of the Krylov
iterations on one field, the same on many right-hand sides, the learned preconditioner's
inference and training, and whole solves. ``exact`` gives the same results from plain
torch in 64 bits: natural arrays [t, z, y, x, ...], rolled along the four directions.
"""
import math

import numpy as np
import torch

from paper_1109_2935_gb300 import dirac

PREC = {"f64": dirac.F64, "f32": dirac.F32, "f16": dirac.F16}
WIDTH = {"f64": 8, "f32": 4, "f16": 2}
RECON = {"f64": 18, "f32": 12, "f16": 12}  # stored reals per link, the library's defaults
CSW = 1.0
KAPPA = 0.12           # single-field operators and solves (well below critical: solves converge)
BATCH_KAPPA = (0.130, 0.133, 0.136)
SIGMA = 0.5            # spread of the links around the unit matrix
MASS = 0.01
PTC_CHANNELS = (1, 2, 2, 1)
TOL = 1e-12            # tight enough that the solution itself is good to 1e-9


# ------------------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest whole call: CG on M^dagger M, FP64, plain Wilson on 4^4 (a check run;
        # launches and host work between them are all of its time)
        {"name": "cg_f64_4x4x4x4", "op": "cg", "dims": "4x4x4x4"},
        # the operator of the FP32 iterations at the size of a production lattice
        {"name": "m_f32_24x24x24x128", "op": "m", "prec": "f32", "dims": "24x24x24x128", "dagger": False},
        # the same in 16-bit storage: the inner operator of the mixed-precision solves
        {"name": "m_f16_24x24x24x128", "op": "m", "prec": "f16", "dims": "24x24x24x128", "dagger": False},
        # even-odd (Schur) operator of the even-odd solvers, 16-bit storage, a mid-size lattice
        {"name": "eo_f16_16x16x16x32", "op": "eo", "prec": "f16", "dims": "16x16x16x32", "dagger": False},
        # staggered normal operator, one iteration of the asqtad CG, the largest lattice
        {"name": "asqtad_f32_48x48x48x144", "op": "asqtad", "prec": "f32", "dims": "48x48x48x144"},
        # block-Schwarz preconditioner of GCR-DD (4^4 blocks, 6 minimal-residual steps)
        {"name": "schwarz_f16_24x24x24x128", "op": "schwarz", "prec": "f16", "dims": "24x24x24x128"},
        # many right-hand sides on lattices of uneven sizes, one planned launch (propagator runs)
        {"name": "batch_f16_3lat_12rhs", "op": "batch", "prec": "f16", "dims": "16x16x16x32,24x24x24x64,32x32x32x64",
         "nrhs": 12},
        # an odd number of right-hand sides on one ragged lattice, FP32, no plan
        {"name": "multi_f32_12x12x12x20_7rhs", "op": "multi", "prec": "f32", "dims": "12x12x12x20", "nrhs": 7},
        # the learned preconditioner's forward pass inside flexible GCR (default FP32 layers)
        {"name": "ptc_f32_24x24x24x64", "op": "ptc", "dims": "24x24x24x64"},
        # two Adam steps of its training on four pairs (forward, backward, update)
        {"name": "ptc_train_16x16x16x16", "op": "ptc_train", "dims": "16x16x16x16", "pairs": 4},
        # a whole mixed-precision solve: GCR with the Schwarz preconditioner
        {"name": "gcr_dd_16x16x16x32", "op": "gcr_dd", "dims": "16x16x16x32"},
        # many small systems solved together (8 right-hand sides on each of 4 lattices)
        {"name": "bicgstab_many_4lat_8rhs", "op": "bicgstab_many",
         "dims": "8x8x8x8,8x8x8x16,12x12x12x16,16x16x16x16", "nrhs": 8},
    ]


def _dims(rng, low, high, extents=(4, 6, 8, 10, 12, 14, 16, 18, 20, 24, 28, 32, 36, 40, 48, 64, 96, 128, 144)):
    """Four even extents whose volume is spread over the logarithm of [low, high]."""
    want = math.exp(rng.uniform(math.log(low), math.log(high)))
    while True:
        side = want ** 0.25
        d = [rng.choice([e for e in extents if 0.5 * side <= e <= 2 * side] or [4]) for _ in range(3)]
        t = min(extents, key=lambda e: abs(math.log(e * d[0] * d[1] * d[2] / want)))
        d.append(t)
        if low <= math.prod(d) <= high:
            return "x".join(map(str, d))


def draw(rng):
    op = rng.choice(["m", "m", "eo", "asqtad", "schwarz", "batch", "multi", "ptc", "ptc_train", "cg", "gcr_dd",
                     "bicgstab_many"])
    big, mid = 24 ** 3 * 128, 24 ** 3 * 64
    if op in ("m", "eo"):
        prec = rng.choice(["f32", "f32", "f16", "f16", "f64"])
        return {"op": op, "prec": prec, "dims": _dims(rng, 256, big if prec != "f64" else mid),
                "dagger": rng.random() < 0.3}
    if op == "asqtad":
        prec = rng.choice(["f32", "f32", "f16", "f64"])
        return {"op": op, "prec": prec, "dims": _dims(rng, 1024, 32 ** 3 * 64)}
    if op == "schwarz":
        return {"op": op, "prec": rng.choice(["f16", "f16", "f32"]), "dims": _dims(rng, 256, big)}
    if op == "batch":
        return {"op": op, "prec": rng.choice(["f16", "f16", "f32"]), "nrhs": rng.randint(2, 16),
                "dims": ",".join(_dims(rng, 512, mid // 2) for _ in range(rng.randint(1, 3)))}
    if op == "multi":
        prec = rng.choice(["f16", "f32"])
        return {"op": op, "prec": prec, "nrhs": rng.randint(2, 20), "dims": _dims(rng, 256, mid // 2)}
    if op == "ptc":
        return {"op": op, "dims": _dims(rng, 256, mid)}
    if op == "ptc_train":
        return {"op": op, "dims": _dims(rng, 256, 16 ** 4), "pairs": rng.randint(1, 4)}
    if op == "cg":
        return {"op": op, "dims": _dims(rng, 256, 4096)}
    if op == "gcr_dd":
        return {"op": op, "dims": _dims(rng, 4096, 16 ** 3 * 32)}
    return {"op": op, "nrhs": rng.randint(2, 8),
            "dims": ",".join(_dims(rng, 1024, 12 ** 3 * 16) for _ in range(rng.randint(1, 4)))}


def _lattices(case):
    return [tuple(int(v) for v in d.split("x")) for d in case["dims"].split(",")]


def _kappa(case, l):
    return BATCH_KAPPA[l % 3] if case["op"] in ("batch", "multi") else KAPPA


def _csw(case):
    return 0.0 if case["op"] == "cg" else CSW


# ----------------------------------------------------------------------------- inputs
def _gauss(shape, g):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.complex64).to(torch.complex128)


def _unitary(z):
    """SU(3) from the first two rows of 3x3 matrices: Gram-Schmidt, third row conj(row 1 x row 2)."""
    a = z[..., 0, :]
    a = a / torch.linalg.vector_norm(a, dim=-1, keepdim=True)
    b = z[..., 1, :]
    b = b - (a.conj() * b).sum(-1, keepdim=True) * a
    b = b / torch.linalg.vector_norm(b, dim=-1, keepdim=True)
    return torch.stack([a, b, torch.linalg.cross(a, b).conj()], dim=-2)


def _links(dims, g, kind):
    """[t, z, y, x, mu, 3, 3]: "near" SU(3) spread around 1, "haar" SU(3), "fat" Gaussian / 8."""
    shape = dims[::-1]
    out = torch.empty(shape + (4, 3, 3), dtype=torch.complex128, device="cuda")
    for mu in range(4):
        z = _gauss(shape + (3, 3), g)
        if kind == "near":
            z = _unitary(0.5 * SIGMA * z + torch.eye(3, dtype=z.dtype, device=z.device))
        elif kind == "haar":
            z = _unitary(z)
        else:
            z = z / 8
        out[..., mu, :, :] = z
    return out


def _natural(case, seed):
    """The fields of a case in natural layout: per lattice the links and the spinors."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    got = []
    for dims in _lattices(case):
        shape = dims[::-1]
        if case["op"] == "asqtad":
            got.append((_links(dims, g, "fat"), _links(dims, g, "haar"), _gauss((1,) + shape + (3,), g)))
        else:
            n = case.get("nrhs", case.get("pairs", 1))
            got.append((_links(dims, g, "near"), _gauss((n,) + shape + (4, 3), g)))
    return got


def _weights(seed):
    """Initial weights [path, out, in, 4, 4] per layer: channel 0 passed through, small noise."""
    g = torch.Generator().manual_seed(seed + 1)
    ws = []
    for l in range(len(PTC_CHANNELS) - 1):
        w = 0.05 * torch.randn((9, PTC_CHANNELS[l + 1], PTC_CHANNELS[l], 4, 4), generator=g, dtype=torch.complex64)
        w[0, 0, 0] += torch.eye(4)
        ws.append(w.numpy())
    return ws


def _import(lat, prec, spinors, parity=dirac.PARITY_FULL):
    fb = lat.field_bytes(prec, parity)
    x = torch.empty(len(spinors) * fb, dtype=torch.uint8, device="cuda")
    for r, s in enumerate(spinors):
        lat.import_spinor(x[r * fb:(r + 1) * fb], prec, parity, s)
    return x


def _numbers(lat, f, prec):
    """The numbers of a field, as the library lays them out."""
    if prec == dirac.F64:
        return f.view(torch.float64)
    if prec == dirac.F32:
        return f.view(torch.float32)
    vh, w = lat.volume // 2, 2 * lat.nr  # 16-bit values of a half-field, then its per-site norms
    f = f.view(-1, (w + 4) * vh)
    return [f[:, :w * vh].view(torch.float16), f[:, w * vh:].view(torch.float32)]


def prepare(case, seed):
    op = case["op"]
    solve = op in ("cg", "gcr_dd", "bicgstab_many")
    prec = PREC[case.get("prec", "f64" if solve else "f32")]
    mask = {"cg": 1, "gcr_dd": 5, "bicgstab_many": 5}.get(op, 1 << prec)
    parity = dirac.PARITY_EVEN if op in ("asqtad", "eo") else dirac.PARITY_FULL
    st = {"op": op, "prec": prec, "parity": parity, "nrhs": case.get("nrhs", 1), "dagger": case.get("dagger", False),
          "lats": [], "ins": [], "outs": [], "numbers": []}
    for l, (dims, fields) in enumerate(zip(_lattices(case), _natural(case, seed))):
        if op == "asqtad":
            lat = dirac.Lattice(dims, dirac.ASQTAD, mass=MASS, prec_mask=mask)
            lat.load_gauge(fields[0], 1)
            lat.load_gauge(fields[1], 2)
        else:
            lat = dirac.Lattice(dims, dirac.WILSON_CLOVER, kappa=_kappa(case, l), csw=_csw(case), mr_steps=6,
                                prec_mask=mask)
            lat.load_gauge(fields[0])
        st["lats"].append(lat)
        st["ins"].append(_import(lat, prec, fields[-1], parity))
        st["outs"].append(torch.zeros_like(st["ins"][-1]))
        st["numbers"].append(_numbers(lat, st["outs"][-1], prec))
    if op == "batch":
        st["plan"] = dirac.Batch(st["lats"], st["outs"], st["ins"], [st["nrhs"]] * len(st["lats"]), prec)
    if op in ("ptc", "ptc_train"):
        st["net"] = dirac.Ptc(st["lats"][0], PTC_CHANNELS)
        st["weights"] = _weights(seed)
        st["net"].set_weights(st["weights"])
        n = st["lats"][0].field_bytes(prec)
        st["pairs"] = list(st["ins"][0].split(n))
    torch.cuda.synchronize()
    return st


# -------------------------------------------------------------------------------- run
def run(st):
    op, lat, x, y, prec = st["op"], st["lats"][0], st["ins"][0], st["outs"][0], st["prec"]
    if op == "m":
        (lat.apply_dagger if st["dagger"] else lat.apply)(y, x, st["parity"], prec)
    elif op == "eo":
        lat.apply_eo(y, x, prec, st["dagger"])
    elif op == "asqtad":
        lat.apply_normal(y, x, st["parity"], prec)
    elif op == "schwarz":
        lat.schwarz(y, x, prec)
    elif op == "batch":
        st["plan"].apply()
    elif op == "multi":
        lat.apply_multi(y, x, st["nrhs"], prec)
    elif op == "ptc":
        st["net"].apply(y, x)
    elif op == "ptc_train":
        net = st["net"]
        net.set_weights(st["weights"])
        loss = net.train(st["pairs"], steps=2, batch=len(st["pairs"]), lr=1e-2, seed=1)
        # losses and weights are 32-bit numbers in the library
        return [loss.astype(np.float32)] + [w.astype(np.complex64) for w in net.get_weights()]
    elif op == "cg":
        lat.solve(y, x, dirac.CG_NORMAL, tol=TOL)
    elif op == "gcr_dd":
        lat.solve(y, x, dirac.GCR_DD, tol=TOL, k_max=16, delta=0.1, prec_sloppy=dirac.F16, prec_precond=dirac.F16)
    else:
        dirac.solve_many(st["lats"], st["outs"], st["ins"], [st["nrhs"]] * len(st["lats"]), tol=TOL, delta=0.1,
                         prec_sloppy=dirac.F16)
    return st["numbers"]


# ------------------------------------------------------------------------------- work
def work(case):
    """Every input read once and every output written once, and the arithmetic of the
    formulas: hopping term 1320 flop per site, clover 504, sum 48; asqtad 1146. For a solve
    one pass over its fields and one operator application: how often it iterates is its own
    business."""
    op, total = case["op"], {"bytes": 0, "flops": 0}
    w = WIDTH[case.get("prec", "f32" if op in ("ptc", "ptc_train") else "f64")]
    rec = RECON[{8: "f64", 4: "f32", 2: "f16"}[w]]
    norm = 4 if w == 2 else 0
    for dims in _lattices(case):
        v, n = math.prod(dims), case.get("nrhs", 1)
        spinor, clover, links = 24 * w + norm, 72 * w + norm, 4 * rec * w
        if op in ("m", "schwarz", "batch", "multi"):
            b, f = links + clover + 2 * n * spinor, 1872 * n
            f = 6 * (1872 + 192) if op == "schwarz" else f
        elif op == "eo":  # links of both parities, Ahat on one and its inverse on the other
            b, f = links + clover + spinor, 1320 + 504 + 24
        elif op == "asqtad":  # fat (18 reals) and long links, half-field in and out
            b, f = 4 * (18 + rec) * w + 6 * w + norm, 1146 + 12
        elif op in ("ptc", "ptc_train"):
            b, f = links + 2 * spinor, 36096
            if op == "ptc_train":  # two steps: forward, weight gradients, gradients of the activations
                b, f = links + 2 * case["pairs"] * spinor, 2 * 3 * case["pairs"] * f
        else:
            b, f = links + (clover if op != "cg" else 0) + 2 * n * spinor, 1872 * n
        total["bytes"] += b * v
        total["flops"] += f * v
    return total


# ------------------------------------------------------------------------------ exact
def _shift(f, mu, n, sign=True):
    """f(x + n mu) for [..., t, z, y, x, a, b] fields (periodic; antiperiodic in t for fermions)."""
    d = f.dim() - 3 - mu
    out = torch.roll(f, -n, dims=d)
    if mu == 3 and sign:
        lt = f.shape[d]
        t = torch.arange(lt, device=f.device)
        s = 1.0 - 2.0 * (torch.div(t + n, lt, rounding_mode="floor").abs() % 2)
        out = out * s.view([lt] + [1] * (f.dim() - 1 - d))
    return out


def _mul(u, f):
    """u[..., a, b] f[..., s, b], colour by colour."""
    out = u[..., None, :, 0] * f[..., :, 0, None]
    for b in (1, 2):
        out = out + u[..., None, :, b] * f[..., :, b, None]
    return out


def _dag(u):
    return u.conj().transpose(-1, -2)


def _gammas():
    i = 1j
    b = np.array([[[0, i], [i, 0]], [[0, -1], [1, 0]], [[i, 0], [0, -i]], [[1, 0], [0, 1]]], dtype=complex)
    g = np.zeros((4, 4, 4), dtype=complex)
    g[:, :2, 2:] = b
    g[:, 2:, :2] = b.conj().transpose(0, 2, 1)
    return g


def _spin(m, f):
    """A 4x4 spin matrix on f[..., s, c]: its few nonzero entries only."""
    rows = []
    for s in range(4):
        acc = None
        for t in range(4):
            if m[s, t] != 0:
                p = complex(m[s, t]) * f[..., t, :]
                acc = p if acc is None else acc + p
        rows.append(acc)
    return torch.stack(rows, dim=-2)


class _Wilson:
    """M = Ahat - kappa D with Ahat = 1 + 2 kappa A (A: clover term from the plaquette leaves)."""

    def __init__(self, u, kappa, csw, block=None):
        self.u, self.kappa, self.g = u, kappa, _gammas()
        self.dims = u.shape[3::-1]
        self.ahat = self._clover(csw) if csw else None
        self.block = block

    def _clover(self, csw):
        u, s = self.u, lambda f, mu, n: _shift(f, mu, n, False)
        one = [torch.eye(3, dtype=u.dtype, device=u.device)[a] for a in range(3)]
        a = torch.zeros(u.shape[:4] + (4, 3, 4, 3), dtype=u.dtype, device=u.device)
        for mu in range(4):
            for nu in range(mu + 1, 4):
                m, n = u[..., mu, :, :], u[..., nu, :, :]
                m_n, n_m = s(m, nu, 1), s(n, mu, 1)
                mb, nb = s(m, mu, -1), s(n, nu, -1)
                q = m @ n_m @ _dag(m_n) @ _dag(n)
                q += n @ _dag(s(mb, nu, 1)) @ _dag(s(n, mu, -1)) @ mb
                q += _dag(mb) @ _dag(s(nb, mu, -1)) @ s(mb, nu, -1) @ nb
                q += _dag(nb) @ s(m, nu, -1) @ s(nb, mu, 1) @ _dag(m)
                f = (q - _dag(q)) / 8
                tr = torch.diagonal(f, dim1=-2, dim2=-1).sum(-1) / 3
                f = f - tr[..., None, None] * torch.stack(one)
                sig = 0.5j * (self.g[mu] @ self.g[nu] - self.g[nu] @ self.g[mu])
                for i in range(4):
                    for j in range(4):
                        if sig[i, j] != 0:
                            a[..., i, :, j, :] += complex(0.5j * csw * sig[i, j]) * f
        a = 2 * self.kappa * a.reshape(u.shape[:4] + (12, 12))
        return a + torch.eye(12, dtype=u.dtype, device=u.device)

    def site(self, mat, f):
        if mat is None:
            return f
        v = f.reshape(f.shape[:-2] + (12,))
        out = mat[..., 0] * v[..., 0, None]
        for j in range(1, 12):
            out = out + mat[..., j] * v[..., j, None]
        return out.view(f.shape)

    def _inside(self, mu, forward):
        """Sites whose hop stays within its block (None: all)."""
        if self.block is None or self.block[mu] == self.dims[mu]:
            return None
        x = torch.arange(self.dims[mu], device=self.u.device) % self.block[mu]
        keep = (x != self.block[mu] - 1) if forward else (x != 0)
        return keep.view([-1] + [1] * (mu + 2))

    def hop(self, f, dagger=False):
        out = torch.zeros_like(f)
        for mu in range(4):
            u, p = self.u[..., mu, :, :], np.eye(4) - (-1 if dagger else 1) * self.g[mu]
            for forward in (True, False):
                v = _mul(u, _shift(f, mu, 1)) if forward else _shift(_mul(_dag(u), f), mu, -1)
                v = _spin(p if forward else 2 * np.eye(4) - p, v)
                keep = self._inside(mu, forward)
                out += v if keep is None else v * keep
        return out

    def m(self, f, dagger=False):
        return self.site(self.ahat, f) - self.kappa * self.hop(f, dagger)

    def eo(self, f, dagger=False):
        ev = _even(self.dims)[..., None, None]
        inv = torch.linalg.inv(self.ahat)
        f = f * ev
        t = self.site(inv, self.hop(f, dagger) * ~ev)
        return (self.site(self.ahat, f) - self.kappa ** 2 * self.hop(t, dagger)) * ev

    def schwarz(self, f, steps):
        d, b = self.dims[::-1], self.block[::-1]
        cut = [v for n, k in zip(d, b) for v in (n // k, k)]

        def dots(p, r):
            s = (p.conj() * r).sum((-1, -2)).reshape(cut).sum((1, 3, 5, 7), keepdim=True)
            return s.expand(cut).reshape(d)[..., None, None]

        x, r = torch.zeros_like(f), f
        for _ in range(steps):
            p = self.m(r)
            a = dots(p, r) / dots(p, p)
            x, r = x + a * r, r - a * p
        return x

    def solve(self, b, normal=False):
        """x with M x = b (M^dagger M x = b where normal): conjugate gradients on M^dagger M."""
        op = lambda v: self.m(self.m(v), True)
        dot = lambda v, w: (v.conj() * w).sum((-1, -2, -3, -4, -5, -6), keepdim=True).real
        x, r = torch.zeros_like(b), b if normal else self.m(b, True)
        p, rr = r, dot(r, r)
        stop = 1e-28 * rr
        for _ in range(2000):
            ap = op(p)
            a = rr / dot(p, ap).clamp_min(1e-300)
            x, r = x + a * p, r - a * ap
            new = dot(r, r)
            if bool((new <= stop).all()):
                break
            p, rr = r + new / rr * p, new
        return x


def _even(dims):
    lx, ly, lz, lt = dims
    r = [torch.arange(n, device="cuda") for n in (lt, lz, ly, lx)]
    return (r[0].view(-1, 1, 1, 1) + r[1].view(-1, 1, 1) + r[2].view(-1, 1) + r[3]) % 2 == 0


def _asqtad(fat, lng, f):
    """(m^2 - D D / 4) f on the even sites (f zero on the odd ones)."""
    dims = fat.shape[3::-1]
    r = [torch.arange(n, device="cuda") for n in dims]

    def hop(v):
        out = torch.zeros_like(v)
        for mu in range(4):
            par = torch.zeros((1, 1, 1, 1), dtype=torch.int64, device="cuda")
            for nu in range(mu):
                par = par + r[nu].view([-1] + [1] * nu)
            eta = (1.0 - 2.0 * (par % 2))[..., None, None]
            for links, n in ((fat, 1), (lng, 3)):
                u = links[..., mu, :, :]
                out += eta * (_mul(u, _shift(v, mu, n)) - _shift(_mul(_dag(u), v), mu, -n))
        return out

    ev = _even(dims)[..., None, None]
    f = f.unsqueeze(-2) * ev
    return ((MASS * MASS * f - 0.25 * hop(hop(f))) * ev).squeeze(-2)


def _ptc(u, ws, f):
    """out_c = sum over paths p and channels c' of W[p, c, c'] (T_p f_c'), layer by layer."""
    chans = [f]
    for w in ws:
        outs = [0] * w.shape[1]
        for ci, c in enumerate(chans):
            for p in range(9):
                mu, back = (p - 1) // 2, (p - 1) % 2
                if p == 0:
                    t = c
                elif back:
                    t = _shift(_mul(_dag(u[..., mu, :, :]), c), mu, -1)
                else:
                    t = _mul(u[..., mu, :, :], _shift(c, mu, 1))
                for co in range(w.shape[1]):
                    outs[co] = outs[co] + torch.matmul(w[p, co, ci], t)
        chans = outs
    return chans[0]


def _train(wil, v):
    """Losses and weights of two Adam steps on all pairs (M v, v)."""
    r = wil.m(v)

    def go(ws, steps=2, lr=1e-2, b1=0.9, b2=0.999, eps=1e-8):
        ws = [torch.from_numpy(w).to("cuda", torch.complex128) for w in ws]
        m, s, losses = [0.0] * len(ws), [0.0] * len(ws), []
        for t in range(1, steps + 1):
            ws = [w.detach().requires_grad_(True) for w in ws]
            loss = 0.0
            for k in range(len(v)):
                part = (_ptc(wil.u, ws, r[k]) - v[k]).abs().square().sum() / v[k].abs().square().sum() / len(v)
                part.backward()
                loss += float(part)
            losses.append(loss)
            with torch.no_grad():
                for i, w in enumerate(ws):
                    g = torch.view_as_real(w.grad.resolve_conj())
                    m[i] = b1 * m[i] + (1 - b1) * g
                    s[i] = b2 * s[i] + (1 - b2) * g * g
                    step = (m[i] / (1 - b1 ** t)) / ((s[i] / (1 - b2 ** t)).sqrt() + eps)
                    ws[i] = w - lr * torch.view_as_complex(step)
        return [torch.tensor(losses, dtype=torch.float64)] + [w.detach() for w in ws]

    return go


def _laid_out(f, prec, halves=(0, 1)):
    """Natural fields [n, t, z, y, x, ...] as the library stores them: per field and parity
    (checkerboard order) chunks of a site's reals, chunk by chunk; 16-bit values relative to
    the site's largest one, which follows as its norm."""
    n, shape = f.shape[0], f.shape[1:5]
    real = torch.view_as_real(f.resolve_conj().contiguous()).reshape(n, math.prod(shape), -1)
    nr = real.shape[-1]
    even = _even(shape[::-1]).reshape(-1)
    vals, norms = [], []
    for h in halves:
        s = real[:, even if h == 0 else ~even]
        chunk = {"f64": 2, "f32": 4 if nr == 24 else 2, "f16": 8 if nr == 24 else 2}[prec]
        norm = s.abs().amax(-1)
        if prec == "f16":
            s = s / norm[..., None]
        vals.append(s.reshape(n, -1, nr // chunk, chunk).transpose(1, 2).reshape(n, -1))
        norms.append(norm)
    if prec != "f16":
        return torch.stack(vals, 1).reshape(-1)
    return [torch.stack(v, 1).reshape(n * len(halves), -1) for v in (vals, norms)]


def exact(case, seed):
    op = case["op"]
    solve = op in ("cg", "gcr_dd", "bicgstab_many")
    prec = case.get("prec", "f64" if solve else "f32")
    dagger = case.get("dagger", False)
    got = []
    for l, (dims, fields) in enumerate(zip(_lattices(case), _natural(case, seed))):
        if op == "asqtad":
            got.append(_laid_out(_asqtad(*fields[:2], fields[2][0])[None], prec, (0,)))
            continue
        u, f = fields
        if op == "ptc":
            ws = [torch.from_numpy(w).to("cuda", torch.complex128) for w in _weights(seed)]
            got.append(_laid_out(_ptc(u, ws, f[0])[None], prec))
            continue
        block = tuple(next(b for b in (4, 2, 1) if d % b == 0) for d in dims)
        wil = _Wilson(u, _kappa(case, l), _csw(case), block if op == "schwarz" else None)
        if op == "ptc_train":
            return _train(wil, f)(_weights(seed))
        if solve:
            out = wil.solve(f, op == "cg")
        elif op == "eo":
            out = torch.stack([wil.eo(v, dagger) for v in f])
        elif op == "schwarz":
            out = torch.stack([wil.schwarz(v, 6) for v in f])
        else:
            out = torch.stack([wil.m(v, dagger) for v in f])
        got.append(_laid_out(out, prec, (0,) if op == "eo" else (0, 1)))
        del wil, out
    return got
