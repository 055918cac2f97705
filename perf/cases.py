"""Performance cases of the library: what its users have it do, by kind of call.

A case names a kind of call, a lattice and the options of that call:

  dslash      D_oe and D_eo on fields that view torch tensors (FP32, FP64), or
              on library fields exported to torch tensors (double-float)
  apply_M     M = m^2 - D_eo D_oe on one even field
  upload      a new gauge configuration: the three-link products, the upload
              and the first operator application on it
  cg          a source imported, solved for by plain CG, the solution exported
  cg_mixed    the same with mixed-precision CG (FP32 or 16-bit iterations)
  multishift  one source, several shifts (rational approximations)
  batched     several sources, on one or two lattices at once
  learned     mixed-precision flexible CG with the network preconditioner
  net_grad    the network's training objective and its weight gradients

Gauge fields are special unitary matrices scattered about the unit matrix,
with the spread the repository's own synthetic configurations have; sources
are Gaussian.  Every case is solved without tuning the lattice first, as a
program that makes one call on a new lattice does.
"""
import math

import numpy as np
import torch

from paper_1411_2087_gb300 import stag

C1, C3 = stag.C1_NAIK, stag.C3_NAIK
BC = stag.BC_DEFAULT


# ---------------------------------------------------------------- the cases
def _case(name, kind, dims, **more):
    c = {"kind": kind, "Lx": dims[0], "Ly": dims[1], "Lz": dims[2], "Lt": dims[3]}
    c.update(more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one operator application on the test lattice,
        # where latency is all; the production precision
        _case("dslash_df64_8x8x8x8", "dslash", (8, 8, 8, 8), prec="df64", comp="none"),
        # an operator application inside a user's own FP32 solver, on 12-real
        # links and a lattice with no powers of two in its extents
        _case("dslash_f32c12_20x12x28x36", "dslash", (20, 12, 28, 36), prec="f32", comp="all"),
        # IEEE double, for programs that want no other format
        _case("M_f64_16x16x16x32", "apply_M", (16, 16, 16, 32), prec="f64", comp="none", mass=0.05),
        # the step from one gauge configuration to the next (every molecular-
        # dynamics step of a gauge-field ensemble, every measured configuration)
        _case("upload_24x24x24x48", "upload", (24, 24, 24, 48), comp="all"),
        # a solve on the parity configuration of the tests: launches count
        _case("cg_df64_8x8x8x8", "cg", (8, 8, 8, 8), prec="df64", mass=0.1),
        # a solve on a small, uneven lattice (tuning runs, smearing studies)
        _case("cg_df64_12x16x20x24", "cg", (12, 16, 20, 24), prec="df64", mass=0.05),
        # the headline workload
        _case("cg_df64_32x32x32x64", "cg", (32, 32, 32, 64), prec="df64", mass=0.02),
        # the largest lattice, in the fastest solver
        _case("cg_f16c12_48x48x48x96", "cg_mixed", (48, 48, 48, 96), inner="f16", comp="all", mass=0.01),
        # a rational approximation's solve: twelve shifts of one operator
        _case("multishift_24x24x24x48", "multishift", (24, 24, 24, 48), prec="df64", mixed="none", shifts=12,
              mass=0.02),
        # propagators: several sources at once on an ensemble of two lattices
        _case("batched_16x16x16x16_24x24x24x48", "batched", (24, 24, 24, 48), mixed="none", n=4, Lx2=16, Ly2=16,
              Lz2=16, Lt2=16, n2=4, mass=0.05),
        # light quarks with the network preconditioner
        _case("learned_f16_32x32x32x64", "learned", (32, 32, 32, 64), inner="f16", mass=0.005),
        # one gradient of the network's training, forward and backward
        _case("net_grad_16x16x16x16", "net_grad", (16, 16, 16, 16), mass=0.05, pairs=8, stride=4, loss="residual"),
    ]


# sites of the lattices each kind is called on
RANGES = {"dslash": (8 ** 4, 1 << 21), "apply_M": (8 ** 4, 1 << 21), "upload": (8 ** 4, 24 ** 3 * 48),
          "cg": (8 ** 4, 1 << 20), "cg_mixed": (8 ** 4, 40 ** 3 * 64), "multishift": (8 ** 4, 24 ** 3 * 48),
          "batched": (8 ** 4, 16 ** 3 * 32), "learned": (8 ** 4, 1 << 20), "net_grad": (8 ** 4, 16 ** 3 * 32)}


def _draw_dims(rng, lo, hi):
    """Even extents with a volume spread over [lo, hi] on a logarithmic scale, time the longest or nearly so."""
    while True:
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        side = (v / rng.uniform(1.0, 2.0)) ** 0.25
        xyz = [max(4, 2 * round(side * math.exp(rng.uniform(-0.35, 0.35)) / 2)) for _ in range(3)]
        t = max(4, 2 * round(v / (xyz[0] * xyz[1] * xyz[2]) / 2))
        if lo * 0.8 <= xyz[0] * xyz[1] * xyz[2] * t <= hi and t <= 128:
            return tuple(xyz) + (t,)


def draw(rng):
    kind = rng.choice(["dslash", "dslash", "apply_M", "upload", "cg", "cg", "cg_mixed", "cg_mixed", "multishift",
                       "batched", "learned", "net_grad"])
    dims = _draw_dims(rng, *RANGES[kind])
    mass = round(math.exp(rng.uniform(math.log(0.02), math.log(0.2))), 4)
    if kind in ("dslash", "apply_M"):
        prec = rng.choice(["df64", "df64", "f32", "f64"])
        comp = rng.choice(["none", "all", "long"]) if prec == "f32" else "none"
        more = {} if kind == "dslash" else {"mass": mass}
        return _case(None, kind, dims, prec=prec, comp=comp, **more)
    if kind == "upload":
        return _case(None, kind, dims, comp=rng.choice(["none", "all", "long"]))
    if kind == "cg":
        return _case(None, kind, dims, prec=rng.choice(["df64", "df64", "df64", "f64"]), mass=mass)
    if kind == "cg_mixed":
        return _case(None, kind, dims, inner=rng.choice(["f32", "f16"]), comp=rng.choice(["none", "all", "long"]),
                     mass=mass)
    if kind == "multishift":
        return _case(None, kind, dims, prec="df64", mixed=rng.choice(["none", "none", "f32"]),
                     shifts=rng.randint(2, 12), mass=mass)
    if kind == "batched":
        small = _draw_dims(rng, 8 ** 4, 16 ** 4)
        return _case(None, kind, dims, mixed=rng.choice(["none", "f32", "f16"]), n=rng.randint(1, 8), Lx2=small[0],
                     Ly2=small[1], Lz2=small[2], Lt2=small[3], n2=rng.randint(0, 4), mass=mass)
    if kind == "learned":
        return _case(None, kind, dims, inner=rng.choice(["f16", "f32", "none"]), mass=mass)
    return _case(None, kind, dims, mass=mass, pairs=rng.randint(2, 8), stride=rng.randint(2, 5),
                 loss=rng.choice(["residual", "error"]))


def _dims(case, second=False):
    return tuple(int(case[k + ("2" if second else "")]) for k in ("Lx", "Ly", "Lz", "Lt"))


def _volume(dims):
    return dims[0] * dims[1] * dims[2] * dims[3]


# relative residuals asked for: the repository's own, and for the solvers that iterate in a low precision the
# tighter one of a solve whose result enters an energy difference
TOL = 1e-10
TOL_MIXED = 1e-11


# ------------------------------------------------------------------- inputs
def _gen(seed, which):
    g = torch.Generator(device="cuda")
    g.manual_seed((int(seed) * 1000003 + which) & 0x7FFFFFFFFFFF)
    return g


def _links(dims, seed, which=0, eps=0.3):
    """SU(3) links [4][V][3][3] about the unit matrix: rows 0 and 1 of 1 + i eps H (H Hermitian, Gaussian)
    made orthonormal, row 2 their conjugate cross product."""
    n = 4 * _volume(dims)
    gen = _gen(seed, 10 + which)
    out = torch.empty((n, 3, 3), dtype=torch.complex128, device="cuda")
    for a in range(0, n, 1 << 22):
        m = min(n, a + (1 << 22)) - a
        w = torch.randn((m, 8), generator=gen, device="cuda", dtype=torch.float64) * (0.5 * eps)
        d0, d1 = w[:, 2] + w[:, 7] / math.sqrt(3), -w[:, 2] + w[:, 7] / math.sqrt(3)
        one = torch.ones_like(d0)
        r0 = torch.stack([torch.complex(one, d0), torch.complex(w[:, 1], w[:, 0]), torch.complex(w[:, 4], w[:, 3])], 1)
        r1 = torch.stack([torch.complex(-w[:, 1], w[:, 0]), torch.complex(one, d1),
                          torch.complex(w[:, 6], w[:, 5])], 1)
        r0 = r0 / torch.linalg.vector_norm(r0, dim=1, keepdim=True)
        r1 = r1 - (r0.conj() * r1).sum(1, keepdim=True) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=1, keepdim=True)
        out[a:a + m, 0], out[a:a + m, 1] = r0, r1
        out[a:a + m, 2] = torch.linalg.cross(r0, r1, dim=1).conj()
    return out.view(4, -1, 3, 3)


def _source(dims, seed, which):
    v = torch.randn((_volume(dims) // 2, 3, 2), generator=_gen(seed, 100 + which), device="cuda", dtype=torch.float64)
    return torch.view_as_complex(v)


def _shift_list(n):
    return [float(s) for s in np.geomspace(1e-4, 0.5, n)] if n > 1 else [1e-4]


def _net_weights(mass):
    """A network that is the degree-one polynomial 1 - M / lambda of the one-link operator (what training
    approaches): layer 1 gives each hop a channel of its own, layer 3 weighs the second hop."""
    lam = 64.0 + mass * mass
    w1 = np.zeros((9, 8, 1), np.complex128)
    w2 = np.zeros((9, 8, 8), np.complex128)
    w3 = np.zeros((9, 1, 8), np.complex128)
    w1[0, 0, 0] = 1.0
    w2[0] = np.eye(8)
    sign = [1.0 if d % 2 == 0 else -1.0 for d in range(8)]
    for d in range(8):
        w1[1 + d, d, 0] = sign[d]
        w3[1 + d, 0, :] = sign[d] / lam
    w3[0, 0, 0] = 1.0
    return [w1, w2, w3]


def _comp(case):
    return {"none": False, "all": True, "long": "long"}[case["comp"]]


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.kind = dict(case), case["kind"]
    dims = _dims(case)
    vh = _volume(dims) // 2
    fat = _links(dims, seed)
    s.lat = stag.Lattice(dims)
    if s.kind in ("dslash", "apply_M"):
        prec = case["prec"]
        torch.cuda.synchronize()
        s.lat.upload_gauge(fat, None, precisions=(prec,), compress12=_comp(case))
        stride = s.lat.field_bytes("f64") // 48
        s.ins, s.outs, s.vals = [], [], []
        parities = [stag.EVEN, stag.ODD] if s.kind == "dslash" else [stag.EVEN]
        for k, par in enumerate(parities):
            s.ins.append(s.lat.field(par, prec, _source(dims, seed, k)))
            opar = 1 - par if s.kind == "dslash" else par
            if prec == "df64":  # exported: its storage is pairs of floats
                s.outs.append(s.lat.field(opar, prec))
                s.vals.append(torch.empty((vh, 3), dtype=torch.complex128, device="cuda"))
            else:  # a view of a tensor [3][stride] of the user's
                t = torch.zeros((3, stride), dtype=torch.complex64 if prec == "f32" else torch.complex128,
                                device="cuda")
                torch.cuda.synchronize()
                s.outs.append(s.lat.wrap_field(t, opar, prec))
                s.vals.append(t)
    elif s.kind == "upload":
        s.fat = fat
        s.lng = torch.empty_like(fat)
        stride = s.lat.field_bytes("f64") // 48
        s.b = _source(dims, seed, 0)
        s.vals = [torch.empty((vh, 3), dtype=torch.complex128, device="cuda"),
                  torch.zeros((3, stride), dtype=torch.complex64, device="cuda")]
        torch.cuda.synchronize()
        s.ins = [s.lat.field(stag.EVEN, "df64", s.b), s.lat.field(stag.EVEN, "f32", s.b)]
        s.outs = [s.lat.field(stag.ODD, "df64"), s.lat.wrap_field(s.vals[1], stag.ODD, "f32")]
    elif s.kind in ("cg", "cg_mixed", "learned", "multishift"):
        hi = case.get("prec", "df64")
        precs, comp = {hi}, False
        if s.kind == "cg_mixed":
            precs.add(case["inner"])
            comp = _comp(case)
        elif s.kind == "learned" and case["inner"] != "none":
            precs.add(case["inner"])
        elif s.kind == "multishift" and case["mixed"] != "none":
            precs |= {"f32", case["mixed"]}
        torch.cuda.synchronize()
        s.lat.upload_gauge(fat, None, precisions=tuple(sorted(precs)), compress12=comp)
        s.b = _source(dims, seed, 0)
        n = case["shifts"] if s.kind == "multishift" else 1
        s.fb = s.lat.field(stag.EVEN, hi)
        s.fx = [s.lat.field(stag.EVEN, hi) for _ in range(n)]
        s.vals = [torch.empty((vh, 3), dtype=torch.complex128, device="cuda") for _ in range(n)]
        if s.kind == "learned":
            s.net = stag.Net(s.lat, fat, 8, 1)
            s.net.set_weights(_net_weights(case["mass"]))
    elif s.kind == "batched":
        precs = {"df64"} | ({"f32", case["mixed"]} if case["mixed"] != "none" else set())
        torch.cuda.synchronize()
        s.lat.upload_gauge(fat, None, precisions=tuple(sorted(precs)))
        groups = [(s.lat, dims, case["n"])]
        if case["n2"]:
            d2 = _dims(case, True)
            s.lat2 = stag.Lattice(d2)
            fat2 = _links(d2, seed, 1)
            torch.cuda.synchronize()
            s.lat2.upload_gauge(fat2, None, precisions=tuple(sorted(precs)))
            groups.append((s.lat2, d2, case["n2"]))
        s.b, s.systems, s.vals = [], [], []
        for lat, d, n in groups:
            for _ in range(n):
                s.b.append(_source(d, seed, len(s.b)))
                s.systems.append((lat, lat.field(stag.EVEN, "df64"), lat.field(stag.EVEN, "df64"), case["mass"]))
                s.vals.append(torch.empty((_volume(d) // 2, 3), dtype=torch.complex128, device="cuda"))
    else:  # net_grad
        torch.cuda.synchronize()
        s.lat.upload_gauge(fat, None, precisions=("df64", "f32"))
        s.net = stag.Net(s.lat, fat, 8, 1)
        s.net.set_weights(_net_weights(case["mass"]))
        s.net.set_loss(case["loss"])
        b = s.lat.field(stag.EVEN, "df64", _source(dims, seed, 0))
        s.net.collect_pairs(b, case["mass"], TOL, case["stride"], case["pairs"])
    torch.cuda.synchronize()
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    case, kind = s.case, s.kind
    if kind in ("dslash", "apply_M"):
        for o, i in zip(s.outs, s.ins):
            if kind == "dslash":
                s.lat.dslash(o, i)
            else:
                s.lat.apply_M(o, i, case["mass"])
        if case["prec"] == "df64":
            for o, v in zip(s.outs, s.vals):
                o.export(v)
        return s.vals
    if kind == "upload":
        s.lat.long_links(s.fat, s.lng)
        s.lat.upload_gauge(s.fat, s.lng, precisions=("df64", "f32", "f16"), compress12=_comp(case))
        for o, i in zip(s.outs, s.ins):
            s.lat.dslash(o, i)
        s.outs[0].export(s.vals[0])
        return [s.lng] + s.vals
    if kind == "net_grad":
        loss, grads = s.net.loss_grad(0, s.net.num_pairs())
        return [loss] + [g.astype(np.complex64) for g in grads]
    if kind == "batched":
        for (_, _, fb, _), b in zip(s.systems, s.b):
            fb.import_(b)
        stag.cg_batched(s.systems, TOL, 5000, mixed=None if case["mixed"] == "none" else case["mixed"])
        for (_, fx, _, _), v in zip(s.systems, s.vals):
            fx.export(v)
        return s.vals
    s.fb.import_(s.b)
    mass = case["mass"]
    if kind == "cg":
        s.lat.cg(s.fx[0], s.fb, mass, TOL, 5000)
    elif kind == "cg_mixed":
        s.lat.cg_mixed(s.fx[0], s.fb, mass, TOL_MIXED, 5000, inner=case["inner"])
    elif kind == "learned":
        if case["inner"] == "none":
            s.net.cg(s.fx[0], s.fb, mass, TOL_MIXED, 5000)
        else:
            s.net.cg_mixed(s.fx[0], s.fb, mass, TOL_MIXED, 5000, inner=case["inner"])
    else:
        s.lat.cg_multishift(s.fx, s.fb, _shift_list(case["shifts"]), mass, TOL, 5000,
                            mixed=None if case["mixed"] == "none" else case["mixed"])
    for f, v in zip(s.fx, s.vals):
        f.export(v)
    return s.vals


# ------------------------------------------------- bytes and operations needed
def _iterations(mass, dims):
    """CG iterations, about: the lowest mode of an antiperiodic direction of Lt sites, and the mass."""
    return (40.0 + 6.2 * dims[3]) / math.sqrt(1.0 + (mass * dims[3] / 8.0) ** 2)


def work(case):
    """One pass: the paper's model of the operator (16 links, one vector read, one written; 1146 flops a site),
    and for a solve that of its iterations, with the vectors each read and written once."""
    dims, kind = _dims(case), case["kind"]
    vh = _volume(dims) / 2
    real = {"f64": 8, "df64": 8, "f32": 4, "f16": 2}
    link = {"none": 18.0, "all": 12.0, "long": 15.0}

    def op(p, comp="none"):
        return (16 * link[comp] + 12) * real[p]

    if kind == "dslash":
        return {"bytes": 2 * vh * op(case["prec"], case["comp"]), "flops": 2 * 1146 * vh}
    if kind == "apply_M":
        return {"bytes": 2 * vh * op(case["prec"], case["comp"]), "flops": (2 * 1146 + 12) * vh}
    if kind == "upload":
        # links in and products out, both read again for the copies, the copies written; the applications
        copies = 8 * (18 * 8 + 18 * 4 + 18 * 2)
        if case["comp"] != "none":
            copies += 8 * link[case["comp"]] * (4 + 2)
        return {"bytes": 2 * vh * (2 * 4 * 144 + copies) + vh * (op("df64") + op("f32", case["comp"])),
                "flops": 2 * vh * 4 * 2 * 198 + 2 * 1146 * vh}
    if kind == "net_grad":
        # per pair: r and the net's two 8-link stencils forward and backward, the residual loss's M twice
        m = 4.0 * op("f32") if case["loss"] == "residual" else 0.0
        return {"bytes": case["pairs"] * vh * (4 * 8 * 72 + m), "flops": case["pairs"] * vh * 4 * (8 * 66 + 600.0)}
    it = _iterations(case["mass"], dims)
    if kind == "batched":
        vh2 = _volume(_dims(case, True)) / 2 if case["n2"] else 0.0
        p = "df64" if case["mixed"] == "none" else "f32"
        sites = case["n"] * vh + case["n2"] * vh2
        links = 2 * 288 * real[p]
        return {"bytes": it * (links * (vh + vh2) + sites * (2 * 12 + 60) * real[p]), "flops": it * sites * 2364.0}
    if kind == "multishift":
        p = "df64" if case["mixed"] == "none" else "f32"
        return {"bytes": it * vh * (2 * op(p) + 18 * 8 + 24 * 8 * case["shifts"]),
                "flops": it * vh * (2292.0 + 12 + 24 * case["shifts"])}
    p = case.get("prec") or case["inner"]
    if kind != "cg":
        it *= 1.1  # one more decade of the residual
    if p == "none":
        p = "df64"
    net = 0.0
    if kind == "learned":
        it *= 0.56
        net = 16 * 24 + 2 * 128 + 36
    return {"bytes": it * vh * (2 * op(p, case.get("comp", "none")) + 60 * real[p] + net), "flops": it * vh * 2364.0}


# ------------------------------------------------------------ 64-bit reference
class _Op:
    """The operator in plain torch, complex128: per parity one [Vh][3][48] matrix (the 16 hops side by side) and
    the 16 neighbours of every site."""

    def __init__(self, dims, fat, lng, c1=C1, c3=C3, naik=True):
        dev = fat.device
        L = dims
        V = _volume(dims)
        i = torch.arange(V, device=dev)
        x = [i % L[0], i // L[0] % L[1], i // (L[0] * L[1]) % L[2], i // (L[0] * L[1] * L[2])]
        step = [1, L[0], L[0] * L[1], L[0] * L[1] * L[2]]
        par = (x[0] + x[1] + x[2] + x[3]) & 1
        self.sites = [torch.nonzero(par == p).flatten() for p in (0, 1)]
        self.A, self.idx = [], []
        for p in (0, 1):
            site = self.sites[p]
            A = torch.empty((site.numel(), 3, 48 if naik else 24), dtype=torch.complex128, device=dev)
            idx = torch.empty((site.numel(), 16 if naik else 8), dtype=torch.int64, device=dev)
            h = 0
            for s, G, c in ((1, fat, c1), (3, lng, c3))[: 2 if naik else 1]:
                for mu in range(4):
                    xm = x[mu][site]
                    es = sum((x[nu][site] for nu in range(mu)), torch.zeros_like(xm))
                    eta = 1.0 - 2.0 * (es & 1).double()
                    for d in (s, -s):
                        y = torch.remainder(xm + d, L[mu])
                        w = torch.div(xm + d - y, L[mu], rounding_mode="floor").abs()
                        b = torch.where((w & 1) == 1, BC[mu], 1.0).double() if BC[mu] < 0 else torch.ones_like(eta)
                        j = site + (y - xm) * step[mu]
                        M = G[mu][site] if d > 0 else -G[mu][j].conj().transpose(1, 2)
                        A[:, :, 3 * h:3 * h + 3] = M * (c * eta * b)[:, None, None]
                        idx[:, h] = j >> 1
                        h += 1
            self.A.append(A)
            self.idx.append(idx)

    def hops(self, p, v):
        """The neighbours' vectors of parity 1 - p, [Vh][hops][3]."""
        return v[self.idx[p]]

    def D(self, p, v):
        out = torch.empty((self.A[p].shape[0], 3), dtype=torch.complex128, device=v.device)
        for a in range(0, out.shape[0], 1 << 18):
            b = min(out.shape[0], a + (1 << 18))
            g = v[self.idx[p][a:b]].reshape(b - a, 1, -1)
            out[a:b] = (self.A[p][a:b] * g).sum(2)
        return out

    def M(self, v, m2):
        return m2 * v - self.D(0, self.D(1, v))


def _dot(a, b):
    return torch.sum(a.real * b.real + a.imag * b.imag)


def _cg(op, b, mass, tol=2e-14, limit=4000, keep=None):
    """Plain CG in 64 bits; keep(k, r): called with the residual of every iteration."""
    m2 = mass * mass
    x, r, p = torch.zeros_like(b), b.clone(), b.clone()
    rr = _dot(r, r)
    stop = tol * tol * rr
    for k in range(limit):
        if keep is not None and keep(k, x, r):
            break
        if (keep is not None or k % 10 == 0) and bool(rr <= stop):
            break
        Ap = op.M(p, m2)
        al = rr / _dot(p, Ap)
        x = x + al * p
        r = r - al * Ap
        new = _dot(r, r)
        p = r + (new / rr) * p
        rr = new
    return x


def _multishift(op, b, mass, shifts, tol=2e-14, limit=4000):
    """Jegerlehner's shifted CG in 64 bits (the smallest shift is the base system)."""
    base = min(shifts)
    n = len(shifts)
    dl = torch.tensor([s - base for s in shifts], dtype=torch.float64, device=b.device)
    x = [torch.zeros_like(b) for _ in range(n)]
    p = [b.clone() for _ in range(n)]
    r, q = b.clone(), b.clone()
    z = torch.ones(n, dtype=torch.float64, device=b.device)
    zp = z.clone()
    al0, be0 = torch.ones((), dtype=torch.float64, device=b.device), torch.zeros((), dtype=torch.float64, device=b.device)
    rr = _dot(r, r)
    stop = tol * tol * rr
    for k in range(limit):
        if k % 10 == 0 and bool(rr <= stop):
            break
        Ap = op.M(q, mass * mass + base)
        al = rr / _dot(q, Ap)
        zn = z * zp * al0 / (al * be0 * (zp - z) + zp * al0 * (1 + dl * al))
        for s in range(n):
            x[s] = x[s] + (al * zn[s] / z[s]) * p[s]
        r = r - al * Ap
        new = _dot(r, r)
        be = new / rr
        q = r + be * q
        for s in range(n):
            p[s] = zn[s] * r + (be * (zn[s] / z[s]) ** 2) * p[s]
        zn = torch.where(zn.abs() > 1e-150, zn, torch.full_like(zn, 1e-150))
        zp, z, al0, be0, rr = z, zn, al, be, new
    return x


def _naik(dims, U):
    """N_mu(x) = U_mu(x) U_mu(x+mu) U_mu(x+2mu), periodic."""
    def mul(a, b):
        return torch.stack([(a[:, :, k, None] * b[:, k, None, :]) for k in range(3)]).sum(0)

    out = []
    for mu in range(4):
        u = U[mu].view(dims[3], dims[2], dims[1], dims[0], 3, 3)
        ax = 3 - mu
        u1 = torch.roll(u, -1, ax).reshape(-1, 3, 3)
        u2 = torch.roll(u, -2, ax).reshape(-1, 3, 3)
        out.append(mul(mul(U[mu], u1), u2))
    return torch.stack(out)


def _pad(v, stride):
    """[Vh][3] in a field's storage order [3][stride]."""
    out = torch.zeros((3, stride), dtype=v.dtype, device=v.device)
    out[:, :v.shape[0]] = v.T
    return out


def _net_layers(op1, w, r):
    """The network's three layers on the phased one-link transports; r on the even sites, even sites of the
    result (psi: channels [C][Vh][3] on each parity)."""
    sgn = torch.tensor([1.0, -1.0] * 4, device=r.device)  # op1 carries minus on the backward hops

    def transports(p, v):  # v [C][Vh][3] on 1 - p -> [8][C][Vh][3]
        g = v[:, op1.idx[p]]  # [C][Vh][8][3]
        A = op1.A[p].view(-1, 3, 8, 3)
        return torch.stack([sgn[d] * (A[:, :, d, :] * g[:, :, d, None, :]).sum(-1) for d in range(8)])

    def layer(wl, psi):
        out = []
        for p in (0, 1):
            o = 0
            if psi[p] is not None:
                o = torch.einsum("oi,ixc->oxc", wl[0], psi[p])
            if psi[1 - p] is not None:
                o = o + torch.einsum("doi,dixc->oxc", wl[1:], transports(p, psi[1 - p]))
            out.append(o)
        return out

    psi = [r[None], None]
    for wl in w:
        psi = layer(wl, psi)
    return psi[0][0]


def exact(case, seed):
    dims, kind = _dims(case), case["kind"]
    V = _volume(dims)
    cost = V * {"cg": 1, "cg_mixed": 1, "learned": 1, "multishift": 1.5}.get(kind, 0)
    if kind == "batched":
        cost = V * case["n"] + _volume(_dims(case, True)) * case["n2"]
    if cost > 1.3 * (1 << 21) * 2 or (kind == "net_grad" and V > 16 ** 3 * 32):
        return None
    fat = _links(dims, seed)
    lng = _naik(dims, fat)
    stride = -(-(V // 2) // 256) * 256
    if kind == "dslash":
        op = _Op(dims, fat, lng)
        out = [op.D(1, _source(dims, seed, 0)), op.D(0, _source(dims, seed, 1))]
        return out if case["prec"] == "df64" else [_pad(v, stride) for v in out]
    if kind == "apply_M":
        v = _Op(dims, fat, lng).M(_source(dims, seed, 0), case["mass"] ** 2)
        return [v if case["prec"] == "df64" else _pad(v, stride)]
    if kind == "upload":
        v = _Op(dims, fat, lng).D(1, _source(dims, seed, 0))
        return [lng, v, _pad(v, stride)]
    if kind == "multishift":
        return _multishift(_Op(dims, fat, lng), _source(dims, seed, 0), case["mass"], _shift_list(case["shifts"]))
    if kind == "batched":
        out, k = [], 0
        op = _Op(dims, fat, lng)
        for _ in range(case["n"]):
            out.append(_cg(op, _source(dims, seed, k), case["mass"]))
            k += 1
        if case["n2"]:
            d2 = _dims(case, True)
            fat2 = _links(d2, seed, 1)
            op = _Op(d2, fat2, _naik(d2, fat2))
            for _ in range(case["n2"]):
                out.append(_cg(op, _source(d2, seed, k), case["mass"]))
                k += 1
        return out
    if kind == "net_grad":
        op, op1 = _Op(dims, fat, lng), _Op(dims, fat, None, 1.0, 0.0, naik=False)
        b = _source(dims, seed, 0)
        sol = _cg(op, b, case["mass"], TOL)
        pairs = []

        def keep(k, x, r):
            if k and k % case["stride"] == 0 and len(pairs) < case["pairs"]:
                pairs.append((r, sol - x))
            return len(pairs) >= case["pairs"]

        _cg(op, b, case["mass"], TOL, keep=keep)
        w = [torch.from_numpy(a).cuda().requires_grad_(True) for a in _net_weights(case["mass"])]
        total = 0.0
        for r, e in pairs:
            z = _net_layers(op1, w, r)
            d, n = (op.M(z, case["mass"] ** 2) - r, r) if case["loss"] == "residual" else (z - e, e)
            loss = _dot(d, d) / _dot(n, n)
            loss.backward()
            total += float(loss.detach())
        # torch's gradient of a real value is 2 dL/dW*
        return [total] + [(0.5 * a.grad).cpu().numpy() for a in w]
    return [_cg(_Op(dims, fat, lng), _source(dims, seed, 0), case["mass"])]
