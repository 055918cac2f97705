"""Gauge upload: the bits of the copies and the buffers kept between uploads.

* The double-float split of a link entry, hi = float(d), lo = float(d - hi),
  and the FP32 copy, float(d), for entries of every kind the integer split
  distinguishes (signs, ties to even both ways, carries into the next binade,
  exact floats, the ends of its exponent range and the values beyond it that
  take the plain conversions), read back exactly through D on unit sources.
* A second upload into the first one's buffers (other field, other scale,
  other formats and compression) gives what a fresh lattice gives, and a
  refused one in between leaves no gauge field.
* The SU(3) check decides links on both sides of 1e-6, also where its FP32
  part alone could not tell.
"""
import numpy as np
import pytest

import oracle
from paper_1411_2087_gb300 import stag, synth

pytestmark = pytest.mark.gpu


def special_values(rng, n):
    e = rng.integers(-80, 120, n).astype(np.float64)
    v = np.ldexp(1.0 + rng.random(n), e.astype(int))
    k = n // 8
    ulp = 2.0 ** -23
    v[:k] = 1.0 + ulp * rng.integers(0, 1 << 23, k)                      # exact floats
    v[k:2 * k] = v[:k] + 0.5 * ulp                                        # ties
    v[2 * k:3 * k] = v[:k] + 0.5 * ulp + 2.0 ** -52                       # just above
    v[3 * k:4 * k] = 2.0 - rng.integers(1, 5, k) * 2.0 ** -52             # carry into the next binade
    v[4 * k:4 * k + 6] = [0.0, 2.0 ** -70, 2.0 ** -71, 2.0 ** 126, 2.0 ** 127, 1e-320]
    return v * rng.choice([-1.0, 1.0], n)


@pytest.mark.parametrize("prec", ["df64", "f32", "f64"])
def test_split_of_link_entries(prec):
    dims = (4, 4, 4, 4)
    V = 256
    rng = np.random.default_rng(71)
    U = (special_values(rng, 4 * V * 9) + 1j * special_values(rng, 4 * V * 9)).reshape(4, V, 3, 3)
    N = np.zeros_like(U)

    def want(d):
        with np.errstate(under="ignore"):
            hi = d.astype(np.float32)
            lo = (d - hi).astype(np.float32)
        return d if prec == "f64" else hi.astype(np.float64) + (lo if prec == "df64" else 0.0)

    # even site y, its forward neighbour along mu: out(y + mu) = -U_mu(y)^+ psi(y)
    y = [2, 0, 0, 0]
    iy = y[0] + 4 * (y[1] + 4 * (y[2] + 4 * y[3]))
    with stag.Lattice(dims, bc=(1.0, 1.0, 1.0, 1.0)) as lat:
        lat.upload_gauge(U, N, c1=1.0, c3=0.0, precisions=(prec,))
        for a in range(3):
            psi = np.zeros((V // 2, 3), np.complex128)
            psi[iy >> 1, a] = 1.0
            out = lat.field(stag.ODD, prec)
            lat.dslash(out, lat.field(stag.EVEN, prec, psi))
            got = out.export()
            for mu in range(4):
                x = list(y)
                x[mu] = (x[mu] + 1) % 4
                ix = x[0] + 4 * (x[1] + 4 * (x[2] + 4 * x[3]))
                eta = (-1.0) ** sum(y[:mu])
                row = -eta * np.conj(U[mu, iy, a, :])
                assert np.array_equal(got[ix >> 1].real, want(row.real)), (mu, a)
                assert np.array_equal(got[ix >> 1].imag, want(row.imag)), (mu, a)
                x[mu] = (y[mu] - 1) % 4
                ix = x[0] + 4 * (x[1] + 4 * (x[2] + 4 * x[3]))
                col = eta * U[mu, ix, :, a] if mu == 0 else (-1.0) ** sum(x[:mu]) * U[mu, ix, :, a]
                assert np.array_equal(got[ix >> 1].real, want(col.real)), (mu, a)


def test_second_upload_into_kept_buffers():
    dims = (6, 4, 6, 10)
    Vh = int(np.prod(dims)) // 2
    A, B = synth.su3_field(dims, 0.3, 72).numpy(), synth.su3_field(dims, 0.4, 73).numpy()
    psi = synth.gaussian_colour_field(Vh, 74).numpy()
    seq = [(A, ("f64", "df64", "f32", "f16"), True), (1.5 * B, ("df64", "f32", "f16"), False),
           (B, ("f32", "f16"), "long"), (A, ("f64", "f32"), True), (B, ("df64", "f16"), True)]

    def apply(lat, precs):
        res = []
        for p in precs:
            o = lat.field(stag.ODD, p)
            lat.dslash(o, lat.field(stag.EVEN, p, psi))
            res.append(o.export())
        return res

    with stag.Lattice(dims) as lat:
        for U, precs, comp in seq:
            lat.upload_gauge(U, None, precisions=precs, compress12=comp)
            got = apply(lat, precs)
            with stag.Lattice(dims) as fresh:
                fresh.upload_gauge(U, None, precisions=precs, compress12=comp)
                for g, w in zip(got, apply(fresh, precs)):
                    assert np.array_equal(g, w), (precs, comp)
            if "df64" in precs and "f16" in precs:  # the solvers' graphs follow the upload
                x = lat.field(stag.EVEN, "df64")
                info = lat.cg_mixed(x, lat.field(stag.EVEN, "df64", psi), 0.2, 1e-10, 5000, inner="f16")
                assert info["return"] == stag.OK
                r = psi - oracle.apply_M(dims, U, oracle.long_links(dims, U), 0.2, x.export())
                assert np.linalg.norm(r) <= 1.05e-10 * np.linalg.norm(psi)
            with pytest.raises(stag.StagError):  # not in SU(3)
                lat.upload_gauge(1.01 * A, None, precisions=("f32",), compress12=True)
            with pytest.raises(stag.StagError):
                apply(lat, precs[:1])


@pytest.mark.parametrize("dev,ok", [(0.0, True), (6e-7, True), (9.5e-7, True), (1.05e-6, False), (1e-3, False)])
@pytest.mark.parametrize("kind", ["length", "phase"])
def test_su3_check_at_its_limit(dev, ok, kind):
    dims = (4, 4, 4, 4)
    U = synth.su3_field(dims, 0.3, 75).numpy()
    if kind == "length":
        U[2, 77, 1] *= np.sqrt(1.0 + dev)      # |row 1|^2 = 1 + dev (the determinant moves half as far)
    else:
        U[2, 77] *= np.exp(1j * dev / 3.0)     # det = exp(i dev), still unitary
    N = synth.su3_field(dims, 0.3, 76).numpy()
    with stag.Lattice(dims) as lat:
        if ok:
            lat.upload_gauge(U, N, precisions=("f32",), compress12=True)
        else:
            with pytest.raises(stag.StagError):
                lat.upload_gauge(U, N, precisions=("f32",), compress12=True)


# a warp of the scan takes every 97280th link from its 32 on: one link off in
# its first, second and third chunk and at the end of either field
@pytest.mark.parametrize("field", [0, 1])
@pytest.mark.parametrize("link", [0, 97279, 97280, 97280 + 33, 2 * 97280 + 7, -1])
def test_su3_check_finds_a_link_anywhere(field, link):
    dims = (10, 14, 14, 30)
    V = int(np.prod(dims))
    assert 2 * 97280 + 7 < 4 * V
    U = np.broadcast_to(np.eye(3, dtype=np.complex128), (4, V, 3, 3)).copy()
    bad = U.copy()
    bad.reshape(-1, 3, 3)[link] *= np.exp(1e-5j)
    with stag.Lattice(dims) as lat:
        lat.upload_gauge(U, U, precisions=("f32",), compress12=True)
        with pytest.raises(stag.StagError):
            lat.upload_gauge(*((bad, U) if field == 0 else (U, bad)), precisions=("f32",), compress12=True)
