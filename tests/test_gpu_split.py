"""The split form of the stencil (one site's hops spread over a block's warps,
summed in shared memory) at the sizes where it changes shape:

* sites per parity that do not fill a block of 32 sites, lattices with
  extents below the three-link hop, and both sides of the line between eight
  and four warps per block and of the line to one thread per site: D and M
  against the oracle, to the tolerances of the storage formats;
* the solve's scalars through it: a CG whose <p, Mp> comes from the split M;
* the 16-bit M with partials at a block size without a pair form (512
  threads, full links): its partials are counted for the form that runs.
"""
import numpy as np
import pytest

import oracle
from paper_1411_2087_gb300 import stag, synth

pytestmark = pytest.mark.gpu

TOL = {"f64": 1e-12, "df64": 1e-12, "f32": 2e-6}
TOL_M = {"f64": 1e-12, "df64": 1e-12, "f32": 5e-6}


def rel_err(got, want):
    return np.abs(got - want).max() / np.abs(want).max()


@pytest.mark.parametrize("dims", [
    (2, 2, 2, 2), (2, 6, 4, 2), (6, 4, 6, 10),
    (16, 16, 8, 16),   # 16384 sites per parity: eight warps
    (16, 16, 10, 14),  # 17920: four
    (16, 16, 14, 14),  # 25088: 12-real FP32 links on one thread per site
])
@pytest.mark.parametrize("prec,compress", [("f64", False), ("df64", False), ("f32", False), ("f32", True),
                                           ("f32", "long")])
def test_split_dslash_and_m(dims, prec, compress):
    U = synth.su3_field(dims, 0.3, 61).numpy()
    N = oracle.long_links(dims, U)
    Vh = int(np.prod(dims)) // 2
    psi_e = synth.gaussian_colour_field(Vh, 62).numpy()
    psi_o = synth.gaussian_colour_field(Vh, 63).numpy()
    with stag.Lattice(dims, bc=(1.0, -1.0, 1.0, -1.0)) as lat:
        lat.upload_gauge(U, N, precisions=(prec,), compress12=compress)
        fe, fo = lat.field(stag.EVEN, prec, psi_e), lat.field(stag.ODD, prec, psi_o)
        oo, oe, om = lat.field(stag.ODD, prec), lat.field(stag.EVEN, prec), lat.field(stag.EVEN, prec)
        lat.dslash(oo, fe)
        lat.dslash(oe, fo)
        lat.apply_M(om, fe, 0.3)
        bc = (1.0, -1.0, 1.0, -1.0)
        assert rel_err(oo.export(), oracle.dslash_parity(dims, U, N, 1, psi_e, bc=bc)) <= TOL[prec]
        assert rel_err(oe.export(), oracle.dslash_parity(dims, U, N, 0, psi_o, bc=bc)) <= TOL[prec]
        assert rel_err(om.export(), oracle.apply_M(dims, U, N, 0.3, psi_e, bc=bc)) <= TOL_M[prec]


@pytest.mark.parametrize("dims", [(6, 4, 6, 10), (16, 16, 10, 14)])
@pytest.mark.parametrize("prec", ["f64", "df64"])
def test_solve_through_the_split_m(dims, prec):
    U = synth.su3_field(dims, 0.3, 64).numpy()
    N = oracle.long_links(dims, U)
    Vh = int(np.prod(dims)) // 2
    b = synth.gaussian_colour_field(Vh, 65).numpy()
    _, want = oracle.cg(dims, U, N, 0.2, b, tol=1e-10)
    with stag.Lattice(dims) as lat:
        lat.upload_gauge(U, N, precisions=(prec,))
        x = lat.field(stag.EVEN, prec)
        info = lat.cg(x, lat.field(stag.EVEN, prec, b), 0.2, 1e-10, 5000)
        assert info["return"] == stag.OK
        assert abs(info["iters"] - want["iters"]) <= max(3, 0.01 * want["iters"])
        r = b - oracle.apply_M(dims, U, N, 0.2, x.export())
        assert np.linalg.norm(r) <= 1.05e-10 * np.linalg.norm(b)


def test_pair_request_without_a_pair_form():
    dims = (32, 16, 16, 32)  # above the size up to which the Dslash's last block sums <p, Mp>
    U = synth.su3_field(dims, 0.3, 66)
    Vh = int(np.prod(dims)) // 2
    b = synth.gaussian_colour_field(Vh, 67).numpy()
    iters = []
    with stag.Lattice(dims) as lat:
        lat.upload_gauge(U.numpy(), None, precisions=("df64", "f16"))
        fb = lat.field(stag.EVEN, "df64", b)
        for block, regs in ((128, 1), (512, 3)):
            lat.set_tuning("f16", "dslash", block, regs)
            lat.set_tuning("f16", "M", block, regs)
            x = lat.field(stag.EVEN, "df64")
            info = lat.cg_mixed(x, fb, 0.2, 1e-10, 5000, inner="f16")
            assert info["return"] == stag.OK
            iters.append(info["iters"])
    assert abs(iters[0] - iters[1]) <= max(3, 0.01 * iters[0]), iters
