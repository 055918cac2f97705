"""The Dslash candidates of the autotuner on lattices large enough for the
one-thread-per-site kernels (small ones have a single form without them):
every block size and register variant runs the kernel it names, D and M give
the same bits, and the solvers converge with every M candidate."""
import numpy as np
import pytest
from kernel_trace import launched

import oracle
from paper_1411_2087_gb300 import stag, synth

pytestmark = pytest.mark.gpu

CASES = [("f64", False, 20), ("df64", False, 36), ("f32", False, 36), ("f32", True, 14), ("f32", "long", 14)]
CANDIDATES = [(b, r) for b in (64, 128, 256, 512) for r in (1, 2)]


def kernel_of(prec, compress, epi, block, regs):
    p = stag.PREC[prec]
    cm = {False: 0, True: 3, "long": 2}[compress]
    kind = {1: "dslash_kernel<", 2: "dslash_kernel_capped<"}[regs]
    return f"void {kind}{p}, {epi}, {block}, {cm}"


@pytest.mark.parametrize("prec,compress,Lt", CASES)
def test_every_candidate_runs_and_agrees(prec, compress, Lt):
    dims = (16, 16, 16, Lt)
    U = synth.su3_field(dims, 0.3, 31).numpy()
    psi = synth.gaussian_colour_field(2048 * Lt, 32).numpy()
    with stag.Lattice(dims) as lat:
        lat.upload_gauge(U, None, precisions=(prec,), compress12=compress)
        fe = lat.field(stag.EVEN, prec, psi)
        fo, fm = lat.field(stag.ODD, prec), lat.field(stag.EVEN, prec)
        lat.dslash(fo, fe)
        lat.apply_M(fm, fe, 0.1)
        want_d, want_m = fo.export(), fm.export()
        for block, regs in CANDIDATES:
            lat.set_tuning(prec, "dslash", block, regs)
            names = [n for n in launched(lambda: lat.dslash(fo, fe)) if "dslash" in n]
            assert len(names) == 1 and names[0].startswith(kernel_of(prec, compress, 0, block, regs)), names
            lat.apply_M(fm, fe, 0.1)
            assert np.array_equal(fo.export(), want_d), (block, regs)
            assert np.array_equal(fm.export(), want_m), (block, regs)


@pytest.mark.parametrize("prec,compress,Lt", CASES)
def test_solves_with_every_m_candidate(prec, compress, Lt):
    dims, mass = (16, 16, 16, Lt), 0.5
    U = synth.su3_field(dims, 0.3, 33).numpy()
    N = oracle.long_links(dims, U)
    b = synth.gaussian_colour_field(2048 * Lt, 34).numpy()
    hi = "df64" if prec == "f32" else prec
    with stag.Lattice(dims) as lat:
        lat.upload_gauge(U, N, precisions=tuple({hi, prec}), compress12=compress)
        lat.set_cg_launch("host")  # the solve's kernels, launched one by one
        fb, x = lat.field(stag.EVEN, hi, b), lat.field(stag.EVEN, hi)
        for block, regs in CANDIDATES:
            lat.set_tuning(prec, "M", block, regs)

            def solve():
                info = lat.cg(x, fb, mass, 1e-10, 2000) if hi == prec else lat.cg_mixed(x, fb, mass, 1e-10, 2000, inner=prec)
                assert info["return"] == stag.OK

            names = {n for n in launched(solve) if f"<{stag.PREC[prec]}, 5, " in n}
            assert len(names) == 1 and names.pop().startswith(kernel_of(prec, compress, 5, block, regs)), (block, regs)
            r = b - oracle.apply_M(dims, U, N, mass, x.export())
            assert np.linalg.norm(r) <= 1.05e-10 * np.linalg.norm(b), (block, regs)
