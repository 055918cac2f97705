"""The rules that choose between forms of one kernel: which form runs, on both
sides of each line, and that the forms agree."""
import numpy as np
import pytest
from kernel_trace import launched

import oracle
from paper_1411_2087_gb300 import stag, synth

pytestmark = pytest.mark.gpu


def links(dims, seed):
    return synth.su3_field(dims, 0.3, seed, device="cuda")


def dslash_name(names):
    return [n for n in names if "dslash" in n]


# FP32, one thread per site, 128-thread blocks: 1216 blocks are one wave at
# eight per SM (1024 threads), 1064 at seven, 912 at six
@pytest.mark.parametrize("compress,cases", [
    (False, [(66, 7), (68, 8), (76, 8), (78, 7)]),     # 1056, 1088, 1216, 1248 blocks
    ("long", [(66, 7), (68, 8), (76, 8), (78, 7)]),
    (True, [(56, 6), (58, 8), (76, 8), (78, 6), (248, 6), (296, 8)]),  # 896, 928, 1216, 1248, 3968, 4736
])
def test_fp32_threads_per_sm_by_waves(compress, cases):
    cm = {False: 0, "long": 2, True: 3}[compress]
    for Lt, want in cases:
        dims = (16, 16, 16, Lt)
        Vh = 2048 * Lt
        with stag.Lattice(dims) as lat:
            lat.upload_gauge(links(dims, 91), None, precisions=("f32",), compress12=compress)
            fe = lat.field(stag.EVEN, "f32", synth.gaussian_colour_field(Vh, 92).numpy())
            fo, fm = lat.field(stag.ODD, "f32"), lat.field(stag.EVEN, "f32")

            def run():
                lat.dslash(fo, fe)
                lat.apply_M(fm, fe, 0.1)

            names = dslash_name(launched(run))
            assert names == [f"void dslash_kernel_capped<1, {e}, 128, {cm}, {want}>" for e in (0, 0, 1)], (Lt, names)
            got = fo.export()
            lat.set_tuning("f32", "dslash", 128, 1)  # the compiler's choice of registers
            lat.dslash(fo, fe)
            assert np.array_equal(fo.export(), got), Lt
            lat.set_tuning("f32", "dslash", 256, 2)
            lat.dslash(fo, fe)
            assert np.array_equal(fo.export(), got), Lt


TOL = {"df64": 1e-12, "f32": 2e-6}
TOL_M = {"df64": 1e-12, "f32": 5e-6}


# both sides of the lines between the split form and one thread per site
@pytest.mark.parametrize("prec,Lt,split", [("df64", 34, True), ("df64", 36, False), ("df64", 56, False),
                                           ("df64", 58, True), ("f32", 28, True), ("f32", 30, False)])
def test_single_calls_across_the_split_lines(prec, Lt, split):
    dims = (16, 16, 16, Lt)
    Vh = 2048 * Lt
    U = links(dims, 93).cpu().numpy()
    N = oracle.long_links(dims, U)
    psi_e = synth.gaussian_colour_field(Vh, 94).numpy()
    psi_o = synth.gaussian_colour_field(Vh, 95).numpy()
    with stag.Lattice(dims) as lat:
        lat.upload_gauge(U, N, precisions=(prec,))
        fe, fo = lat.field(stag.EVEN, prec, psi_e), lat.field(stag.ODD, prec, psi_o)
        oo, oe, om = lat.field(stag.ODD, prec), lat.field(stag.EVEN, prec), lat.field(stag.EVEN, prec)

        def run():
            lat.dslash(oo, fe)
            lat.dslash(oe, fo)
            lat.apply_M(om, fe, 0.3)

        names = dslash_name(launched(run))
        assert len(names) == 4 and all(("split" in n) == split for n in names), names
        for got, want, tol in ((oo, oracle.dslash_parity(dims, U, N, 1, psi_e), TOL),
                               (oe, oracle.dslash_parity(dims, U, N, 0, psi_o), TOL),
                               (om, oracle.apply_M(dims, U, N, 0.3, psi_e), TOL_M)):
            assert np.abs(got.export() - want).max() <= tol[prec] * np.abs(want).max()


@pytest.mark.parametrize("inner,Lt,split", [(None, 34, True), (None, 36, False), (None, 56, False), (None, 58, True),
                                            ("f32", 34, True), ("f32", 36, False)])
def test_solves_across_the_split_lines(inner, Lt, split):
    dims, mass = (16, 16, 16, Lt), 0.5
    U = links(dims, 96).cpu().numpy()
    N = oracle.long_links(dims, U)
    b = synth.gaussian_colour_field(2048 * Lt, 97).numpy()
    with stag.Lattice(dims) as lat:
        lat.upload_gauge(U, N, precisions=("df64", "f32"))
        fb, x = lat.field(stag.EVEN, "df64", b), lat.field(stag.EVEN, "df64")

        def solve():
            info = lat.cg_mixed(x, fb, mass, 1e-10, 2000, inner=inner) if inner else lat.cg(x, fb, mass, 1e-10, 2000)
            assert info["return"] == stag.OK
            r = b - oracle.apply_M(dims, U, N, mass, x.export())
            assert np.linalg.norm(r) <= 1.05e-10 * np.linalg.norm(b)

        solve()
        lat.set_cg_launch("host")  # the same kernels, launched one by one
        p = 1 if inner else 3
        names = [n for n in launched(solve) if f"<{p}, " in n and "dslash" in n]
        assert names and all(("split" in n) == split for n in names), set(names)


@pytest.mark.parametrize("Lt,pair", [(72, False), (76, True)])  # 147456, 155648 sites per parity
def test_16_bit_pair_form_is_the_untuned_default(Lt, pair):
    """16-bit D on 12-real links, nothing tuned, against the oracle (the
    storage format's tolerance), and the bits of the one-site form."""
    dims = (16, 16, 16, Lt)
    Vh = 2048 * Lt
    U = links(dims, 98).cpu().numpy()
    N = oracle.long_links(dims, U)
    psi_e = synth.gaussian_colour_field(Vh, 99).numpy()
    psi_o = synth.gaussian_colour_field(Vh, 100).numpy()
    with stag.Lattice(dims) as lat:
        lat.upload_gauge(U, N, precisions=("f16",), compress12=True)
        fe, fo = lat.field(stag.EVEN, "f16", psi_e), lat.field(stag.ODD, "f16", psi_o)
        oo, oe = lat.field(stag.ODD, "f16"), lat.field(stag.EVEN, "f16")

        def run():
            lat.dslash(oo, fe)
            lat.dslash(oe, fo)

        names = dslash_name(launched(run))
        assert len(names) == 2 and all(("pair16" in n) == pair for n in names), names
        got = oo.export(), oe.export()
        for g, want in zip(got, (oracle.dslash_parity(dims, U, N, 1, psi_e), oracle.dslash_parity(dims, U, N, 0, psi_o))):
            assert np.abs(g - want).max() <= 3e-4 * np.abs(want).max()
        lat.set_tuning("f16", "dslash", 128, 1)
        run()
        assert np.array_equal(oo.export(), got[0]) and np.array_equal(oe.export(), got[1])


@pytest.mark.parametrize("prec,compress,Lt", [("f32", False, 32), ("f32", True, 72), ("df64", False, 34),
                                              ("f16", True, 76)])
def test_decomposed_dslash_takes_the_single_calls_form(prec, compress, Lt):
    """Between the single calls' line and the solves' (and where their launches
    differ otherwise) the slab-decomposed Dslash keeps the single call's bits."""
    dims = (16, 16, 16, Lt)
    with stag.Lattice(dims) as lat:
        lat.upload_gauge(links(dims, 101), None, precisions=(prec,), compress12=compress)
        fe = lat.field(stag.EVEN, prec, synth.gaussian_colour_field(2048 * Lt, 102).numpy())
        one, slabs, rank = (lat.field(stag.ODD, prec) for _ in range(3))
        lat.dslash(one, fe)
        lat.dd_dslash(slabs, fe, 3)
        comm = stag.HostComm(0, 1, lambda p, n: (n, p), lambda v: v)
        d = stag.DDRank(lat, comm)
        d.dslash(rank, fe)
        want = one.export()
        assert np.array_equal(slabs.export(), want)
        assert np.array_equal(rank.export(), want)
        d.close()


def test_training_pairs_give_the_same_numbers_alone_and_in_groups():
    """Between the solves' line and the training launches' (groups of three
    pairs here): the kernels are the same per pair, so a group's loss and
    gradient are the sums of its pairs' up to FP64 rounding."""
    dims, mass = (16, 16, 16, 36), 0.1
    U = links(dims, 103).cpu().numpy()
    with stag.Lattice(dims) as lat:
        lat.upload_gauge(U, None, precisions=("df64", "f32"))
        net = stag.Net(lat, U, 8, 5)
        net.set_loss("residual")
        b = lat.field(stag.EVEN, "df64", synth.gaussian_colour_field(2048 * 36, 104).numpy())
        assert net.collect_pairs(b, mass, 1e-10, 3, 4) == 4
        loss, grads = net.loss_grad(0, 4)
        parts = [net.loss_grad(k, 1) for k in range(4)]
        assert abs(loss - sum(p[0] for p in parts)) <= 1e-10 * abs(loss)
        for layer, g in enumerate(grads):
            want = sum(p[1][layer] for p in parts)
            assert np.abs(g - want).max() <= 1e-10 * max(np.abs(p[1][layer]).max() for p in parts)
