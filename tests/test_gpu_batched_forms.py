"""The two forms of the batched double-float and FP64 Dslash: one thread per
(site, system) above 70000 (FP64: 100000, and 68097 to 77824) items of a batch,
at both block sizes, and the split form below, with groups of three systems, whose blocks
end inside a site.  Residuals recomputed by the oracle, and the kernel that
ran read from a trace."""
import numpy as np
import pytest
from kernel_trace import launched

import oracle
from paper_1411_2087_gb300 import stag, synth

pytestmark = pytest.mark.gpu


# (Lt, systems): 16^3 x Lt, 2048 Lt items per system, in groups of four and of
# the rest; the two lattices' batches lie on both sides of each line
@pytest.mark.parametrize("prec,sizes,split", [
    ("df64", [(10, 3)], True),           # 61440 items
    ("df64", [(4, 7), (2, 3)], True),    # 69632, three groups
    ("df64", [(12, 3)], False),          # 73728
    ("df64", [(8, 7), (2, 3)], False),   # 126976
    ("f64", [(16, 3)], True),            # 98304
    ("f64", [(6, 7), (2, 3)], True),     # 98304
    ("f64", [(18, 3)], False),           # 110592
    ("f64", [(12, 3)], False),           # 73728: one wave of the other form
    ("f64", [(10, 4)], True),            # 81920
    ("f64", [(8, 7), (2, 3)], False),    # 126976
])
def test_batched_forms(prec, sizes, split):
    mass = 0.5
    lats, fields, host = [], [], []
    for k, (Lt, n) in enumerate(sizes):
        dims = (16, 16, 16, Lt)
        U = synth.su3_field(dims, 0.3, 21 + k).numpy()
        N = oracle.long_links(dims, U)
        lat = stag.Lattice(dims)
        lats.append(lat)
        lat.upload_gauge(U, N, precisions=(prec,))
        for i in range(n):
            b = synth.gaussian_colour_field(2048 * Lt, 100 + 10 * k + i).numpy()
            fields.append((lat, lat.field(stag.EVEN, prec), lat.field(stag.EVEN, prec, b), mass * (1 + 0.1 * i)))
            host.append((dims, U, N, b))
    for block in (128, 256):
        for lat in lats:
            lat.set_tuning(prec, "batch", block, 0, 4)

        def solve():
            for _, x, _, _ in fields:
                x.zero()
            st, infos = stag.cg_batched(fields, 1e-10, 2000)
            assert st == stag.OK, infos

        names = {n for n in launched(solve) if "batch_dslash" in n}
        form = "batch_dslash_split_kernel<" if split else "batch_dslash_lanes_kernel<"
        assert names and all(n.startswith("void " + form) for n in names), names
        if not split:
            assert all(f", {block}, " in n for n in names), names
        for (lat, x, _, m), (dims, U, N, b) in zip(fields, host):
            r = np.linalg.norm(b - oracle.apply_M(dims, U, N, m, x.export())) / np.linalg.norm(b)
            assert r <= 1.05e-10, (dims, m, block, r)
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("prec", ["df64", "f64"])
def test_tuner_times_the_form_with_block_sizes(prec):
    """65536 items per group of four: alone such a group would run in split form."""
    dims = (16, 16, 16, 8)
    with stag.Lattice(dims) as lat:
        lat.upload_gauge(synth.su3_field(dims, 0.3, 41).numpy(), None, precisions=(prec,))
        names = [n for n in launched(lambda: lat.autotune_all(prec, force=True)) if "batch_dslash" in n]
        assert names and all("batch_dslash_lanes_kernel<" in n for n in names), set(names)
        assert {b for b in (128, 256) for n in names if f", {b}, " in n} == {128, 256}
