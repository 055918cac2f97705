"""The rules that choose between forms of one kernel: which form runs, on both
sides of each line, and that the forms agree."""
import numpy as np
import pytest
from kernel_trace import launched

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
