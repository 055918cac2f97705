"""stag_apply_M_noalloc refuses buffers off a 16-byte boundary before any CUDA
call (it reads complex numbers whole and allocates nothing to copy them to)."""
import ctypes

import pytest

from paper_1411_2087_gb300 import build, stag


@pytest.mark.parametrize("which", range(4))
def test_misaligned_buffer_refused(which):
    build.build()
    L = stag.lib()
    ptrs = [0x1000, 0x2000, 0x3000, 0x4000]  # never dereferenced: the checks fail first
    ptrs[which] += 8
    fat, lng, i, o = (ctypes.c_void_p(p) for p in ptrs)
    st = L.stag_apply_M_noalloc((ctypes.c_int * 4)(4, 4, 4, 4), None, 1.125, -1 / 24, fat, lng, 0.1, i, o, None)
    assert st == stag.ERR_ARG
    assert b"16-byte" in L.stag_last_error_message()
