"""Device links that start on an 8-byte, not a 16-byte boundary (any double
array may): gauge upload, three-link products and the net take them and give
the bits that the same links give on a 16-byte boundary."""
import ctypes

import numpy as np
import pytest

from paper_1411_2087_gb300 import stag, synth

pytestmark = pytest.mark.gpu

DIMS = (6, 4, 6, 10)
V = int(np.prod(DIMS))


def on_device(a, off):
    """(pointer, tensor): the doubles of `a` on the device, `off` doubles past a 16-byte boundary."""
    import torch
    flat = torch.from_numpy(np.ascontiguousarray(a).view(np.float64).reshape(-1))
    buf = torch.zeros(flat.numel() + 2, dtype=torch.float64, device="cuda")
    buf[off:off + flat.numel()] = flat.to("cuda")
    torch.cuda.synchronize()
    p = buf.data_ptr() + 8 * off
    assert p % 16 == 8 * off
    return ctypes.c_void_p(p), buf


@pytest.mark.parametrize("offs", [(1, 1), (1, 0), (0, 1), (1, None)])
@pytest.mark.parametrize("mask", [0, 1 << stag.PREC["f32"] | stag.COMPRESS12])
def test_upload(offs, mask):
    U = synth.su3_field(DIMS, 0.3, 81).numpy()
    with stag.Lattice(DIMS) as lat:
        N = np.empty_like(U)
        lat.long_links(U, N)
        prec = "f32" if mask else "df64"
        fe = lat.field(stag.EVEN, prec, synth.gaussian_colour_field(V // 2, 82).numpy())
        out = lat.field(stag.ODD, prec)

        def dslash(fat_off, lng_off):
            pf, keep_f = on_device(U, fat_off)
            pl, keep_l = on_device(N, lng_off) if lng_off is not None else (None, None)
            assert stag.lib().stag_gauge_upload(lat.handle, pf, pl, 1.125, -1 / 24, stag.PTR_DEVICE, mask) == stag.OK
            lat.dslash(out, fe)
            return out.export()

        want = dslash(0, 0 if offs[1] is not None else None)
        assert np.array_equal(dslash(*offs), want)


@pytest.mark.parametrize("fat_off,out_off", [(1, 0), (0, 1), (1, 1)])
def test_long_links(fat_off, out_off):
    import torch
    U = synth.su3_field(DIMS, 0.3, 83).numpy()
    with stag.Lattice(DIMS) as lat:
        want = lat.long_links(U)
        pf, keep_f = on_device(U, fat_off)
        po, buf = on_device(np.zeros_like(U), out_off)
        edge = buf.clone()
        assert stag.lib().stag_long_links_build(lat.handle, pf, po, stag.PTR_DEVICE) == stag.OK
        torch.cuda.synchronize()
        n = U.size * 2
        got = buf[out_off:out_off + n].cpu().numpy().view(np.complex128).reshape(U.shape)
        assert np.array_equal(got, want)
        assert torch.equal(buf[:out_off], edge[:out_off]) and torch.equal(buf[out_off + n:], edge[out_off + n:])


def test_net():
    U = synth.su3_field(DIMS, 0.3, 84).numpy()
    with stag.Lattice(DIMS) as lat:
        lat.upload_gauge(U, None, precisions=("df64",))
        src = lat.field(stag.EVEN, "df64", synth.gaussian_colour_field(V // 2, 85).numpy())
        res = []
        for off in (0, 1):
            pf, keep = on_device(U, off)
            h = ctypes.c_void_p()
            assert stag.lib().stag_net_create(lat.handle, pf, stag.PTR_DEVICE, 8, 5, ctypes.byref(h)) == stag.OK
            for flags in (0, 7):  # nine-entry FP32 links; 12-real 16-bit links
                out = lat.field(stag.EVEN, "df64")
                assert stag.lib().stag_net_apply(h, out.handle, src.handle, flags) == stag.OK
                res.append(out.export())
            stag.lib().stag_net_destroy(h)
        assert np.array_equal(res[0], res[2]) and np.array_equal(res[1], res[3])
