"""What a new lattice allocates on the device: one buffer per copy of the links
and per field, and no scratch of its own for an upload, an import or a solve's
check of its source."""
import numpy as np
import pytest
from kernel_trace import traced

from paper_1411_2087_gb300 import stag, synth

pytestmark = pytest.mark.gpu


def test_upload_and_import_allocate_the_copies_only():
    import torch
    dims = (6, 4, 6, 10)
    U = synth.su3_field(dims, 0.3, 11).to("cuda")
    psi = synth.gaussian_colour_field(int(np.prod(dims)) // 2, 12).to("cuda")
    N = torch.empty_like(U)
    lats = []

    def upload():
        lat = stag.Lattice(dims)  # one buffer of partial sums, one of scalars
        lats.append(lat)
        lat.long_links(U, N)
        lat.upload_gauge(U, N, precisions=("df64", "f32"))

    names = traced(upload)
    assert names.count("cudaMalloc") == 4, names

    def again():
        for lat in lats[-1:]:
            f = lat.field(stag.EVEN, "df64")
            f.import_(psi)

    assert traced(again).count("cudaMalloc") == 1
    for lat in lats:
        lat.close()
