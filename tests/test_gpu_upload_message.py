"""A refused 12-real upload names the deviation of both fields from SU(3), also
that of a field which would have passed."""
import numpy as np
import pytest

from paper_1411_2087_gb300 import stag, synth

pytestmark = pytest.mark.gpu


def stretched(U, dev):
    """One row's squared length off by dev (the determinant by half as much)."""
    V = U.copy()
    V[1, 33, 2] *= np.sqrt(1.0 + dev)
    return V


@pytest.mark.parametrize("fat,lng", [(3e-7, 2e-3), (2e-3, 3e-7), (4e-6, 9e-7)])
def test_both_deviations_in_the_message(fat, lng):
    dims = (4, 4, 4, 4)
    U, N = synth.su3_field(dims, 0.3, 51).numpy(), synth.su3_field(dims, 0.3, 52).numpy()
    with stag.Lattice(dims) as lat:
        with pytest.raises(stag.StagError) as e:
            lat.upload_gauge(stretched(U, fat), stretched(N, lng), precisions=("f32",), compress12=True)
    assert f"{fat:.2e} (fat) / {lng:.2e} (long)" in str(e.value)
