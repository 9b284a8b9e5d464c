"""The FP64 4^4 sweep (a block on a cluster of two CTAs): sums run over fixed groups of
sites in a fixed order, so a right-hand side gives the same bits alone and in a
batch of 24, for one and several cycles and MR steps."""
import numpy as np
import pytest

from gpu_util import make_lattice, to_dev, to_host
from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ncy,nmr", [(1, 1), (2, 4), (3, 3)])
def test_sap_f64_batched_equals_single(ncy, nmr):
    lat, _, _ = make_lattice((8, 16, 16, 16), eps=0.3, csw=1.2, kappa=0.126, seed=80)
    lat.set_params(block=(4, 4, 4, 4), ncy=ncy, nmr=nmr, precision="f64")
    eta = synth.random_spinor(lat.dims, 31, nrhs=24)
    many = to_host(lat.apply_sap(to_dev(eta), precision="f64"))
    for r in (0, 23):
        one = to_host(lat.apply_sap(to_dev(eta[r:r + 1]), precision="f64"))[0]
        assert np.array_equal(one, many[r])
    lat.close()
