"""Import and export of spinors through shared memory, 64 sites per CTA: volumes
below, at and just above multiples of 64, odd counts of right-hand sides.  The
operator with kappa = 0 and c_sw = 0 is the identity, so FP64 returns the input's
bits and FP32 its rounding to single precision."""
import numpy as np
import pytest

from gpu_util import to_dev, to_host
from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (2, 3, 3, 3), (4, 4, 2, 2), (5, 13, 2, 3), (4, 8, 8, 8)])
@pytest.mark.parametrize("n", [1, 5])
def test_layout_identity(dims, n):
    from paper_1605_00564_gb300.qcd import Lattice
    lat = Lattice(dims)
    lat.load_gauge(synth.unit_gauge(dims), 0.0, 0.0, -1)
    psi = synth.random_spinor(dims, 41, nrhs=n)
    assert np.array_equal(to_host(lat.apply_dirac(to_dev(psi), precision="f64")), psi)
    out = to_host(lat.apply_dirac(to_dev(psi), precision="f32"))
    assert np.array_equal(out, psi.astype(np.complex64).astype(np.complex128))
    lat.close()
