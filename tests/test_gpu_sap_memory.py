"""SAP when device memory is short: without room for the face links or the
block-ordered vectors of a 4 x 4^3 or 8 x 4^3 block, or for the FP32 block image, the
application runs on the lexicographic vectors or fields; without room for the 16-bit
image it is refused as out of memory.  With room again it gives the usual bits.

The allocation that fails is picked by its size; at two right-hand sides the sizes
below are not those of another buffer allocated after the switch.

Bound: the same operator and the same copies of the fields in another order of the
sums: 6e-8 x sqrt(100 x 2 x 2 x 3) x a safety factor of 8 = 1e-5 per component."""
import ctypes

import pytest
import torch

from gpu_util import elem_err, record, to_dev, to_host
from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu

DIMS = (16, 8, 8, 8)
V = 16 * 8 ** 3


@pytest.mark.parametrize("block", [(4, 4, 4, 4), (8, 4, 4, 4)])
@pytest.mark.parametrize("half", [0, 1, 2])
@pytest.mark.parametrize("short,size", [("face links", 96), ("vectors", 2 * 2 * 96), ("image", 480)])
def test_sap_short_of_memory(block, half, short, size):
    from paper_1605_00564_gb300 import qcd
    lib = qcd.load_library()
    fail = lib.qcd_test_fail_alloc
    fail.argtypes, fail.restype = [ctypes.c_size_t], None
    U = synth.gauge_field(DIMS, 0.3, 101)
    eta = to_dev(synth.random_spinor(DIMS, 31, nrhs=2))

    def context(size, at_load=True):
        lat = qcd.Lattice(DIMS)
        fail(size * V if at_load else 0)
        lat.load_gauge(U, 1.4, 0.127, -1)
        fail(size * V)
        lat.set_params(block=block, ncy=2, nmr=3, sap_half=half)
        return lat

    want = context(0).apply_sap(eta).clone()
    half_image = half and block[0] == 4
    try:
        if short == "image" and half_image:
            lat = context(288, at_load=False)   # (the FP32 clover term has the same size)
            with pytest.raises(qcd.QcdError) as e:
                lat.apply_sap(eta)
            assert e.value.status == 3
        else:
            lat = context(size)
            got = lat.apply_sap(eta)
            # bf16 residuals are rounded anew after another order of the sums: 2^-9 in the
            # neighbours' terms, as the 16-bit copies
            tol = 5e-3 if half == 2 and block[0] == 4 else 1e-5
            e = elem_err(to_host(got), to_host(want))
            assert record("sap_short_%s_%d_h%d" % (short.replace(" ", "_"), block[0], half), e) < tol
    finally:
        fail(0)
    assert torch.equal(lat.apply_sap(eta), want)
