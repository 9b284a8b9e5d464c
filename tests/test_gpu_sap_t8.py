"""SAP on 8 x 4^3 blocks: the boundary terms and block-ordered vectors share their
kernels with the 4^4 blocks, but the faces differ in size and the links across them
are kept for one block shape at a time.

Bounds: against the oracle as for the 4^4 block in FP32 (n_cy x 2 x n_mr block
operators of about 100 terms: 6e-8 x sqrt(100 x 3 x 2 x 3) x a safety factor of 8 =
2e-5 per component); a change of the block shape and back gives the same bits."""
import numpy as np
import pytest
import torch

from gpu_util import elem_err, elem_err_faces, make_lattice, record, to_dev, to_host
from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,n", [((16, 8, 8, 8), 1), ((48, 8, 16, 8), 5), ((32, 16, 8, 24), 13)])
def test_sap_8x4x4x4(dims, n):
    from oracle.sap import SAP
    lat, op, _ = make_lattice(dims, eps=0.3, csw=1.4, kappa=0.127, seed=83)
    eta = synth.random_spinor(lat.dims, 19, nrhs=n)
    dev = to_dev(eta)
    lat.set_params(block=(4, 4, 4, 4), ncy=3, nmr=3, sap_half=0)
    before = lat.apply_sap(dev, precision="f32").clone()
    lat.set_params(block=(8, 4, 4, 4), ncy=3, nmr=3, sap_half=0)
    out = to_host(lat.apply_sap(dev, precision="f32"))
    lat.set_params(block=(4, 4, 4, 4), ncy=3, nmr=3, sap_half=0)
    assert torch.equal(before, lat.apply_sap(dev, precision="f32"))
    s = SAP(op, (8, 4, 4, 4), ncy=3, nmr=3)
    pick = sorted({0, n - 1})
    ref = np.stack([s.apply(eta[r]) for r in pick])
    name = "sap_t8_%s_n%d" % ("x".join(map(str, dims)), n)
    assert record(name, elem_err(out[pick], ref)) < 2e-5
    assert record(name + "_faces", elem_err_faces(out[pick], ref, lat.dims, (8, 4, 4, 4))) < 2e-5
