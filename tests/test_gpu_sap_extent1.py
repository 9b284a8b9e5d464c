"""SAP on blocks with an extent of 1: every site lies on both faces of such a
direction, so its boundary term has two hops, one from either neighbouring block.

Bounds (element-wise) as for the other block shapes: n_cy x 2 x n_mr block operators
of about 100 FP32 terms each, 6e-8 x sqrt(100 x 2 x 2 x 3) x a safety factor of 8 =
1e-5, with 16-bit copies of links and clover term 5e-3; FP64 1e-13.  (A missing hop is
an error of order kappa.)"""
import numpy as np
import pytest

from gpu_util import elem_err, make_lattice, record, to_dev, to_host
from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lattice():
    return make_lattice((8, 8, 8, 8), eps=0.3, csw=1.4, kappa=0.127, seed=89)


@pytest.mark.parametrize("block", [(1, 4, 4, 4), (4, 1, 4, 2), (2, 4, 4, 1), (4, 1, 2, 4), (1, 4, 2, 4)])
@pytest.mark.parametrize("prec,half,tol", [("f32", 0, 1e-5), ("f32", 1, 5e-3), ("f64", 0, 1e-13)])
def test_sap_extent_1(lattice, block, prec, half, tol):
    from oracle.sap import SAP
    lat, op, _ = lattice
    lat.set_params(block=block, ncy=2, nmr=3, sap_half=half)
    eta = synth.random_spinor(lat.dims, 23, nrhs=2)
    out = to_host(lat.apply_sap(to_dev(eta), precision=prec))
    s = SAP(op, block, ncy=2, nmr=3)
    ref = np.stack([s.apply(e) for e in eta])
    name = "sap_extent1_%s_h%d_%s" % (prec, half, "x".join(map(str, block)))
    assert record(name, elem_err(out, ref)) < tol
