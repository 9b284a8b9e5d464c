"""The two-lane FP32 SAP sweep at the edges of its dispatch, against the oracle:
the smallest block (32 sites, one warp per CTA), a block between the staged
sizes, the largest (1024 sites, links and clover term read from global memory),
one and thirteen right-hand sides, odd n_mr.

Bounds (element-wise, gpu_util.elem_err): a component passes n_cy x 2 x n_mr
block operators of about 100 FP32 terms each (6e-8 relative per term, adding up
like a random walk): 6e-8 x sqrt(100 x 2 x 2 x 3) x a safety factor of 8 = 1e-5;
with 16-bit copies of links and clover term their rounding (4.9e-4 relative)
takes its place, 5e-3 (as the parity test of the 4^4 block)."""
import numpy as np
import pytest

from gpu_util import elem_err, elem_err_faces, make_lattice, record, to_dev, to_host
from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lattice():
    return make_lattice((16, 16, 8, 8), eps=0.3, csw=1.4, kappa=0.127, seed=79)


@pytest.mark.parametrize("block,n,nmr", [((4, 2, 2, 2), 1, 3), ((4, 4, 4, 4), 13, 3), ((2, 8, 4, 2), 3, 4),
                                         ((8, 4, 4, 4), 1, 3), ((8, 8, 4, 4), 3, 4)])
@pytest.mark.parametrize("half,tol", [(0, 1e-5), (1, 5e-3)])
def test_sap_block_shapes(lattice, block, n, nmr, half, tol):
    from oracle.sap import SAP
    lat, op, _ = lattice
    lat.set_params(block=block, ncy=2, nmr=nmr, sap_half=half)
    eta = synth.random_spinor(lat.dims, 17, nrhs=n)
    out = to_host(lat.apply_sap(to_dev(eta), precision="f32"))
    s = SAP(op, block, ncy=2, nmr=nmr)
    pick = sorted({0, n // 2, n - 1})
    ref = np.stack([s.apply(eta[r]) for r in pick])
    name = "sap_pair_h%d_%s_n%d" % (half, "x".join(map(str, block)), n)
    assert record(name, elem_err(out[pick], ref)) < tol
    assert record(name + "_faces", elem_err_faces(out[pick], ref, lat.dims, block)) < tol
