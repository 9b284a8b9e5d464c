"""Deflated preconditioner at the edges of its tiling: numbers of fields and
right-hand sides that fill the 4 x 3 output tiles only partly, more right-hand
sides than one little solve takes (24), a block of 32 sites, one of 512.

Sources D Phi e (the operator on a random combination of the block fields) are
solved by the low-mode part alone: projection, little solve and prolongation
give back Phi e up to the little solve's residual, which 32 steps on these 32 to
256 blocks bring below 1e-3 (bound of the existing little-solve test), and the
SAP correction only lowers the rest.  So one GCR iteration meets 1e-2, a decade
above; a wrong tile, chunk or field anywhere leaves a residual of order one there.
The iterate of a full solve meets 1e-10 in the oracle's operator (margin 1.1 as in
the other solve tests)."""
import numpy as np
import pytest

from gpu_util import make_lattice, to_dev, to_host
from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lattice():
    return make_lattice((16, 8, 8, 8), eps=0.3, csw=1.0, kappa=0.130, seed=160500564)


@pytest.mark.parametrize("block,ns,n", [((4, 4, 4, 4), 7, 1), ((4, 4, 4, 4), 12, 26), ((4, 2, 2, 2), 3, 5),
                                        ((8, 4, 4, 4), 9, 4)])
def test_deflated_solve_shapes(lattice, block, ns, n):
    lat, op, _ = lattice
    lat.set_params(block=block, ncy=5, nmr=4, nkv=16, precision="f32", sap_half=0, dfl=0, rhs_tile=n,
                   dfl_little_iters=16)
    from oracle.deflation import Deflation
    eta = synth.random_spinor(lat.dims, 21, nrhs=n)
    try:
        lat.deflation_setup(to_dev(synth.random_spinor(lat.dims, 22, nrhs=ns)), 3)
        d = Deflation(op, block)
        d.phi = to_host(lat.deflation_fields())
        lat.set_params(dfl=1, dfl_little_iters=32)
        v = np.random.default_rng(4).standard_normal((n, d.nb, ns)) * (1 + 0.5j)
        low = np.stack([op.D(d.prolong(e)) for e in v])
        _, st1 = lat.solve(to_dev(low), 1e-2)
        assert all(s["outer_iters"] == 1 for s in st1)
        psi, st = lat.solve(to_dev(eta), 1e-10)
        x = lat.deflation_little(v, 1, m=32)
        back = lat.deflation_little(x, 0)
    finally:
        lat.set_params(rhs_tile=0, dfl=0)
    psi = to_host(psi)
    for r in sorted({0, n // 2, n - 1}):
        res = np.linalg.norm(eta[r] - op.D(psi[r])) / np.linalg.norm(eta[r])
        assert st[r]["status"] == "QCD_OK" and res <= 1.1e-10, (r, res)
        assert np.linalg.norm(back[r] - v[r]) / np.linalg.norm(v[r]) < 1e-3
