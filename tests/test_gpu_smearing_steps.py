"""Gaussian smearing with an odd and an even number of steps (after an odd number the
result is copied back from the scratch field): of whole fields, and of a source that is
smeared on its own time-slice only.

Bounds: as for the even counts, 1e-13 element-wise for the FP64 stencil, 1e-10 per
time-slice for correlators from exact (1e-12) solves."""
import numpy as np
import pytest

from gpu_util import elem_err, record, to_dev, to_host
from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu

DIMS = (8, 4, 4, 4)
ALPHA, N_APE, KAPPA_G = 0.5, 2, 0.25


@pytest.fixture(scope="module")
def setup():
    from oracle import smearing
    from oracle.dirac import Operator
    from paper_1605_00564_gb300.qcd import Lattice
    U = synth.gauge_field(DIMS, 0.4, 3141)
    lat = Lattice(DIMS)
    lat.load_gauge(U, 1.3, 0.12, -1)
    lat.set_params(block=(4, 2, 2, 2), ncy=5, nmr=4, nkv=16, precision="f32", dfl=0)
    lat.smear_links(ALPHA, N_APE)
    yield lat, Operator(U, 0.12, 1.3, -1), smearing.ape_smear(U, ALPHA, N_APE)
    lat.close()


@pytest.mark.parametrize("steps", [1, 2, 3])
def test_field(setup, steps):
    from oracle import smearing
    lat, _, Uape = setup
    lat.set_smearing(KAPPA_G, steps)
    psi = synth.random_spinor(DIMS, 5, nrhs=2)
    try:
        out = to_host(lat.smear_gaussian(to_dev(psi)))
    finally:
        lat.set_smearing(0.0, 0)
    ref = np.stack([smearing.gaussian_smear(Uape, p, KAPPA_G, steps) for p in psi])
    assert record("gaussian_smear_%d" % steps, elem_err(out, ref)) < 1e-13


@pytest.mark.parametrize("steps,src,direction", [(3, (4, 2, 0, 2), 1), (2, (0, 0, 2, 2), -1), (1, (4, 0, 0, 0), -1)])
def test_source_and_sink(setup, steps, src, direction):
    from oracle import smearing, threept
    lat, op, Uape = setup
    t_sep = 3
    lat.set_smearing(KAPPA_G, steps)
    try:
        r = lat.ama_nucleon([src], 1, sloppy_tol=1e-3, exact_tol=1e-12, t_sep=t_sep, direction=direction)
    finally:
        lat.set_smearing(0.0, 0)
    K = smearing.timeslice_matrices(Uape, KAPPA_G, steps)
    ref3, ref2 = threept.three_point(op, src, t_sep, direction, a2a=threept.AllToAll(op), smear=(K,))
    c3, c2 = r["c3_all"][1], r["c2_all"][1]                      # the exact position
    for k, name in enumerate(("A3", "S", "T12")):
        floor = np.sqrt(np.mean(np.abs(ref3[k]) ** 2))
        e = float(np.max(np.abs(c3[k] - ref3[k]) / np.maximum(np.abs(ref3[k]), floor)))
        assert record("smeared_3pt_%s_n%d" % (name, steps), e) < 1e-10, (name, e)
    got2 = c2[0 if direction > 0 else 1, (direction * t_sep) % DIMS[0]]
    assert record("smeared_2pt_n%d" % steps, abs(got2 - ref2) / abs(ref2)) < 1e-10
