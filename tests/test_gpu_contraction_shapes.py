"""The diquark form of the nucleon contraction on lattices whose spatial volume
fills a CTA's sites only partly (largest power of two dividing it: 1, 2, 8, 32),
in both precisions, against the oracle's enumeration of the Wick contractions.

Bounds: a site sums about 1000 products; rounding grows like the square root,
sqrt(1000) x 1.1e-16 = 3.5e-15 (FP64) and 1.9e-6 (FP32) of a typical term, the
sum over a time-slice adds and averages them alike, and |C(t)| of random
propagators is a few times a term: 1e-13 and 5e-6 leave a factor of 3."""
import numpy as np
import pytest

from gpu_util import record, timeslice_err, to_dev
from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(3, 3, 5, 7), (4, 6, 5, 3), (2, 4, 6, 5), (3, 8, 4, 6)])
@pytest.mark.parametrize("prec,tol", [("f64", 1e-13), ("f32", 5e-6)])
def test_contraction_ragged(dims, prec, tol):
    import torch
    from oracle import nucleon
    from paper_1605_00564_gb300.qcd import Lattice, nucleon_2pt_noalloc
    lat = Lattice(dims)
    lat.load_gauge(synth.unit_gauge(dims), 1.0, 0.12, -1)
    prop = np.random.default_rng(8).standard_normal(lat.spinor_shape(12) + (2,)) @ np.array([1, 1j])
    src = (1, 0, 1, 2)
    ref = nucleon.two_point(prop, src[0])
    out = lat.nucleon_2pt(to_dev(prop), src, precision=prec)
    assert record("contract_ragged_%s_%s" % (prec, "x".join(map(str, dims))), timeslice_err(out, ref)) <= tol
    corr = torch.zeros(2 * dims[0] * 2, dtype=torch.float64, device="cuda")
    nucleon_2pt_noalloc(dims, to_dev(prop), src, corr, precision=prec)
    na = corr.cpu().numpy().reshape(2, dims[0], 2)
    assert timeslice_err(na[..., 0] + 1j * na[..., 1], ref) <= tol
    lat.close()
