"""The operator writing the caller's layout itself, at the edges of its runs: volumes
that are no multiple of a run (64 or 128 sites), on both sides of the volume where the
FP64 operator changes its form, and right-hand sides in pairs and alone.

Bounds (element-wise): a component sums about 200 products, so 200^1/2 x 1.1e-16 x a
safety factor of 60 = 1e-13 in FP64 and 200^1/2 x 6e-8 x 6 = 5e-6 in FP32 (the bounds of
the parity tests); a right-hand side gives the same bits alone and in any batch."""
import numpy as np
import pytest
import torch

from gpu_util import elem_err, make_lattice, record, to_dev, to_host
from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 6, 6, 6), (10, 10, 10, 10), (6, 32, 8, 8)])
@pytest.mark.parametrize("prec,tol", [("f64", 1e-13), ("f32", 5e-6)])
def test_dirac_caller_layout(dims, prec, tol):
    lat, op, _ = make_lattice(dims, eps=0.3, csw=1.3, kappa=0.127, seed=91)
    psi = synth.random_spinor(lat.dims, 23, nrhs=5)
    dev = to_dev(psi)
    for dagger in (False, True):
        ref = np.stack([op.D(p, dagger=dagger) for p in psi])
        out = lat.apply_dirac(dev, dagger=dagger, precision=prec)
        name = "dirac_layout_%s_%s_%d" % (prec, "x".join(map(str, dims)), dagger)
        assert record(name, elem_err(to_host(out), ref)) < tol
        for n in (1, 2):
            part = lat.apply_dirac(dev[:n].contiguous(), dagger=dagger, precision=prec)
            assert torch.equal(part, out[:n])
