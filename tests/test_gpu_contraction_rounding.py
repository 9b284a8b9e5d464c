"""The FP32 contraction's rounding error on random propagators, against its FP64 form
(whose own is nine digits smaller): rms over time-slices, projections and seeds, relative
to the rms correlator.

Rounding the three propagators of a term to FP32 alone gives sqrt(3) x 3.4e-8 = 6e-8.
The sum over the 36 colour permutations gave 9.4e-8; the bound is 1.12 times that (the
sampling error of 60 x 2 x 64 values is 1 %).  Chains of 32 products gave 1.18e-7."""
import numpy as np
import pytest
import torch

from gpu_util import record
from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(64, 8, 8, 8), (64, 6, 6, 6)])
def test_f32_rounding(dims):
    from paper_1605_00564_gb300.qcd import Lattice
    lat = Lattice(dims)
    lat.load_gauge(synth.unit_gauge(dims), 1.0, 0.12, -1)
    err = size = 0.0
    for seed in range(60):
        g = torch.Generator(device="cuda").manual_seed(seed)
        prop = torch.randn(lat.spinor_shape(12), dtype=torch.complex128, device="cuda", generator=g)
        c64, c32 = (lat.nucleon_2pt(prop, (0, 0, 0, 0), precision=p) for p in ("f64", "f32"))
        err += np.sum(np.abs(c32 - c64) ** 2)
        size += np.sum(np.abs(c64) ** 2)
    assert record("contract_f32_rounding_%d" % dims[1], float(np.sqrt(err / size))) < 1.05e-7
    lat.close()
