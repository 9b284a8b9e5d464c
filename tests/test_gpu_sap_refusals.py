"""Lattices that no default block shape fits: a SAP application or a solve with the
default parameters is refused with an argument error before any launch (the
checkerboard of blocks would leave the lattice), while what needs no blocks works."""
import pytest
import torch

from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(6, 6, 6, 6), (5, 4, 4, 4), (8, 8, 2, 8)])
@pytest.mark.parametrize("prec", ["f32", "f64"])
def test_default_blocks_that_do_not_fit(dims, prec):
    from paper_1605_00564_gb300.qcd import Lattice, QcdError
    lat = Lattice(dims)
    lat.load_gauge(synth.unit_gauge(dims), 1.0, 0.12, -1)
    eta = torch.ones(lat.spinor_shape(1), dtype=torch.complex128, device="cuda")
    with pytest.raises(QcdError) as e:
        lat.apply_sap(eta, precision=prec)
    assert e.value.status == 1
    with pytest.raises(QcdError) as e:
        lat.solve(eta, 1e-3)
    assert e.value.status == 1
    # the free field on a constant vector: D = 1 - 8 kappa in the bulk
    out = lat.apply_dirac(eta, precision=prec)
    assert torch.allclose(out[:, 1:-1], (1 - 8 * 0.12) * eta[:, 1:-1], atol=1e-5)
    lat.close()
