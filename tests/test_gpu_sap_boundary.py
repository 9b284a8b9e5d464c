"""The time boundary belongs to the gauge field: after a field with the other sign
has been loaded into a context with a stream of its own (whose SAP applications are
replayed from captured graphs), an application gives the bits of a fresh context."""
import pytest
import torch

from gpu_util import to_dev
from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu

DIMS = (8, 8, 8, 8)


@pytest.mark.parametrize("block,prec", [((4, 4, 4, 4), "f32"), ((4, 4, 4, 2), "f32"), ((4, 4, 4, 4), "f64")])
def test_boundary_sign_of_a_new_field(block, prec):
    from paper_1605_00564_gb300.qcd import Lattice
    U = synth.gauge_field(DIMS, 0.3, 97)
    eta = to_dev(synth.random_spinor(DIMS, 29, nrhs=2))

    def applied(*signs):
        lat = Lattice(DIMS, stream=torch.cuda.Stream())
        try:
            for bc in signs:
                lat.load_gauge(U, 1.4, 0.127, bc)
                lat.set_params(block=block, ncy=2, nmr=3)
                out = lat.apply_sap(eta, precision=prec).clone()
            torch.cuda.synchronize()
        finally:
            lat.close()
        return out

    anti, per = applied(-1), applied(1)
    assert not torch.equal(anti, per)
    assert torch.equal(applied(-1, 1), per)
    assert torch.equal(applied(1, -1, 1, -1), anti)
