"""Device memory that a context holds, per site: the gauge field and clover term in
FP64 and FP32 (576 + 192 + 576 + 288 bytes) after loading a field; with parameters set,
also the one block image that they use (FP32 480, 16-bit 288) and the face links of
4 x 4^3 blocks (96), whatever was set before.  An image is 38 or 63 MB here, the face
links 13 MB; the bounds leave 4 MB for the granularity of the allocations."""
import pytest
import torch

from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu

DIMS = (32, 16, 16, 16)
FIELDS = 576 + 192 + 576 + 288


def held(steps):
    """Bytes per site that a new context holds after load_gauge and the parameter sets of steps."""
    from paper_1605_00564_gb300.qcd import Lattice
    U = torch.from_numpy(synth.unit_gauge(DIMS)).cuda()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    lat = Lattice(DIMS)
    for s in steps:
        if s == "load":
            lat.load_gauge(U, 1.0, 0.12, -1)
        else:
            lat.set_params(**s)
    n = before - torch.cuda.mem_get_info()[0]
    lat.close()
    return n / (32 * 16 ** 3)


@pytest.mark.parametrize("steps,per_site", [
    (["load"], FIELDS),
    (["load", dict(sap_half=1)], FIELDS + 288 + 96),
    ([dict(sap_half=1), "load"], FIELDS + 288 + 96),
    (["load", dict(sap_half=0), dict(sap_half=1)], FIELDS + 288 + 96),
    ([dict(sap_half=1), "load", dict(sap_half=0)], FIELDS + 480 + 96),
    (["load", dict(sap_half=1), dict(block=(4, 4, 4, 2))], FIELDS + 288),
    (["load", dict(sap_half=0), dict(precision="f64")], FIELDS),
    (["load", dict(block=(8, 8, 4, 4))], FIELDS),     # more than 512 sites: no image
])
def test_memory_held(steps, per_site):
    held(["load"])     # the kernels' own memory
    assert abs(held(steps) - per_site) < 4e6 / (32 * 16 ** 3), held(steps)
