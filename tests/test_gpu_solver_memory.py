"""The tile of right-hand sides is chosen so that a solve's field-sized workspace fits
the free device memory: what a solve allocates is what the choice counts per right-hand
side, up to the small arrays (little vectors, partial sums, scalars: below 40 MB here,
a field of all right-hand sides is 151 MB)."""
import ctypes

import pytest
import torch

from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu

DIMS = (32, 16, 16, 16)


@pytest.mark.parametrize("dfl,half,prec", [(0, 0, "f32"), (0, 1, "f32"), (1, 0, "f32"), (1, 1, "f32"), (0, 0, "f64")])
def test_counted_workspace(dfl, half, prec):
    from paper_1605_00564_gb300 import qcd
    lib = qcd.load_library()
    lib.qcd_test_solver_bytes.restype, lib.qcd_test_solver_bytes.argtypes = ctypes.c_size_t, [ctypes.c_void_p]
    n, nkv = 12, 4
    lat = qcd.Lattice(DIMS)
    lat.load_gauge(torch.from_numpy(synth.unit_gauge(DIMS)).cuda(), 1.0, 0.11, -1)
    # max_outer = 1: every buffer is in use after one iteration
    lat.set_params(precision=prec, nkv=nkv, max_outer=1, rhs_tile=n, dfl=0, basis_half=half, sap_half=half)
    eta = torch.randn(lat.spinor_shape(n), dtype=torch.complex128, device="cuda")
    lat.apply_sap(eta[:1], precision=prec)   # the block image and kernels' own memory
    if dfl:
        lat.deflation_setup(eta[:4], 0)
        lat.set_params(dfl=1)
    psi0 = torch.zeros_like(eta)
    lat.apply_dirac(eta[:1], precision="f64")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    keep = torch.empty_like(eta), psi0      # solve()'s copy of psi0 takes the freed block
    del keep
    before = torch.cuda.mem_get_info()[0]
    lat.solve(eta, 1e-14, psi0=psi0, check=False)
    grown = before - torch.cuda.mem_get_info()[0]
    counted = n * lib.qcd_test_solver_bytes(lat._ctx)
    assert counted - 151e6 / 2 < grown < counted + 40e6, (grown, counted)
    lat.close()
