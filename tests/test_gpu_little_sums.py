"""The dots of the little GCR over blocks of very different size: a few products are
summed in FP32, the sums of a thread over its blocks (seven here) are not.

(q_j, q) with q_j equal to q on an eighth of the blocks (at random) and 2^-23 of it on the
others.  The bound: 16 roundings of 6e-8 in each of the at least 500 FP32 sums of the
large blocks, adding up like a random walk, 6e-8 x 4 / sqrt(500) x a safety factor of 3 =
3e-8 of the result; an FP32 sum over the blocks of a thread loses the small ones behind a
large one, several 1e-7."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DIMS, BLOCK = (32, 16, 16, 16), (4, 2, 2, 2)
NBLK = 8 ** 4


@pytest.mark.parametrize("ns,n,nj", [(20, 3, 5), (7, 2, 24), (32, 24, 3), (1, 1, 1)])
def test_dots_over_uneven_blocks(ns, n, nj):
    from paper_1605_00564_gb300 import qcd, synth
    lib = qcd.load_library()
    vp = ctypes.c_void_p
    lib.qcd_test_little_dots.argtypes = [vp, vp, vp, ctypes.c_int, ctypes.c_int, vp, vp]
    lat = qcd.Lattice(DIMS)
    lat.load_gauge(torch.from_numpy(synth.unit_gauge(DIMS)).cuda(), 1.0, 0.11, -1)
    lat.set_params(block=BLOCK, dfl=0)
    g = torch.Generator(device="cuda").manual_seed(ns)
    lat.deflation_setup(torch.randn(lat.spinor_shape(ns), dtype=torch.complex128, device="cuda", generator=g), 0)
    p = torch.randn((n, NBLK, ns, 2), device="cuda", generator=g)
    q, dots = torch.zeros_like(p), torch.zeros((nj, n, 2), dtype=torch.float64, device="cuda")
    w = torch.where(torch.rand((nj, 1, NBLK, 1, 1), device="cuda", generator=g) < 0.125, 1.0, 2.0 ** -23)

    def run(qj):
        torch.cuda.synchronize()
        ptr = [vp(t.data_ptr()) for t in (p, qj, q, dots)]
        assert lib.qcd_test_little_dots(lat._ctx, ptr[0], ptr[1], nj, n, ptr[2], ptr[3]) == 0

    run(torch.zeros((nj, *p.shape), device="cuda"))
    ref = lat.deflation_little((p[..., 0] + 1j * p[..., 1]).cpu().numpy(), 0)    # the FP64 matrix
    got = (q[..., 0] + 1j * q[..., 1]).cpu().numpy()
    assert np.linalg.norm(got - ref) < 1e-6 * np.linalg.norm(ref)
    qj = (w * q).contiguous()
    run(qj)
    a, b = qj.double(), q.double()
    s = lambda x: x.sum((-2, -1))  # noqa: E731
    want = torch.stack([s(a[..., 0] * b[..., 0] + a[..., 1] * b[..., 1]),
                        s(a[..., 0] * b[..., 1] - a[..., 1] * b[..., 0])], -1)
    assert float(((dots - want).abs() / want[..., :1]).max()) < 3e-8
    lat.close()
