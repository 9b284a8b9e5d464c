"""The sums of the Gram-Schmidt passes over sites of very different size.  Up to 155,648
sites a site's inner product is formed in FP32, and nothing of it is lost in the sum over
the sites (compensated pairs, then FP64).

A quarter of the sites (at random) holds components of size 1, the others of size 2^-13:
every product is a power of two and every site's sum exact in FP32, so the results are
those of 64 bits up to the rounding of the FP64 sums (below 1e-12; the bound is 1e-11).
FP32 sums over several sites lose the small ones beside a large one, 1e-8 of the
result."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(16, 8, 8, 8), (6, 10, 6, 14), (16, 16, 16, 16), (32, 16, 16, 16), (38, 16, 16, 16)])
@pytest.mark.parametrize("k,n", [(3, 1), (12, 2), (20, 1)])
def test_sums_of_uneven_sites(dims, k, n):
    from paper_1605_00564_gb300 import qcd
    lib = qcd.load_library()
    vp = ctypes.c_void_p
    lib.qcd_test_gs.argtypes = [vp, vp, vp, ctypes.c_int, ctypes.c_int, vp, vp, vp, vp, vp]
    lat = qcd.Lattice(dims)
    V = int(np.prod(dims))
    g = torch.Generator(device="cuda").manual_seed(V + k)

    def field(*lead):
        """Signs times the site's size, [.., 6, V, 4] FP32."""
        sign = torch.randint(0, 2, (*lead, 6, V, 4), generator=g, device="cuda") * 2 - 1
        return sign.float() * size[:, None]

    size = torch.where(torch.rand(V, generator=g, device="cuda") < 0.25, 1.0, 2.0 ** -13)
    chi, rho = field(k + 1, n), field(n)
    # mostly of one sign, so that the sums do not cancel
    chi, rho = torch.where(torch.rand_like(chi) < 0.9, chi.abs(), chi), torch.where(torch.rand_like(rho) < 0.9, rho.abs(), rho)

    def dot(a, b):      # (a, b) per right-hand side
        a, b = a.double(), b.double()
        ar, ai, br, bi = a[..., 0::2], a[..., 1::2], b[..., 0::2], b[..., 1::2]
        s = lambda x: x.sum((-3, -2, -1))  # noqa: E731
        return torch.stack([s(ar * br + ai * bi), s(ar * bi - ai * br)], -1)

    want_dots, want_n2 = torch.stack([dot(chi[j], chi[k]) for j in range(k)]), dot(chi[k], chi[k])
    want_c, want_rn2 = dot(chi[k], rho), dot(rho, rho)
    f64 = dict(dtype=torch.float64, device="cuda")
    inv, ck = torch.ones(n, **f64), torch.zeros(n, 2, **f64)
    dots, n2c, rn2 = torch.zeros(k, n, 2, **f64), torch.zeros(2, n, 2, **f64), torch.zeros(n, 2, **f64)
    torch.cuda.synchronize()
    p = lambda t: t.data_ptr()  # noqa: E731
    assert lib.qcd_test_gs(lat._ctx, p(chi), p(rho), k, n, p(inv), p(ck), p(dots), p(n2c), p(rn2)) == 0
    scale = want_n2[:, :1]
    for got, want in ((dots, want_dots), (n2c[0, :, :1], want_n2[:, :1]), (n2c[1], want_c), (rn2[:, :1], want_rn2[:, :1])):
        assert float(((got - want).abs() / scale).max()) < 1e-11
    lat.close()
