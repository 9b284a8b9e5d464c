"""The work a user of the library has it do, as cases that can be timed: the
operator, the SAP preconditioner, solves at both tolerances, the deflated
solve, the nucleon contraction, smearing, the differentiable correlator and a
whole all-mode-averaging call, each through the public binding
(paper_1605_00564_gb300.qcd) and from the smallest lattice of the repository's
configurations to its production size.

A case is a dict of plain values; ``kind`` says which entry point it runs.
``exact`` recomputes the outputs with plain torch in 64 bits from the
definitions, without the library.

Results of the FP32 paths (FP32 operator, FP32 preconditioner, solves to a
sloppy tolerance, correlators of those) come back in complex64, the precision
their caller asked for and keeps them in; everything FP64 stays complex128.
"""
import itertools
import math

import numpy as np
import torch

from paper_1605_00564_gb300 import qcd

SMEAR = {"alpha": 0.5, "n_ape": 3, "kappa_g": 0.25}


def _dims(c):
    return c["T"], c["X"], c["Y"], c["Z"]


def _case(name, kind, dims, n, **kw):
    c = {"kind": kind, "T": dims[0], "X": dims[1], "Y": dims[2], "Z": dims[3], "n": n}
    c.update({"eps": 0.15, "csw": 1.9, "kappa": 0.13})
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one FP64 operator application on the 8^3x16 lattice
        # (launches and the final synchronisation are all of it)
        _case("dirac_f64_8c16_n1", "dirac", (16, 8, 8, 8), 1, prec="f64", dagger=False, eps=0.3, csw=1.0),
        # the FP32 operator on the 12 spin-colour components at production size
        _case("dirac_f32_32c64_n12", "dirac", (64, 32, 32, 32), 12, prec="f32", dagger=False),
        # the FP64 adjoint operator on a few vectors of the second lattice (residual checks, gamma_5 tests)
        _case("dirac_f64_dag_24c48_n4", "dirac", (48, 24, 24, 24), 4, prec="f64", dagger=True),
        # the preconditioner as the production solves run it: 16-bit block copies, 12 RHS, 32^3x64
        _case("sap_half_32c64_n12", "sap", (64, 32, 32, 32), 12, prec="f32", block="4,4,4,4", ncy=5, nmr=4, half=1),
        # the other block shape of the production comparison (8x4^3), FP32 copies, a lattice of
        # unequal extents and an odd number of right-hand sides
        _case("sap_8x444_48x24x8x16_n5", "sap", (48, 24, 8, 16), 5, prec="f32", block="8,4,4,4", ncy=4, nmr=4, half=0),
        # the plain method on the small lattice: everything in FP64, 1e-10
        _case("solve_f64_8c16_n12", "solve", (16, 8, 8, 8), 12, prec="f64", tol=1e-10, half=0, source="point", eps=0.3,
              csw=1.0),
        # one sloppy tile of the AMA batch: 12 components of a point source at 1e-3
        _case("solve_sloppy_24c48_n12", "solve", (48, 24, 24, 24), 12, prec="f32", tol=1e-3, half=1, source="point"),
        # a single exact mixed-precision solve with the default FP32 block copies
        _case("solve_exact_24c48_n1", "solve", (48, 24, 24, 24), 1, prec="f32", tol=1e-12, half=0, source="random"),
        # the locally deflated solver on the 12 components, where deflation pays (kappa 0.126)
        _case("deflated_16c32_n12", "deflated", (32, 16, 16, 16), 12, tol=1e-12, half=1, ns=20, rounds=3, little=24,
              kappa=0.126),
        # the nucleon two-point contraction of one propagator in FP64 (every exact solve ends in one)
        _case("nucleon_f64_24c48", "nucleon", (48, 24, 24, 24), 12, prec="f64"),
        # the differentiable correlator: forward solves and contraction, adjoint solves for both gradients
        _case("fh_gradient_16c32", "fh", (32, 16, 16, 16), 12, m0=0.2, csw=1.3, eps=0.3, kappa=1.0 / 8.4),
        # a whole AMA measurement: smeared two- and three-point functions of two positions,
        # fixed-iteration sloppy solves, one position exact
        _case("ama_16c32", "ama", (32, 16, 16, 16), 2, kappa=0.126, n_iter_2pt=6, n_iter_3pt=8, t_sep=8, direction=1,
              half=1, n_gauss=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["dirac", "dirac", "sap", "sap", "sap", "solve", "solve", "deflated", "nucleon", "smear", "fh", "ama"])
    if kind in ("dirac", "nucleon", "smear"):
        # any extents, odd ones among them, from a few thousand sites to production size
        while True:
            dims = (_log_int(rng, 4, 64),) + tuple(_log_int(rng, 4, 32) for _ in range(3))
            n = 12 if kind == "nucleon" else _log_int(rng, 1, 12)
            V = math.prod(dims)
            if 2000 <= V and V * n <= 8_000_000:
                break
        if kind == "smear":
            return _case(None, kind, dims, n, n_gauss=_log_int(rng, 2, 20))
        prec = rng.choice(["f32", "f64"])
        if kind == "nucleon":
            return _case(None, kind, dims, n, prec=prec)
        return _case(None, kind, dims, n, prec=prec, dagger=rng.random() < 0.3, kappa=round(rng.uniform(0.12, 0.136), 4))
    if kind == "sap":
        block = rng.choice([(4, 4, 4, 4), (4, 4, 4, 4), (4, 4, 4, 4), (8, 4, 4, 4), (4, 2, 4, 2), (4, 4, 4, 2)])
        prec = rng.choice(["f32", "f32", "f32", "f64"])
        while True:
            dims = tuple(2 * b * rng.randint(1, (64 if k == 0 else 32) // (2 * b)) for k, b in enumerate(block))
            n = _log_int(rng, 1, 12)
            if 2000 <= math.prod(dims) and math.prod(dims) * n <= (8_000_000 if prec == "f32" else 600_000):
                break
        return _case(None, kind, dims, n, prec=prec, block=",".join(map(str, block)), ncy=rng.randint(3, 6),
                     nmr=rng.randint(3, 5), half=rng.choice([0, 1, 1]), kappa=round(rng.uniform(0.12, 0.132), 4))
    while True:
        dims = (8 * rng.randint(1, 6),) + tuple(8 * rng.randint(1, 3) for _ in range(3))
        V = math.prod(dims)
        n = 2 if kind == "ama" else 12 if kind in ("fh", "deflated") else _log_int(rng, 1, 12)
        if V * n <= {"solve": 3_000_000, "deflated": 1_600_000, "fh": 1_600_000, "ama": 270_000}[kind]:
            break
    if kind == "solve":
        tol = rng.choice([1e-3, 1e-3, 1e-12])
        return _case(None, kind, dims, n, prec="f32", tol=tol, half=rng.choice([0, 1]),
                     source=rng.choice(["point", "random"]), kappa=round(rng.uniform(0.12, 0.13), 4))
    if kind == "deflated":
        return _case(None, kind, dims, n, tol=1e-12, half=1, ns=rng.choice([12, 20]), rounds=3,
                     little=rng.choice([16, 24]), kappa=round(rng.uniform(0.12, 0.1265), 4))
    if kind == "fh":
        m0 = round(rng.uniform(0.1, 0.4), 3)
        return _case(None, kind, dims, n, m0=m0, csw=1.3, eps=0.3, kappa=1.0 / (2 * m0 + 8))
    return _case(None, kind, dims, n, n_iter_2pt=rng.randint(4, 10), n_iter_3pt=rng.randint(4, 10),
                 t_sep=rng.randint(2, dims[0] // 2), direction=rng.choice([1, -1]), half=1, n_gauss=rng.randint(2, 10),
                 kappa=round(rng.uniform(0.12, 0.126), 4))


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _generator(seed, k):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + k)


def _complex_normal(shape, seed, k):
    g = _generator(seed, k)
    return torch.view_as_complex(torch.randn(tuple(shape) + (2,), dtype=torch.float64, device="cuda", generator=g))


def _mat_mul(a, b):
    """3x3 product of component-first matrix fields a, b [3, 3, ...]."""
    o = torch.empty_like(a)
    for i in range(3):
        for j in range(3):
            o[i, j] = a[i, 0] * b[0, j] + a[i, 1] * b[1, j] + a[i, 2] * b[2, j]
    return o


def _dag(a):
    return a.transpose(0, 1).conj()


def _gauge(case, seed):
    """Links U = exp(i eps H), H traceless Hermitian with normal entries: (T, Z, Y, X, 4, 3, 3)."""
    T, X, Y, Z = _dims(case)
    out = torch.empty((T, Z, Y, X, 4, 3, 3), dtype=torch.complex128, device="cuda")
    for mu in range(4):
        A = _complex_normal((3, 3, T, Z, Y, X), seed, 10 + mu)
        H = 0.5 * (A + _dag(A))
        tr = (H[0, 0] + H[1, 1] + H[2, 2]) / 3.0
        for a in range(3):
            H[a, a] -= tr
        H = (1j * case["eps"]) * H
        U = H.clone()                    # the exponential series by Horner's rule
        for k in range(12, 0, -1):
            U = U / k if k == 12 else _mat_mul(H, U) / k
            for a in range(3):
                U[a, a] += 1.0
        r0 = U[0] / torch.linalg.vector_norm(U[0], dim=0)
        r1 = U[1] - (r0.conj() * U[1]).sum(0) * r0
        r1 = r1 / torch.linalg.vector_norm(r1, dim=0)
        r2 = torch.stack([(r0[1] * r1[2] - r0[2] * r1[1]).conj(), (r0[2] * r1[0] - r0[0] * r1[2]).conj(),
                          (r0[0] * r1[1] - r0[1] * r1[0]).conj()])
        for i, r in enumerate((r0, r1, r2)):
            out[..., mu, i, :] = r.permute(1, 2, 3, 4, 0)
    return out


def _site_source(case, seed):
    """A source position on the SAP blocks (multiples of 8 here), moved with the seed."""
    r = np.random.default_rng(int(seed))
    return tuple(8 * int(r.integers(L // 8)) for L in _dims(case))


def _point_sources(dims, src, n):
    T, X, Y, Z = dims
    eta = torch.zeros((n, T, Z, Y, X, 4, 3), dtype=torch.complex128, device="cuda")
    t, x, y, z = src
    for r in range(n):
        eta[r, t, z, y, x, (r % 12) // 3, r % 3] = 1.0
    return eta


def _sources(case, seed):
    T, X, Y, Z = _dims(case)
    if case.get("source") == "point" or case["kind"] == "deflated":
        return _point_sources(_dims(case), _site_source(case, seed), case["n"])
    return _complex_normal((case["n"], T, Z, Y, X, 4, 3), seed, 1)


def _weights(case, seed):
    return torch.from_numpy(np.random.default_rng(int(seed) + 7).standard_normal(case["T"]))


def _ama_sources(case):
    """Two positions whose difference maps the SAP domains onto themselves (an even number of blocks)."""
    T, X, Y, Z = _dims(case)
    return [(0, 0, 0, 0), ((T // 2) // 8 * 8, (X // 2) // 8 * 8, 0, 0)]


def prepare(case, seed):
    kind, dims = case["kind"], _dims(case)
    s = {"case": case}
    U = _gauge(case, seed)
    # a lattice context on a stream of its own, as the solver's CUDA graphs want it
    lat = s["lat"] = qcd.Lattice(dims, stream=torch.cuda.Stream())
    lat.load_gauge(U, case["csw"], case["kappa"], -1)
    if kind == "dirac":
        s["psi"] = _sources(case, seed)
    elif kind == "sap":
        lat.set_params(block=tuple(int(b) for b in case["block"].split(",")), ncy=case["ncy"], nmr=case["nmr"],
                       sap_half=case["half"])
        s["eta"] = _sources(case, seed)
    elif kind in ("solve", "deflated"):
        lat.set_params(block=(4, 4, 4, 4), sap_half=case["half"], precision=case.get("prec", "f32"),
                       dfl=int(kind == "deflated"))
        if kind == "deflated":
            lat.set_params(dfl_little_iters=case["little"])
            T, X, Y, Z = dims
            lat.deflation_setup(_complex_normal((case["ns"], T, Z, Y, X, 4, 3), seed, 2), case["rounds"])
        s["eta"] = _sources(case, seed)
    elif kind == "nucleon":
        # a propagator falls off from its source: normal entries under an exponential in time
        T, X, Y, Z = dims
        p = _complex_normal((12, T, Z, Y, X, 4, 3), seed, 3)
        t = torch.arange(T, device="cuda", dtype=torch.float64)
        s["prop"] = p * torch.exp(-0.05 * torch.minimum(t, T - t))[None, :, None, None, None, None, None]
    elif kind == "smear":
        s["psi"] = _sources(case, seed)
    elif kind == "fh":
        lat.set_params(block=(4, 4, 4, 4), dfl=0)
        s.update(U=U, src=_site_source(case, seed), w=_weights(case, seed))
    elif kind == "ama":
        lat.set_params(block=(4, 4, 4, 4), sap_half=case["half"], dfl=0)
        lat.smear_links(SMEAR["alpha"], SMEAR["n_ape"])
        lat.set_smearing(SMEAR["kappa_g"], case["n_gauss"])
    return s


def run(s):
    c, lat = s["case"], s["lat"]
    kind = c["kind"]
    if kind == "dirac":
        out = lat.apply_dirac(s["psi"], dagger=c["dagger"], precision=c["prec"])
        return out if c["prec"] == "f64" else out.to(torch.complex64)
    if kind == "sap":
        out = lat.apply_sap(s["eta"], precision=c["prec"])
        return out if c["prec"] == "f64" else out.to(torch.complex64)
    if kind in ("solve", "deflated"):
        psi, _ = lat.solve(s["eta"], c["tol"])
        return psi if c["tol"] < 1e-6 else psi.to(torch.complex64)
    if kind == "nucleon":
        corr = lat.nucleon_2pt(s["prop"], (0, 0, 0, 0), precision=c["prec"])
        return corr if c["prec"] == "f64" else corr.astype(np.complex64)
    if kind == "smear":
        # once per configuration the links, then the sources
        lat.smear_links(SMEAR["alpha"], SMEAR["n_ape"])
        lat.set_smearing(SMEAR["kappa_g"], c["n_gauss"])
        return lat.smear_gaussian(s["psi"])
    if kind == "fh":
        m = torch.tensor(c["m0"], dtype=torch.float64, requires_grad=True)
        lam = torch.tensor(0.0, dtype=torch.float64, requires_grad=True)
        C = qcd.nucleon_fh(m, lam, lat, s["U"], c["csw"], s["src"], 1e-12)
        (s["w"] * C[0, :, 0]).sum().backward()
        return {"C": C.detach(), "dm0": m.grad, "dlambda": lam.grad}
    r = lat.ama_nucleon(_ama_sources(c), 1, exact_tol=1e-12, n_iter_2pt=c["n_iter_2pt"], n_iter_3pt=c["n_iter_3pt"],
                        t_sep=c["t_sep"], direction=c["direction"])
    f = np.complex64
    return {"c2_exact": r["c2_all"][2:], "c3_exact": r["c3_all"][2:], "c2_sloppy": r["c2_all"][:2].astype(f),
            "c3_sloppy": r["c3_all"][:2].astype(f), "c2_ama": r["c2_ama"].astype(f), "c3_ama": r["c3_ama"].astype(f)}


# --------------------------------------------------------------------------
# the least a pass has to do
# --------------------------------------------------------------------------
def _sap_flops(V, n, block, ncy, nmr):
    face = sum(2.0 / b for b in block)
    return ncy * V * n * (nmr * (1320.0 * (1.0 - face / 8.0) + 504.0 + 192.0) + 165.0 * face)


def _solve_work(V, n, its, prec="f32", half=0):
    """`its` GCR iterations: a preconditioner and an operator application, Gram-Schmidt against 8 vectors on average."""
    b = 192.0 if prec == "f64" else 96.0
    links = 1152.0 if prec == "f64" else 288.0 if half else 480.0
    flops = its * (_sap_flops(V, n, (4, 4, 4, 4), 5, 4) + V * n * (1824.0 + 8 * 2 * 96.0))
    return {"bytes": its * V * (n * b * (10 * 5 + 2 + 2 * 8 + 8) / 2 + 6 * links) + V * n * 2 * 192.0, "flops": flops}


def _iterations(case, tol):
    """GCR iterations per right-hand side on these fields, about."""
    per_decade = 2.5 if case["kind"] == "fh" else 5.0 if case["kappa"] < 0.127 else 10.0
    return max(3.0, per_decade * -math.log10(tol))


def work(case):
    V, n, kind = math.prod(_dims(case)), case["n"], case["kind"]
    if kind == "dirac":
        f64 = case["prec"] == "f64"
        return {"bytes": V * (n * (192 + (192 if f64 else 96)) + (1152 if f64 else 480)), "flops": 1824.0 * V * n}
    if kind == "sap":
        f64 = case["prec"] == "f64"
        block = [int(b) for b in case["block"].split(",")]
        return {"bytes": V * (n * (192 + (192 if f64 else 96)) + (1152 if f64 else 288 if case["half"] else 480)),
                "flops": _sap_flops(V, n, block, case["ncy"], case["nmr"])}
    if kind in ("solve", "deflated"):
        its = _iterations(case, case["tol"]) * (0.6 if kind == "deflated" else 1.0)
        w = _solve_work(V, n, its, case.get("prec", "f32"), case["half"])
        if kind == "deflated":
            w["flops"] += its * V * n * (1824.0 + 2 * 8 * 12 * case["ns"])
            w["bytes"] += its * V * 2 * 96.0 * (case["ns"] + n)
        return w
    if kind == "nucleon":
        # diquark form: 9 colour pairs, 4 terms each of 16 spin products twice, then two 4x4 traces
        return {"bytes": V * 2304.0, "flops": V * 9 * (4 * 2 * 64 + 2 * 16) * 8.0}
    if kind == "smear":
        # per step and spinor: 6 links on 4 spins; the links: 12 staples of two products, a projection
        return {"bytes": V * (n * 384.0 + 2 * 576.0),
                "flops": V * (n * case["n_gauss"] * 6 * 4 * 72.0 + SMEAR["n_ape"] * 3 * (4 * 2 * 216.0 + 10 * 200.0))}
    if kind == "fh":
        w = _solve_work(V, 36, _iterations(case, 1e-12))
        w["flops"] += V * 36 * 6 * 200 * 8.0
        w["bytes"] += V * 36 * 3 * 192.0
        return w
    a = _solve_work(V, 2 * 12, case["n_iter_2pt"], half=1)
    b = _solve_work(V, 2 * 24, case["n_iter_3pt"], half=1)
    e = _solve_work(V, 36, _iterations(case, 1e-12), half=1)
    sm = V * 3 * 36 * case["n_gauss"] * 6 * 4 * 72.0
    return {"bytes": a["bytes"] + b["bytes"] + e["bytes"], "flops": a["flops"] + b["flops"] + e["flops"] + sm}


# --------------------------------------------------------------------------
# the same in 64 bits, from the definitions (plain torch; component-first fields)
# --------------------------------------------------------------------------
_AX = (-4, -1, -2, -3)          # axis of direction t, x, y, z in (..., T, Z, Y, X)
# gamma_mu = [[0, e], [e^+, 0]]: e_0 = -1, e_k = -i sigma_k
_E = [np.array([[-1, 0], [0, -1]], dtype=complex), np.array([[0, -1j], [-1j, 0]], dtype=complex),
      np.array([[0, -1], [1, 0]], dtype=complex), np.array([[-1j, 0], [0, 1j]], dtype=complex)]


def _gamma(mu):
    z = np.zeros((2, 2))
    return np.diag([1, 1, -1, -1]).astype(complex) if mu == 5 else np.block([[z, _E[mu]], [_E[mu].conj().T, z]])


def _at(f, mu, step):
    """f(x + step mu), periodic."""
    return torch.roll(f, -step, _AX[mu])


class _Exact:
    """The Wilson-clover operator in 64 bits; spinors [4, 3, n, T, Z, Y, X]."""

    def __init__(self, U, case):
        self.kappa, self.block = case["kappa"], None
        self.U = [U[..., mu, :, :].permute(4, 5, 0, 1, 2, 3).contiguous() for mu in range(4)]
        V = self.U[0].shape[2:]
        eye = torch.eye(6, dtype=torch.complex128, device="cuda")
        self.A = [eye[:, :, None, None, None, None].expand(6, 6, *V).clone() for _ in range(2)]
        for mu, nu in itertools.combinations(range(4), 2):
            F = self._field_strength(mu, nu)
            s = 0.5j * (_gamma(mu) @ _gamma(nu) - _gamma(nu) @ _gamma(mu)) * (1j * case["kappa"] * case["csw"])
            for ch in range(2):
                for r, q in itertools.product(range(2), range(2)):
                    w = complex(s[2 * ch + r, 2 * ch + q])
                    if w:
                        self.A[ch][3 * r:3 * r + 3, 3 * q:3 * q + 3] += w * F

    def _field_strength(self, mu, nu):
        a, b = self.U[mu], self.U[nu]
        Q = _mat_mul(_mat_mul(a, _at(b, mu, 1)), _dag(_mat_mul(b, _at(a, nu, 1))))
        am, bm = _at(a, mu, -1), _at(b, nu, -1)
        Q += _mat_mul(_mat_mul(b, _dag(_at(am, nu, 1))), _mat_mul(_dag(_at(b, mu, -1)), am))
        Q += _mat_mul(_mat_mul(_dag(am), _dag(_at(bm, mu, -1))), _mat_mul(_at(am, nu, -1), bm))
        Q += _mat_mul(_mat_mul(_dag(bm), _at(a, nu, -1)), _mat_mul(_at(bm, mu, 1), _dag(a)))
        return (Q - _dag(Q)) / 8.0

    def _wall(self, f, mu, last):
        """Zero (blocks) or sign (time boundary) on the sites whose hop leaves."""
        L, ax = f.shape[_AX[mu]], _AX[mu]
        if self.block:
            b = self.block[mu]
            for k in range(b - 1 if last else 0, L, b):
                f.select(ax, k).zero_()
        elif mu == 0:
            f.select(ax, L - 1 if last else 0).neg_()
        return f

    def D(self, psi, dagger=False, block=None):
        """D psi, D^+ psi, or with `block` the operator restricted to the blocks."""
        self.block = block
        out = torch.empty_like(psi)
        for ch in range(2):
            v, o = psi[2 * ch:2 * ch + 2].reshape(6, *psi.shape[2:]), out[2 * ch:2 * ch + 2].view(6, *psi.shape[2:])
            for i in range(6):
                o[i] = sum(self.A[ch][i, j] * v[j] for j in range(6))
        for mu in range(4):
            e = _E[mu]
            for fwd in (True, False):
                sg = -1.0 if fwd != dagger else 1.0
                h = torch.empty_like(psi[:2])
                for r in range(2):
                    q = 0 if e[r, 0] else 1
                    h[r] = psi[r] + complex(sg * e[r, q]) * psi[2 + q]
                if fwd:
                    h = _at(h, mu, 1)
                    g = sum(self.U[mu][:, b][None, :, None] * h[:, b][:, None] for b in range(3))
                    g = self._wall(g, mu, True)
                else:
                    g = sum(self.U[mu][b].conj()[None, :, None] * h[:, b][:, None] for b in range(3))
                    g = self._wall(_at(g, mu, -1), mu, False)
                g *= -self.kappa
                out[:2] += g
                for r in range(2):
                    q = 0 if e.conj().T[r, 0] else 1
                    out[2 + r] += complex(sg * e.conj().T[r, q]) * g[q]
        return out

    def sap(self, eta, block, ncy, nmr):
        n, (T, Z, Y, X) = eta.shape[2], eta.shape[3:]
        bt, bx, by, bz = block
        split = (n, T // bt, bt, Z // bz, bz, Y // by, by, X // bx, bx)

        def blocksum(f):
            t = f.reshape(split).sum((2, 4, 6, 8), keepdim=True)
            return t.expand(split).reshape(n, T, Z, Y, X)

        par = sum(torch.div(torch.arange(L, device="cuda"), b, rounding_mode="floor").view(sh) for L, b, sh in
                  ((T, bt, (-1, 1, 1, 1)), (Z, bz, (-1, 1, 1)), (Y, by, (-1, 1)), (X, bx, (-1,))))
        psi, rho = torch.zeros_like(eta), eta.clone()
        for _ in range(ncy):
            for colour in range(2):
                m = ((par % 2) == colour).to(torch.float64)
                r, x = rho * m, torch.zeros_like(rho)
                for _ in range(nmr):
                    p = self.D(r, block=block)
                    pp = blocksum((p.real ** 2 + p.imag ** 2).sum((0, 1)))
                    pr = blocksum((p.conj() * r).sum((0, 1)))
                    a = torch.where(pp > 0, pr / torch.where(pp > 0, pp, 1.0), 0.0)
                    x += a * r
                    r -= a * p
                psi += x
                rho -= self.D(x)
        return psi

    def solve(self, eta):
        """D x = eta to a relative residual of 1e-13: BiCGStab, restarted from the true residual."""
        dot = lambda a, b: (a.conj() * b).sum((0, 1, 3, 4, 5, 6))[:, None, None, None, None]  # noqa: E731
        x, norm = torch.zeros_like(eta), dot(eta, eta).real
        for _ in range(6):
            r = eta - self.D(x)
            if bool((dot(r, r).real <= 1e-26 * norm).all()):
                return x
            x += self._bicgstab(r, 1e-10, dot)
        return None

    def _bicgstab(self, eta, tol, dot):
        """Every right-hand side with its own scalars."""
        x, r, r0, p = torch.zeros_like(eta), eta.clone(), eta.clone(), eta.clone()
        rho = dot(eta, eta)
        norm = rho.real
        for _ in range(2000):
            v = self.D(p)
            a = rho / dot(r0, v)
            s = r - a * v
            t = self.D(s)
            tt = dot(t, t)
            w = torch.where(tt.abs() > 0, dot(t, s) / tt, 0.0)
            x += a * p + w * s
            r = s - w * t
            if bool((dot(r, r).real <= tol ** 2 * norm).all()):
                break
            new = dot(r0, r)
            p = r + (new / rho) * (a / w) * (p - w * v)
            rho = new
        return x


def _inward(psi):
    return psi.permute(5, 6, 0, 1, 2, 3, 4).contiguous()


def _outward(psi):
    return psi.permute(2, 3, 4, 5, 6, 0, 1).contiguous()


_EPS = [(a, b, c, float(np.linalg.det(np.eye(3)[[a, b, c]]))) for a, b, c in itertools.permutations(range(3))]


def _wick(Su, Sd):
    """tr[P+- <N N-bar>] per site, from S [4, 3, 4, 3, sites] (sink spin, colour, source spin, colour): [2, sites]."""
    g5, g0 = _gamma(5), _gamma(0)
    G = _gamma(0) @ _gamma(2) @ g5
    Gs = g0 @ G.conj().T @ g0.T
    t = lambda m: torch.tensor(m, dtype=torch.complex128, device="cuda")  # noqa: E731
    P = [t(0.5 * (np.eye(4) + g0)), t(0.5 * (np.eye(4) - g0))]
    Q = torch.einsum("ij,jakbs,kl->ialbs", t(G), Sd, t(Gs))
    out = 0.0
    for a, b, c, e in _EPS:
        for d, f, h, e2 in _EPS:
            # G = eps eps' { S^{cc'} tr[S^{aa'T} G S^{bb'} G'] - S^{ca'} (G S^{bb'} G')^T S^{ac'} }
            tr = (Su[:, a, :, d] * Q[:, b, :, f]).sum((0, 1))
            M = torch.einsum("ijs,kjs,kls->ils", Su[:, c, :, d], Q[:, b, :, f], Su[:, a, :, h])
            Z = Su[:, c, :, h] * tr - M
            out = out + e * e2 * torch.stack([torch.einsum("ij,jis->s", p, Z) for p in P])
    return out


def _two_point(Su, Sd, t0):
    """Correlators [2, T] from propagators [4, 3, 12, T, Z, Y, X], one time-slice at a time."""
    T = Su.shape[3]
    C = []
    for t in range(T):
        s = [S[:, :, :, t].reshape(4, 3, 4, 3, -1) for S in (Su, Sd)]
        C.append(_wick(*s).sum(-1) * (-1.0 if t < t0 else 1.0))
    return torch.stack([C[(t0 + k) % T] for k in range(T)], 1)


def _exact_smeared_links(U):
    """APE steps on the spatial links; the projection by Newton's iteration for the polar factor."""
    U = [u.permute(2, 3, 4, 5, 0, 1) for u in U]
    roll = lambda f, mu, k: torch.roll(f, -k, (0, 3, 2, 1)[mu])  # noqa: E731
    for _ in range(SMEAR["n_ape"]):
        new = list(U)
        for k in range(1, 4):
            W = U[k].clone()
            for j in range(1, 4):
                if j != k:
                    W += SMEAR["alpha"] * (U[j] @ roll(U[k], j, 1) @ roll(U[j], k, 1).mH)
                    d = roll(U[j], j, -1)
                    W += SMEAR["alpha"] * (d.mH @ roll(U[k], j, -1) @ roll(d, k, 1))
            W = W / (torch.linalg.matrix_norm(W)[..., None, None] / math.sqrt(3.0))
            for _ in range(20):
                W = 0.5 * (W + torch.linalg.inv(W).mH)
            det = torch.linalg.det(W)
            new[k] = W * torch.polar(torch.ones_like(det.real), -torch.angle(det) / 3.0)[..., None, None]
        U = new
    return [u.permute(4, 5, 0, 1, 2, 3) for u in U]


def _exact_gauss(U, psi, n):
    k = SMEAR["kappa_g"]
    for _ in range(n):
        out = psi.clone()
        for mu in range(1, 4):
            f, b = _at(psi, mu, 1), None
            out += k * sum(U[mu][:, c][None, :, None] * f[:, c][:, None] for c in range(3))
            b = sum(U[mu][c].conj()[None, :, None] * psi[:, c][:, None] for c in range(3))
            out += k * _at(b, mu, -1)
        psi = out / (1.0 + 6.0 * k)
    return psi


def exact(case, seed):
    V, n, kind = math.prod(_dims(case)), case["n"], case["kind"]
    if kind == "nucleon":
        p = _inward(prepare(case, seed)["prop"])
        return _two_point(p, p, 0).cpu().numpy()
    if kind in ("solve", "deflated") and V * n > 2_000_000:
        return None                                    # minutes in plain 64-bit torch
    ex = _Exact(_gauge(case, seed), case)
    if kind == "smear":
        return _outward(_exact_gauss(_exact_smeared_links(ex.U), _inward(_sources(case, seed)), case["n_gauss"]))
    if kind in ("dirac", "sap"):
        src = _sources(case, seed)
        out = torch.empty_like(src)
        for r in range(n):                             # one at a time: the memory of a batch
            v = _inward(src[r:r + 1])
            if kind == "dirac":
                v = ex.D(v, dagger=case["dagger"])
            else:
                v = ex.sap(v, tuple(int(b) for b in case["block"].split(",")), case["ncy"], case["nmr"])
            out[r:r + 1] = _outward(v)
        return out
    if kind in ("solve", "deflated"):
        x = ex.solve(_inward(_sources(case, seed)))
        return None if x is None else _outward(x)
    if V > 140_000:
        return None
    if kind == "ama":
        src = _ama_sources(case)[0]
        links = _exact_smeared_links(ex.U)
        S = ex.solve(_exact_gauss(links, _inward(_point_sources(_dims(case), src, 12)), case["n_gauss"]))
        if S is None:
            return None
        S = _exact_gauss(links, S, case["n_gauss"])
        return {"c2_exact": _two_point(S, S, src[0])[None].cpu().numpy(), "c3_exact": None, "c2_sloppy": None,
                "c3_sloppy": None, "c2_ama": None, "c3_ama": None}
    # the differentiable correlator: S = D_w^-1 = 2 kappa D^-1, H = dL/dS slot by slot, Y = (D_w^+)^-1 H
    k2, src = 2.0 * case["kappa"], _site_source(case, seed)
    S = ex.solve(_inward(_point_sources(_dims(case), src, 12)))
    if S is None:
        return None
    Su, Sd = (k2 * S).requires_grad_(), (k2 * S).detach().clone().requires_grad_()
    C = _two_point(Su, Sd, src[0])
    (_weights(case, seed).cuda() * C[0].real).sum().backward()
    g5 = torch.tensor([1.0, 1.0, -1.0, -1.0], dtype=torch.float64, device="cuda").view(4, 1, 1, 1, 1, 1, 1)
    dm = dl = 0.0
    g35 = torch.tensor(_gamma(3) @ _gamma(5), device="cuda")
    GS = torch.einsum("rq,qancdef->rancdef", g35, Su.detach())
    for H, sg in ((Su.grad, 1.0), (Sd.grad, -1.0)):
        Y = ex.solve(g5 * H)
        if Y is None:
            return None
        Y = k2 * g5 * Y
        dm -= float((Y.conj() * Su.detach()).sum().real)
        dl -= sg * float((Y.conj() * GS).sum().real)
    Cr = torch.view_as_real(C.detach()).cpu()
    return {"C": Cr, "dm0": torch.tensor(dm, dtype=torch.float64), "dlambda": torch.tensor(dl, dtype=torch.float64)}
