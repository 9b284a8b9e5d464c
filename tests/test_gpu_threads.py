"""Contexts used from several host threads at once share the kernels: no call may
change what another thread's launches are allowed.  The sizes below make each kernel's
shared memory differ between the contexts: 32 and 3 deflation fields (the little
operator and the projection), spatial volumes of 8^3 and 6^3 sites (the contraction and
its derivative), blocks of 256 and 32 sites (the sweeps)."""
import threading

import numpy as np
import pytest
import torch

from gpu_util import to_dev
from paper_1605_00564_gb300 import synth

pytestmark = pytest.mark.gpu


def run_together(works, repeat):
    """Runs each work `repeat` times on a thread of its own, all at once; raises what a thread raised."""
    errors, start = [], threading.Barrier(len(works))

    def loop(work):
        try:
            start.wait(60)
            for _ in range(repeat):
                work()
        except Exception as e:      # noqa: BLE001 (handed to the test)
            errors.append(e)

    th = [threading.Thread(target=loop, args=(w,)) for w in works]
    for t in th:
        t.start()
    for t in th:
        t.join()
    if errors:
        raise errors[0]


def context(dims, seed, **params):
    from paper_1605_00564_gb300.qcd import Lattice
    lat = Lattice(dims, stream=torch.cuda.Stream())
    lat.load_gauge(synth.gauge_field(dims, 0.3, seed), 1.0, 0.12, -1)
    lat.set_params(**params)
    return lat


def test_deflated_solves():
    dims = (8, 8, 8, 8)
    lats = [context(dims, 5, block=(4, 4, 4, 4), dfl=0, dfl_little_iters=24),
            context(dims, 6, block=(4, 2, 2, 2), dfl=0, dfl_little_iters=24)]
    works = []
    for lat, ns, n in zip(lats, (32, 3), (12, 1)):
        lat.deflation_setup(to_dev(synth.random_spinor(dims, 7, nrhs=ns)), 1)
        lat.set_params(dfl=1)
        eta = to_dev(synth.random_spinor(dims, 8, nrhs=n))
        ref = lat.solve(eta, 1e-6)[0].clone()

        def work(lat=lat, eta=eta, ref=ref):
            assert torch.equal(lat.solve(eta, 1e-6)[0], ref)
        works.append(work)
    torch.cuda.synchronize()
    run_together(works, 20)
    for lat in lats:
        lat.close()


@pytest.mark.parametrize("half", [0, 1])
def test_sweeps(half):
    dims = (16, 8, 8, 8)
    works, lats = [], []
    for block in ((8, 2, 4, 4), (4, 2, 2, 2)):
        lat = context(dims, 9, block=block, ncy=2, nmr=2, sap_half=half, graphs=0)
        eta = to_dev(synth.random_spinor(dims, 10, nrhs=2))
        ref = lat.apply_sap(eta).clone()

        def work(lat=lat, eta=eta, ref=ref):
            assert torch.equal(lat.apply_sap(eta), ref)
        works.append(work)
        lats.append(lat)
    torch.cuda.synchronize()
    run_together(works, 300)
    for lat in lats:
        lat.close()


def test_contractions():
    from paper_1605_00564_gb300.qcd import Lattice
    works, lats = [], []
    for dims in ((8, 8, 8, 8), (8, 6, 6, 6), (8, 3, 3, 3)):
        lat = Lattice(dims, stream=torch.cuda.Stream())
        lat.load_gauge(synth.unit_gauge(dims), 1.0, 0.12, -1)
        rng = np.random.default_rng(3)
        prop = to_dev(rng.standard_normal(lat.spinor_shape(12) + (2,)) @ np.array([1, 1j]))
        ref = lat.nucleon_2pt(prop, (1, 0, 0, 0))

        def work(lat=lat, prop=prop, ref=ref):
            assert np.array_equal(lat.nucleon_2pt(prop, (1, 0, 0, 0)), ref)
        works.append(work)
        lats.append(lat)
    torch.cuda.synchronize()
    run_together(works, 300)
    for lat in lats:
        lat.close()

