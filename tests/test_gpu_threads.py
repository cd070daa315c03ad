"""Handles of different sizes used from different host threads at the same time."""
import threading

import numpy as np
import pytest

from paper_1908_08553_gb300 import inputs, tn

pytestmark = pytest.mark.gpu


def _together(jobs, repeat):
    """Each job `repeat` times on a thread of its own, all at once; the results by job."""
    out, errors, start = [[] for _ in jobs], [], threading.Barrier(len(jobs))

    def work(k, job):
        try:
            start.wait()
            for _ in range(repeat):
                out[k].append(job())
        except Exception as e:      # noqa: BLE001 -- reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=(k, j)) for k, j in enumerate(jobs)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    return out


# shared memory of 1 KB (chi 2) and 82 KB (chi 16) for the SVDs
def test_boundary_mps_of_different_bonds(ctx_pair):
    L = W = 3
    lats = [tn.tn_create_lattice(c, L, W, 2) for c in ctx_pair]
    try:
        for lat in lats:
            tn.tn_set_site_tensors(lat, inputs.random_lattice(L, W, 2, 5100))
        alone = [tn.tn_bmps_energy(lat, chi, 1.0, 3.04, L, W, tn.TN_FP32)[0].energy
                 for lat, chi in zip(lats, (16, 2))]
        jobs = [lambda lat=lat, chi=chi: tn.tn_bmps_energy(lat, chi, 1.0, 3.04, L, W, tn.TN_FP32)[0].energy
                for lat, chi in zip(lats, (16, 2))]
        for got, ref in zip(_together(jobs, 300), alone):
            assert np.all(np.array(got) == ref)
    finally:
        for lat in lats:
            tn.tn_destroy_lattice(lat)


# 4 KB (D = 2) and 47 KB (D = 3) for the bond updates
def test_evolutions_of_different_bonds(ctx_pair):
    L = W = 3
    lats = [tn.tn_create_lattice(c, L, W, D) for c, D in zip(ctx_pair, (3, 2))]

    def evolve(lat, D):
        tn.tn_set_site_tensors(lat, inputs.random_lattice(L, W, D, 5200))
        return tn.tn_ite_run(lat, L, W, 1.0, 3.04, 0.05, 2, D, 1e-12, 2)[0][0]

    try:
        alone = [evolve(lat, D) for lat, D in zip(lats, (3, 2))]
        jobs = [lambda lat=lat, D=D: evolve(lat, D) for lat, D in zip(lats, (3, 2))]
        for got, ref in zip(_together(jobs, 100), alone):
            assert np.all(np.array(got) == ref)
    finally:
        for lat in lats:
            tn.tn_destroy_lattice(lat)


@pytest.fixture
def ctx_pair():
    import torch
    torch.cuda.init()
    c = [tn.tn_ctx_create(0, 0) for _ in range(2)]
    yield c
    for k in c:
        tn.tn_ctx_destroy(k)
