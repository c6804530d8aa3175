"""Lane groups whose walkers fill a CTA's shared memory to the last byte
(232,448 bytes): batches and servers run what a single handle runs."""
import math

import numpy as np
import pytest

from paper_1312_3004_gb300 import REWL, Batch, Server

pytestmark = pytest.mark.gpu

# W + 1 bins and lattice: 232,448 bytes for one walker; 29,056 for each of eight
ONE = dict(q=10, L=128, h=2, overlap=0.8139, m=1)
EIGHT = dict(q=10, L=80, h=8, overlap=0.1033, m=134)


def job(shape, K):
    return dict(shape, lnf_final=1e-6, flatness=0.8, exchange_interval=K, seed=3)


def test_sizes_are_those_meant():
    for shape, W in ((ONE, 27627), (EIGHT, 1759)):
        n = 2 * shape["L"] ** 2
        assert math.ceil(n / (1 + (shape["h"] - 1) * (1 - shape["overlap"]))) == W


@pytest.mark.parametrize("shape", [ONE, EIGHT])
def test_server(shape):
    s = Server(256 << 20, max_jobs=2)
    i = s.submit(**job(shape, 20))
    for n in range(2):
        s.step(2)
    assert s.poll(i) == "running"
    assert s.info()["flips"] == s.info()["rounds"] * 20 * shape["h"] * shape["m"]


def test_batch():
    j = job(ONE, 300)
    b = Batch([j], lanes=32)
    b.run(2)
    a = REWL(j["q"], j["L"], j["h"], j["overlap"], j["m"], 1e-6, 0.8, 300, 3)
    a.run(2)
    for f in ("spins", "energy", "steps", "lng", "hist", "mask"):
        assert np.array_equal(b.instance(0).get(f), a.get(f)), f


def test_server_job_whose_lattice_does_not_fit_beside_its_window():
    """a single handle keeps such a lattice in global memory; the server runs
    its jobs a thread per walker while one of them is resident"""
    big = dict(q=10, L=200, h=9, overlap=0.75, m=1, lnf_final=1e-6, flatness=0.8, exchange_interval=20, seed=3)
    small = dict(big, L=8, h=2)
    s = Server(256 << 20, max_jobs=4)
    i = s.submit(**small)
    s.step(1)
    k = s.submit(**big)
    s.step(3)
    assert s.mapping()[0] == 1
    assert s.poll(k) == "running" and s.job_info(k)["rounds"] == 3 and s.job_info(i)["rounds"] == 4
    assert s.job_info(k)["flips"] == 3 * 20 * 9
    s.cancel(k)
    s.step(1)
    assert s.mapping()[0] == 32 and s.job_info(i)["rounds"] == 5
