"""The barrier, exchange, set-up and batch kernels at the sizes where their
dispatch changes; every comparison is exact: with the oracle, or with the same
runs alone."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1312_3004_gb300 import REWL, Batch, _lib
from test_gpu_batch_resolution import same
from tie_trace import differing, gpu_state, gpu_ties, oracle_state

pytestmark = pytest.mark.gpu

FIELDS = ("spins", "energy", "replica", "steps", "lng", "hist", "mask", "lnf", "iter", "done", "round")


def like_the_oracle(args, rounds, schedule=0):
    gpu, orc = REWL(*args), O.OracleREWL(*args)
    if schedule:
        gpu.set_option(_lib.OPT_SCHEDULE, 1)
        orc.set_schedule(1)
    gpu.run(rounds)
    orc.run(rounds)
    diff = differing(gpu_state(gpu), oracle_state(orc))
    assert not diff, (diff, gpu_ties(gpu))


@pytest.mark.parametrize("schedule", [0, 1])
@pytest.mark.parametrize("m", [1, 3, 4, 5, 8, 9, 17, 33])  # one pass over the bins up to 4 walkers; a warp per walker above
def test_window_check(m, schedule):
    like_the_oracle((3, 4, 2, 0.75, m, 1e-2, 0.5, 800, 3), 12, schedule)


@pytest.mark.parametrize("h,m", [(65, 256), (67, 256), (66, 251), (3, 1)])  # 8192 partners are held at a time
def test_exchange_in_parts(h, m):
    like_the_oracle((2, 24, h, 0.75, m, 1e-3, 0.8, 3, 5), 4)


@pytest.mark.parametrize("h,m", [(9, 256), (17, 129), (3, 256)])  # 1024 in a batch
@pytest.mark.parametrize("lanes", [1, 32])
def test_batch_exchange_in_parts(h, m, lanes):
    job = dict(q=2, L=8, h=h, overlap=0.75, m=m, lnf_final=1e-3, flatness=0.8, exchange_interval=7, seed=9)
    b = Batch([job, dict(job, seed=10)], lanes=lanes)
    b.run(5)
    for i, seed in enumerate((9, 10)):
        a = REWL(2, 8, h, 0.75, m, 1e-3, 0.8, 7, seed)
        a.run(5)
        for f in FIELDS:
            assert np.array_equal(b.instance(i).get(f), a.get(f)), f


@pytest.mark.parametrize("lanes", [1, 32])
def test_batch_of_many_sizes(lanes):
    """more sweep launches a round than streams beside each other"""
    Ls = [4, 5, 6, 7, 8, 10, 12, 14, 16, 20, 24, 28, 32, 40, 48, 64, 80, 96]
    jobs = [dict(q=(2, 20)[i % 2], L=L, h=1 if L < 6 else 2, overlap=0.75, m=2, lnf_final=1e-6, flatness=0.8,
                 exchange_interval=300, seed=i + 1) for i, L in enumerate(Ls)]
    b = Batch(jobs, lanes=lanes)
    b.run(6)
    for i, j in enumerate(jobs):
        a = REWL(j["q"], j["L"], j["h"], 0.75, 2, 1e-6, 0.8, 300, j["seed"])
        a.run(6)
        for f in FIELDS:
            assert np.array_equal(b.instance(i).get(f), a.get(f)), (j, f)


@pytest.mark.parametrize("L", [181, 182, 200])  # lattices in global memory above 16 KB: fewer conflict marks than sites
def test_far_lattices(L):
    same((10, L, 40, 0.75, 1, 1e-6, 0.8, 2000, 5), 4, 2, 32)
