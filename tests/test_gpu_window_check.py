"""The window check for walkers that are no multiple of eight, on wide windows."""
import time

import numpy as np
import pytest

from paper_1312_3004_gb300 import REWL, _lib
from test_gpu_dispatch import like_the_oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("schedule", [0, 1])
@pytest.mark.parametrize("m", [5, 6, 7, 8, 15, 16, 23])
def test_remainders(m, schedule):
    like_the_oracle((4, 33, 1, 0.75, m, 1e-2, 0.3, 5000, 3), 3, schedule)


def test_five_walkers_take_no_longer_than_eight():
    """(their histogram rows are read with as many loads in flight)"""
    def check(m):
        r = REWL(10, 80, 1, 0.75, m, 1e-12, 0.8, 10, 5)
        r.run(2)
        times = []
        for _ in range(6):
            t = time.perf_counter()
            for _ in range(50):
                r.run_phase(_lib.PHASE_CHECK)
            r.sync()
            times.append(time.perf_counter() - t)
        return min(times)
    assert np.median([check(5) / check(8) for _ in range(3)]) < 1.25
