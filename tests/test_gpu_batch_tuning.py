"""The batch autotuner's candidates and what a batch reports of itself."""
import pytest

from paper_1312_3004_gb300 import Batch

pytestmark = pytest.mark.gpu


def jobs(*Ls):
    return [dict(q=4, L=L, h=2, overlap=0.75, m=2, lnf_final=1e-6, flatness=0.8, exchange_interval=200, seed=i + 1)
            for i, L in enumerate(Ls)]


@pytest.mark.parametrize("Ls,groups", [((8, 10), 2), ((48, 60), 2), ((8, 60), 3)])  # two small walkers, or one large one, a CTA
def test_lane_group_candidates_differ(Ls, groups):
    timed, _ = Batch(jobs(*Ls)).autotune(1)
    for bits in (4, 8):
        kb = [t["cta_kb"] for t in timed if t["lanes"] == 32 and t["spin_bits"] == bits]
        assert len(kb) == groups and all(k > 0 for k in kb)
    assert all(t["cta_kb"] == 0 for t in timed if t["lanes"] == 1)


def test_reported_shared_memory_is_that_of_a_cta():
    small, large = Batch(jobs(8), lanes=32).config(), Batch(jobs(80), lanes=32).config()
    # two walkers of 8 x 8 sites; one of 80 x 80: its ln g shadow of 10,240 bins, sites as bytes, marks
    assert 0 < small["cta_kb"] <= 18
    assert 10_241 * 8 / 1024 < large["cta_kb"] < (10_241 * 8 + 3 * 6400) / 1024 + 1
