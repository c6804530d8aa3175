"""ln g at magnitudes between those of the other comparisons, in both mappings,
against the binary64 reference sweep; exact."""
import numpy as np
import pytest

from paper_1312_3004_gb300 import _lib
from test_gpu_batch_resolution import same

pytestmark = pytest.mark.gpu


def start(offset, lnf, scale=1.0):
    def prepare(r):
        b = np.arange(r.B)
        r.set("lng", scale * (40.0 * np.sin(b / 17.0) ** 2 + 0.37 * b) + offset)
        r.set("lnf", np.full(r.h, lnf))
    return prepare


# (half-units 2^-k of the shadow: k = 27, 26, 25 in the middle three)
@pytest.mark.parametrize("offset", [5e9, 1e10, 2e10, 4e10, 8e10])
@pytest.mark.parametrize("lnf", [0.0, 2.0**-10, 1e-3, 1.0])
@pytest.mark.parametrize("lanes", [1, 32])
def test_where_leading_words_stop(offset, lnf, lanes):
    same((10, 12, 2, 0.75, 2, 1e-300, 0.999, 2000, 13), 4, 3, lanes, start(offset, lnf))


@pytest.mark.parametrize("lattice", [1, 2])
@pytest.mark.parametrize("lnf", [1.0, 0.7])
@pytest.mark.parametrize("lanes", [1, 32])
def test_bins_that_become_exact(lattice, lnf, lanes):
    """values whose low bits the shadow drops take binary64 adds until they have
    grown to where it holds them: both copies of ln g are written in one launch"""
    def prepare(r):
        b = np.arange(r.B)
        r.set("lng", np.where(b % 3 == 0, 1.0 / (b + 3), 1024.0 + b / 7.0))
        r.set("lnf", np.full(r.h, lnf))
    same((10, 8, 2, 0.75, 3, 1e-300, 0.999, 3000, 13), 4, 3, lanes, prepare, options=[(_lib.OPT_LATTICE, lattice)])
