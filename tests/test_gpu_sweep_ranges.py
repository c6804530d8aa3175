"""ln g at magnitudes between those of the other comparisons, in both mappings,
against the binary64 reference sweep; exact."""
import numpy as np
import pytest

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
