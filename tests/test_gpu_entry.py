"""The drawn and entered configurations, a warp and a thread per walker, against
the oracle's; exact."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1312_3004_gb300 import REWL

pytestmark = pytest.mark.gpu


# (152 SMs: a thread per walker above 152 (20 + N / 5) walkers, up to 32 x 32 sites)
@pytest.mark.parametrize("q,L,h,m,bits", [
    (2, 3, 1, 256, 8), (10, 8, 16, 256, 4), (10, 8, 21, 256, 4), (10, 9, 24, 256, 8), (3, 12, 32, 256, 4),
    (30, 16, 48, 256, 8), (10, 32, 160, 230, 4), (10, 33, 160, 256, 4),
])
def test_entered_configurations(q, L, h, m, bits):
    args = (q, L, h, 0.75, m, 1e-6, 0.8, 100, 77)
    gpu, orc = REWL(*args, spin_bits=bits), O.OracleREWL(*args)
    assert np.array_equal(gpu.get("spins"), orc.sigma())
    assert np.array_equal(gpu.get("energy"), orc.E())
    assert np.array_equal(gpu.get("replica"), orc.rep())
