"""Lane groups of 2, 4 and 8 where sites share conflict marks and lattices stay
packed, against the binary64 reference sweep; exact."""
import pytest

from paper_1312_3004_gb300 import _lib
from test_gpu_batch_resolution import same

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice", [1, 2])
@pytest.mark.parametrize("L", [22, 23, 32, 33, 45, 46, 80, 91])  # 512, 1024, 2048 entries
@pytest.mark.parametrize("lanes", [2, 4, 8])
def test_shared_marks(L, lanes, lattice):
    same((10, L, 8, 0.75, 2, 1e-6, 0.8, 1500, 5), 4, 2, lanes, options=[(_lib.OPT_LATTICE, lattice)])
