"""Windows so wide that a walker keeps few conflict marks (ln g shadow and lattice
above 96 KB: 512, which nearly every batch shares): lane groups against the
binary64 reference sweep, production against the oracle; exact."""
import pytest

from test_gpu_batch_resolution import same
from test_gpu_production_batch import compare

pytestmark = pytest.mark.gpu

# shadow 103 KB; 112 KB beside a lattice in global memory; 101 KB with the lattice; 75 KB: 8192 marks for 8281 sites
SHAPES = [(80, 1), (200, 20), (78, 1), (91, 5)]


@pytest.mark.parametrize("L,h", SHAPES)
@pytest.mark.parametrize("q,bits", [(10, 4), (10, 8), (30, 8)])
@pytest.mark.parametrize("lanes", [32, 16, 4])
def test_sweep(L, h, q, bits, lanes):
    same((q, L, h, 0.75, 2, 1e-6, 0.8, 2500, 21), bits, 2, lanes)


@pytest.mark.parametrize("L,h", SHAPES)
@pytest.mark.parametrize("q,bits", [(10, 4), (30, 8)])
def test_production(L, h, q, bits):
    compare((q, L, h, 0.75, 1, 1e-6, 0.8, 1500, 9), bits, 5, rounds=2, wl=1)
