"""Lane groups resolve a whole batch of steps at once; here at the sizes and
states where that can go wrong, against the binary64 reference sweep
(REWL_OPT_SWEEP_KERNEL = 1), which takes one step after another.  Both compute
the same states, so every comparison is exact."""
import numpy as np
import pytest

from paper_1312_3004_gb300 import REWL, _lib

pytestmark = pytest.mark.gpu

FIELDS = ("spins", "energy", "hist", "lng", "mask", "steps")


def same(args, bits, rounds, lanes, prepare=None, options=()):
    a, b = REWL(*args, spin_bits=bits), REWL(*args, spin_bits=bits)
    a.set_option(_lib.OPT_LANES, lanes)
    for o, v in options:
        a.set_option(o, v)
    b.set_option(_lib.OPT_SWEEP_KERNEL, 1)
    for r in (a, b):
        if prepare:
            prepare(r)
        r.run(rounds)
    for f in FIELDS:
        x, y = a.get(f), b.get(f)
        if f == "lng":
            x, y = x.view(np.uint64), y.view(np.uint64)
        assert np.array_equal(x, y), f
    sa, sb = a.stats(), b.stats()
    assert all(sa[k] == sb[k] for k in ("flips", "accepted", "exch_accepted"))


@pytest.mark.parametrize("K", [1, 2, 31, 32, 33, 63, 65])
@pytest.mark.parametrize("lanes", [32, 8, 2])
def test_last_batch_of_a_launch(K, lanes):
    same((10, 8, 3, 0.75, 3, 1e-6, 0.8, K, 5), 4, 6, lanes)


@pytest.mark.parametrize("L", [3, 4, 17, 18, 32, 47, 90, 91])  # twin sites found ahead up to 300 sites; own conflict marks up to 8192
@pytest.mark.parametrize("q,bits", [(2, 8), (10, 4), (20, 8)])
def test_lattice_sizes(L, q, bits):
    h = 1 if L < 5 else 3
    same((q, L, h, 0.75, 2, 1e-6, 0.8, 3000, 7), bits, 3, 32)


@pytest.mark.parametrize("lnf", [0.0, 1.0, 2.0**-7, 2.0**-12, 2.0**-13, 2.0**-20, 2.0**-45, 1e-3, 1e-5, 0.3, 3.7])
@pytest.mark.parametrize("L", [6, 20])
def test_ln_f(lnf, L):
    """counted at once, counted where it matters, not at all; whole units of the
    shadow or not (then every ln f step is a binary64 add)"""
    def prepare(r):
        r.run(4)
        r.set("lnf", np.full(r.h, lnf))
    same((5, L, 2, 0.75, 3, 1e-300, 0.999, 2000, 11), 4, 4, 32, prepare)


@pytest.mark.parametrize("scale,offset", [(1.0, 0.0), (0.125, 0.0), (1e-9, 0.0), (1.0, 1e6), (1.0, 3e9), (1.0, 1e11), (1.0, 1e13), (1.0, 1e15)])
@pytest.mark.parametrize("lnf", [0.0, 2.0**-10, 1.0])
def test_range_of_ln_g(scale, offset, lnf):
    """shadows whose unit is finer and coarser than the draws' (leading words
    that cannot decide send every decision to 64 bits); ln f half-way between two
    last places"""
    def prepare(r):
        b = np.arange(r.B)
        r.set("lng", scale * (40.0 * np.sin(b / 17.0) ** 2 + 0.37 * b) + offset)
        r.set("lnf", np.full(r.h, lnf))
    same((10, 12, 2, 0.75, 2, 1e-300, 0.999, 2000, 13), 4, 3, 32, prepare)


@pytest.mark.parametrize("lat", [1, 2])
@pytest.mark.parametrize("q,bits", [(10, 4), (10, 8), (30, 8)])
def test_lattice_placement(lat, q, bits):
    same((q, 15, 4, 0.75, 3, 1e-6, 0.8, 2500, 17), bits, 4, 32, options=[(_lib.OPT_LATTICE, lat)])


@pytest.mark.parametrize("lattice", [1, 2])  # in global memory, in shared memory
@pytest.mark.parametrize("L", [3, 4, 5, 7, 8, 9, 16, 33])  # neighbours in the word of the site, across its edge, the same word twice
@pytest.mark.parametrize("q,bits", [(2, 8), (10, 4), (20, 8), (2, 4)])
def test_thread_per_walker_words(L, q, bits, lattice):
    h = 1 if L < 5 else 3
    same((q, L, h, 0.75, 2, 1e-6, 0.8, 501, 13), bits, 4, 1, options=[(_lib.OPT_LATTICE, lattice)])


@pytest.mark.parametrize("K", [1, 2, 3])
def test_thread_per_walker_short_rounds(K):
    same((10, 6, 2, 0.75, 3, 1e-6, 0.8, K, 17), 4, 40, 1)
