"""Production by lane groups, at the states and sizes where its shadow of ln g,
its spin counts and its classes can go wrong, against the oracle's production
run.  H(E, O) and the state agree exactly."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_1312_3004_gb300 import REWL
from tie_trace import differing, gpu_state, oracle_state

pytestmark = pytest.mark.gpu


def compare(args, bits, n_obins, lng=None, rounds=2, wl=2):
    gpu, orc = REWL(*args, spin_bits=bits), O.OracleREWL(*args)
    gpu.run(wl)
    orc.run(wl)
    gpu.production_start(n_obins)
    orc.production_start(n_obins)
    if lng is not None:
        v = lng(gpu.get("lng"))
        gpu.set("lng", v)
        orc.set_lng(v)
    gpu.production_run(rounds)
    orc.production_run(rounds)
    assert np.array_equal(gpu.heo(), orc.heo())
    a, b = gpu_state(gpu), oracle_state(orc)
    if lng is not None:  # (ln g itself may hold NaN)
        assert np.array_equal(a.pop("lng"), b.pop("lng"))
    assert not differing(a, b)


@pytest.mark.parametrize("q,L,h,m,K,n_obins,bits", [
    (2, 3, 1, 1, 1, 1, 8), (2, 4, 1, 3, 33, 9, 4), (10, 12, 3, 2, 1000, 1, 4), (10, 12, 3, 2, 1000, 130, 8),
    (30, 9, 2, 2, 777, 50, 8), (200, 9, 2, 1, 300, 20, 8), (10, 33, 4, 3, 1000, 7, 4),
    (10, 184, 64, 1, 200, 64, 4),  # the lattice stays in global memory
])
def test_sizes(q, L, h, m, K, n_obins, bits):
    compare((q, L, h, 0.75, m, 1e-6, 0.8, K, 3), bits, n_obins)


@pytest.mark.parametrize("name,lng", [
    ("shape", lambda g: 30.0 * np.sin(np.arange(g.shape[1]) / 9.0) + 0 * g),             # both signs
    ("far", lambda g: 1e9 + 20.0 * np.sin(np.arange(g.shape[1]) / 9.0) + 0 * g),
    ("flat", lambda g: -7.25 + 0 * g),
    ("small", lambda g: 1e-12 * np.arange(g.shape[1]) + 0 * g),
    ("wide", lambda g: 1e25 * np.cos(np.arange(g.shape[1])) + 0 * g),
    ("wider", lambda g: 1e150 * np.cos(np.arange(g.shape[1])) + 0 * g),
])
def test_values_of_ln_g(name, lng):
    with np.errstate(invalid="ignore"):
        compare((5, 10, 2, 0.75, 2, 1e-6, 0.8, 500, 19), 4, 11, lng)


@pytest.mark.parametrize("bad", [np.nan, -np.inf, np.inf])
def test_ln_g_that_is_no_number(bad):
    """accept iff D >= 0 or u < exp(D) under IEEE comparisons (a NaN accepts nothing)"""
    q, L, K, seed, N = 5, 10, 60, 19, 100
    gpu = REWL(q, L, 1, 0.75, 2, 1e-6, 0.8, K, seed)
    gpu.run(2)
    gpu.production_start(11)
    lng = gpu.get("lng")
    lng[:, np.arange(lng.shape[1]) % 5 == 0] = bad
    gpu.set("lng", lng)
    spins, energy, t0 = gpu.get("spins"), gpu.get("energy"), int(gpu.get("steps")[0])
    for g in range(2):
        s, E = spins[g], int(energy[g])
        for t in range(t0, t0 + K):
            r = [int(x) for x in O.philox4x32_10([t, 0, g, 0], [seed, 0])]
            site, v = (r[0] * N) >> 32, (r[1] * (q - 1)) >> 32
            nw, (y, x) = v + (v >= s[site]), divmod(site, L)
            near = s[[y * L + (x + 1) % L, y * L + (x - 1) % L, (y + 1) % L * L + x, (y - 1) % L * L + x]]
            to = E + int((near == s[site]).sum()) - int((near == nw).sum())
            if -2 * N <= to <= 0:
                u = (((r[2] >> 5) << 26) | (r[3] >> 6)) * 2.0**-53
                with np.errstate(invalid="ignore", over="ignore"):
                    d = lng[g, E + 2 * N] - lng[g, to + 2 * N]
                    if d >= 0 or u < np.exp(d):
                        s[site], E = nw, to
        energy[g] = E
    gpu.production_run(1)
    assert np.array_equal(gpu.get("energy"), energy) and np.array_equal(gpu.get("spins"), spins)
    assert int(gpu.heo().sum()) == 2 * K


@pytest.mark.parametrize("L,h,m", [(10, 8, 64), (12, 40, 256)])  # lane groups; a thread per walker is the faster form
def test_many_walkers_of_many_values(L, h, m):
    compare((255, L, h, 0.75, m, 1e-6, 0.8, 40, 7), 8, 13, rounds=2, wl=1)
