"""Windows whose H(E, O) has more than 2^31 entries: the run in every class must
be the run in few classes, spread out.  (17 GB and more of H(E, O): it stays on
the device, in memory of the caller's.)"""
import numpy as np
import pytest

from paper_1312_3004_gb300 import REWL
from paper_1312_3004_gb300.rewl import set_allocator

pytestmark = pytest.mark.gpu


def production(args, n_obins, rounds, lng):
    r = REWL(*args)
    r.production_start(n_obins)
    r.set("lng", lng(r))
    r.production_run(rounds)
    return r


@pytest.mark.parametrize("args,rounds,tilt", [
    ((10, 200, 1, 0.75, 1, 1e-6, 0.8, 3000, 3), 2, 0.0),   # a thread per walker; E about -N / 5: entries above 2^31
    ((255, 284, 6, 0.0, 1, 1e-6, 0.8, 300_000, 3), 2, 3.0),  # lane groups; ln g falls with E: the last window ends near E = 0
])
def test_entries_beyond_32_bits(args, rounds, tilt):
    import torch

    q, L, h = args[:3]
    N = L * L
    span = N - -(-N // q) + 1
    B = -(-2 * N // h) + 1 if h > 1 else 2 * N + 1
    assert B * span > 2**31
    if torch.cuda.mem_get_info()[0] < 1.3 * 8 * h * B * span:
        pytest.skip("not enough device memory")

    def lng(r):
        return -tilt * np.arange(r.B) * np.ones((r.G, 1))

    few = {n: production(args, n, rounds, lng) for n in (1, 16)}
    blocks = []

    def alloc(n):
        blocks.append(torch.empty(n, dtype=torch.uint8, device="cuda"))
        return blocks[-1].data_ptr()

    set_allocator(alloc)
    try:
        big = production(args, span, rounds, lng)
    finally:
        set_allocator()
    try:
        assert big.B == B
        heo = max(blocks, key=lambda b: b.numel())[:8 * h * B * span].view(torch.int64).view(h, B, span)
        top = torch.nonzero(heo[h - 1].sum(1)).max().item()
        assert top * span > 2**31  # (the run has been there)
        one, sixteen = few[1].heo().astype(np.int64), few[16].heo().astype(np.int64)
        assert np.array_equal(heo.sum(2).cpu().numpy(), one[:, :, 0])
        by_class = heo.sum(1).cpu().numpy()
        cls = np.arange(span) * 16 // span
        assert np.array_equal(np.stack([by_class[:, cls == c].sum(1) for c in range(16)], 1), sixteen.sum(1))
        for f in ("spins", "energy", "steps"):
            assert np.array_equal(big.get(f), few[1].get(f))
    finally:  # (the callbacks keep the list)
        big.close()
        blocks.clear()
        heo = None
        torch.cuda.empty_cache()
