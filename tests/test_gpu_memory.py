"""Device memory of a context: the update lists are as long as the chain that the caller asks
for.  A list entry is a column and a value, 512 entries an update (12 bytes each in FP64), so
walkers of 27 particles with 4 updates hold 24 KB of them, beside 128 KB for the inverse of the
chain's matrix and about 100 KB of everything else; lists for 128 updates would be 768 KB."""
import pytest

pytestmark = pytest.mark.gpu


def test_short_chains_take_short_lists():
    import torch

    from paper_1008_5113_gb300.build import build_library

    build_library()
    from paper_1008_5113_gb300 import vmc

    walkers = 2000
    torch.cuda.synchronize()
    free0 = torch.cuda.mem_get_info()[0]
    ctx = vmc.vmc_create([(3, 0, 1.0, 2.0, 1.45)] * walkers, vmc.params(precision=0, max_updates=4, refactor_lag=0))
    used = free0 - torch.cuda.mem_get_info()[0]
    vmc.vmc_destroy(ctx)
    assert used / walkers < 400e3


def test_a_device_with_little_room_left():
    """Where the whole workspace does not fit the memory that is free, a context does without the
    parts that no result needs (transposed copies, room for full blocks): 96 walkers of 2744
    particles without fill, on what is left beside another allocation.  The ratios are those of
    the whole workspace to the parity tests' 1e-10."""
    import numpy as np
    import torch

    from paper_1008_5113_gb300 import vmc

    walkers, K, MB = 96, 14, 1 << 20
    systems = [(K, 0, 1.0, 2.0, 1.45)] * walkers
    seeds = list(range(1, walkers + 1))

    def room():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    def ratios(ctx):
        vmc.vmc_init_positions(ctx, seeds, 0.1)
        r = vmc.vmc_get_positions(ctx, walkers - 1)[5] + 0.1
        return np.array([vmc.vmc_ratio(ctx, w, 5, r) for w in (0, walkers - 1)])

    def create():
        return vmc.vmc_create(systems, vmc.params(precision=1, lfil_extra=0, refactor_lag=0))

    before = room()
    ctx = create()
    whole = before - room()
    want = ratios(ctx)
    vmc.vmc_destroy(ctx)
    hold = torch.empty(before - whole + 64 * MB, dtype=torch.uint8, device="cuda")  # 64 MB too little
    try:
        before = room()
        assert before < whole
        ctx = create()
        lean = before - room()
        got = ratios(ctx)
        vmc.vmc_destroy(ctx)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert lean < 0.8 * whole
    assert np.all(np.abs(got - want) <= 1e-10 * np.maximum(np.abs(want), 1e-3))
