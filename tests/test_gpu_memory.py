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
