"""Contexts of different sizes driven by different host threads on one device: every launch finds
room for its shared memory, whichever thread launched last."""
import ctypes as C
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vmc():
    import torch

    assert torch.cuda.is_available()
    from paper_1008_5113_gb300.build import build_library

    build_library()
    from paper_1008_5113_gb300 import vmc as v

    return v


def _drive_all(vmc, ctxs, call):
    import torch

    bad = []

    def drive(ctx):
        for _ in range(1500):
            st = call(ctx)
            if st != 0:
                bad.append((st, vmc.vmc_last_error(ctx)))
                return

    threads = [threading.Thread(target=drive, args=(c,)) for c in ctxs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for ctx in ctxs:
        vmc.vmc_destroy(ctx)
    assert not bad


def test_dense_contexts_of_several_sizes(vmc):
    """Walkers whose matrix is singular make no moves, so the launches are short and many."""
    import torch

    ctxs = []
    for K in (7, 8, 9):
        ctxs.append(vmc.vmc_create([(K, 0, 1.0, 2.0, 1.5)], vmc.params(precision=0, engine=vmc.ENGINE_DENSE_SM),
                                   stream=torch.cuda.Stream()))
        with pytest.raises(vmc.VmcError) as e:
            vmc.vmc_set_positions(ctxs[-1], 0, np.full((K ** 3, 3), 0.5 * K))  # most orbitals out of reach
        assert e.value.status == 5
    seeds = torch.zeros(1, dtype=torch.int64, device="cuda")
    torch.cuda.synchronize()
    _drive_all(vmc, ctxs, lambda ctx: vmc.lib().vmc_sweep_async(ctx, 1, 0.1, C.c_void_p(seeds.data_ptr()), None, None))


@pytest.mark.parametrize("prec", [0, 1])
def test_sparse_contexts_with_one_and_two_walkers_an_sm(vmc, prec):
    import torch

    ctxs = []
    for walkers in (1, 160, 2):
        ctxs.append(vmc.vmc_create([(4, 0, 1.0, 2.0, 1.5)] * walkers, vmc.params(precision=prec),
                                   stream=torch.cuda.Stream()))
        vmc.vmc_init_positions(ctxs[-1], list(range(1, walkers + 1)), 0.1)
    _drive_all(vmc, ctxs, lambda ctx: vmc.lib().vmc_kernel_bench(ctx, 1, 1))
