"""The dense engine with its rows split over clusters of 8, 4, 2 and 1 CTAs (by the number of
walkers) against the oracle's Sherman-Morrison chains: two sweeps, with the fresh inverse
between them, at sizes that the cluster and the warps do not divide; and the same walker gives
the same log, bit for bit, whatever the split."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def vmc():
    import torch

    assert torch.cuda.is_available()
    from paper_1008_5113_gb300.build import build_library

    build_library()
    O.build()
    from paper_1008_5113_gb300 import vmc as v

    return v


def _sweeps(vmc, K, walkers, threads=0):
    ctx = vmc.vmc_create([(K, 0, 1.0, 2.0, 1.5)] * walkers,
                         vmc.params(precision=0, engine=vmc.ENGINE_DENSE_SM, block_threads=threads))
    try:
        vmc.vmc_init_positions(ctx, list(range(1, walkers + 1)), 0.1)
        acc, rat = vmc.vmc_sweep(ctx, 2, 0.2, list(range(1, walkers + 1)))
        return acc.reshape(walkers, -1), rat.reshape(walkers, -1), vmc.vmc_get_positions(ctx, walkers - 1)
    finally:
        vmc.vmc_destroy(ctx)


@pytest.mark.parametrize("K,walkers,threads", [(4, 1, 0), (5, 19, 0), (5, 38, 64), (6, 76, 0), (5, 77, 0), (7, 3, 160)])
def test_split_inverse_matches_oracle(vmc, K, walkers, threads):
    acc, rat, pos = _sweeps(vmc, K, walkers, threads)
    s = O.system(K)
    for w in (0, walkers - 1):
        R0 = O.initial_positions(s, w + 1, 0.1)
        R, r_ref, a_ref, u_ref = O.chain(s, w + 1, 0.2, R0, 2, solver=O.SOLVER_SHERMAN_MORRISON)
        bad = np.nonzero(acc[w] != a_ref)[0]
        upto = int(bad[0]) if len(bad) else len(a_ref)
        if upto < len(a_ref):
            assert abs(r_ref[upto] ** 2 - u_ref[upto]) < 1e-9
        assert upto > len(a_ref) // 2
        lim = np.where(np.abs(r_ref[:upto]) >= 1e-3, 1e-10 * np.abs(r_ref[:upto]), 1e-13)
        assert np.all(np.abs(rat[w][:upto] - r_ref[:upto]) <= lim)
        if w == walkers - 1 and upto == len(a_ref):
            assert np.abs(pos - R).max() < 1e-12


def test_the_split_does_not_change_the_results(vmc):
    logs = [_sweeps(vmc, 5, walkers)[1][0] for walkers in (1, 20, 40, 100)]
    for r in logs[1:]:
        assert np.array_equal(logs[0].view(np.uint64), r.view(np.uint64))
