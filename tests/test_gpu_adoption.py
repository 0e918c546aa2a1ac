"""A factor set that a launch finished but did not adopt is adopted by the next launch, whatever
calls lengthened the update chain in between: with more kept updates than the CTA has threads,
the adopted chain still belongs to its factors."""
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


@pytest.mark.parametrize("threads", [64, 96, 256])
def test_adoption_of_a_chain_longer_than_the_cta(vmc, threads):
    """Complete factors (no dropping, room for all fill): A M = I as long as the chain goes with
    them.  Tolerance: rounding grows by the condition number of A (below 1e3 here) and by a
    factor of at most 1 + |u||z_hat| (a few) for the updates that act on one element: 1e-16 to
    1e-12; 1e-8 is far from both that and from a chain with a wrong u list (order 1)."""
    K, lag = 4, 4
    s = O.system(K, 0, 1.0, 2.0, 1.45)
    n = K ** 3
    rng = np.random.default_rng(5)
    ctx = vmc.vmc_create([(K, 0, 1.0, 2.0, 1.45)],
                         vmc.params(precision=0, block_threads=threads, refactor_lag=lag, max_updates=128,
                                    drop_tol=0.0, lfil_extra=n))
    try:
        vmc.vmc_set_positions(ctx, 0, O.initial_positions(s, 1, 0.1))
        while vmc.vmc_get_stats(ctx, 0)["n_updates"] < lag + 1:  # the set of the snapshot at `lag` is ready
            vmc.vmc_advance(ctx, 1, 0.1, [7])
        assert vmc.vmc_get_stats(ctx, 0)["refactors_async"] == 0
        R = vmc.vmc_get_positions(ctx, 0)
        while vmc.vmc_get_stats(ctx, 0)["n_updates"] < 110:
            k = int(rng.integers(n))
            r = R[k] + 0.1 * rng.standard_normal(3)
            if abs(vmc.vmc_ratio(ctx, 0, k, r)) > 0.5:
                vmc.vmc_accept(ctx, 0)
                R[k] = r
        vmc.vmc_advance(ctx, 1, 0.1, [7])
        st = vmc.vmc_get_stats(ctx, 0)
        assert st["refactors_async"] == 1 and st["reorders"] == 0 and st["n_updates"] >= 110 - lag
        A, _, _ = vmc.vmc_get_matrix(ctx, 0)
        v = rng.standard_normal(n)
        z = vmc.vmc_apply_preconditioner(ctx, 0, v)
    finally:
        vmc.vmc_destroy(ctx)
    assert np.abs(A @ z - v).max() <= 1e-8 * np.abs(v).max()
