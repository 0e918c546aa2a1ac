"""Failures that the device reports instead of going on: a factorisation whose rows wait in vain
for one another records VMC_ERR_TIMEOUT in the walker's status and leaves the factors in use
alone, in every form of the triangular solves (the streams and level sets that incomplete rows
would give index out of their arrays), and the context stays usable."""
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


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("kw", [{}, dict(trisolve_group=1), dict(trisolve=1), dict(block_threads=64),
                                dict(engine=1, trisolve_group=1, trisolve_warp_rows=8)])
def test_lost_factorisation_is_reported(vmc, prec, kw):
    K, sigma = 6, 0.2
    s = O.system(K)
    R = O.initial_positions(s, 3, 0.2)
    r = R[7] + 0.1
    ctx = vmc.vmc_create([(K, 0, 1.0, 2.0, 1.5)] * 2, vmc.params(precision=prec, **kw))
    try:
        vmc.vmc_set_positions_all(ctx, [R, R])
        want = vmc.vmc_ratio(ctx, 0, 7, r)
        v = np.random.default_rng(1).standard_normal(K ** 3)
        made = vmc.vmc_get_stats(ctx, 0)["factorizations"]
        steps = [vmc.vmc_get_stats(ctx, 0)[f] for f in ("groups_L", "groups_U", "chunks_L", "chunks_U")]
        assert vmc.vmc_check_factor_timeout(ctx, 0) == 6
        st = vmc.vmc_get_stats(ctx, 0)
        assert st["status"] == 6 and st["factorizations"] == made + 1
        assert steps == [st[f] for f in ("groups_L", "groups_U", "chunks_L", "chunks_U")]  # the old streams
        assert vmc.vmc_get_stats(ctx, 1)["status"] == 0
        assert sorted(vmc.vmc_get_factors(ctx, 0)[2]) == list(range(K ** 3))
        with pytest.raises(vmc.VmcError) as e:  # no move is made with the factors
            vmc.vmc_sweep(ctx, 1, sigma, [1, 2])
        assert e.value.status == 6
        assert np.array_equal(vmc.vmc_get_positions(ctx, 0), R)
        vmc.vmc_set_positions_all(ctx, [R, R])
        assert vmc.vmc_get_stats(ctx, 0)["status"] == 0
        assert vmc.vmc_ratio(ctx, 0, 7, r) == want  # the same state, bit for bit
        z = [vmc.vmc_apply_preconditioner(ctx, w, v) for w in (0, 1)]
        assert np.array_equal(z[0], z[1])
        acc, rat = vmc.vmc_sweep(ctx, 1, sigma, [1, 2])
        assert np.all(np.isfinite(rat))
    finally:
        vmc.vmc_destroy(ctx)


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("K,lat,kw", [(6, 0, {}), (11, 0, dict(lfil_extra=16)), (5, 1, dict(block_threads=64))])
def test_ilutp_variants(vmc, prec, K, lat, kw):
    """Variants 1 and 2 have one row in flight, so no wait that could run out; their factors are
    those of the rows in flight, bit for bit."""
    sysd = (K, 0, 1.0, 2.0, 1.45) if lat == 0 else (K, 1, 2.031, 1.0, 3.39)
    R = O.initial_positions(O.system(*sysd), 5, 0.25 * sysd[2])
    out = []
    for variant, status in ((0, 6), (1, 0), (2, 0)):
        ctx = vmc.vmc_create([sysd], vmc.params(precision=prec, ilutp_variant=variant, **kw))
        try:
            vmc.vmc_set_positions(ctx, 0, R)
            out.append([x.tobytes() for x in vmc.vmc_get_factors(ctx, 0)])
            assert vmc.vmc_check_factor_timeout(ctx, 0) == status
        finally:
            vmc.vmc_destroy(ctx)
    assert out[0] == out[1] == out[2]
