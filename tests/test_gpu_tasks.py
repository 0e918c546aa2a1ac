"""The task streams of the triangular solves (blocked and level by level) against dense
triangular solves with the engine's own factors, at the edges of their layout: systems
smaller than a block, last blocks of one row and of a few, block sizes from 16 to 128 rows,
CTAs of 2 to 8 warps, two tasks in flight instead of four, and the chunk streams that serve
what the tasks do not.

Tolerance: with B the rows of a block, an explicit inverse of a diagonal block multiplies the
rounding of substitution by at most its row sums, a few tens here; 64 rounding errors of a
row of at most 128 terms at growth 16 give 1e5 eps relative to the largest entry of the
result (2e-11 FP64, 6e-3 FP32).  The bounds below, 1e-12 and 1e-5, are those of the existing
apply tests."""
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


CASES = [  # K, lattice, walkers, parameters
    (3, 0, 1, {}),                                       # 27 rows: one short block
    (5, 0, 1, {}),                                       # 125 = 64 + 61
    (4, 0, 1, dict(trisolve_group=2)),                   # 64 = 4 x 16
    (6, 0, 1, dict(trisolve_group=3)),                   # 216 = 9 x 24
    (6, 0, 1, dict(trisolve_group=64)),                  # blocks of 128 rows
    (9, 0, 1, {}),                                       # 729 = 11 x 64 + 25
    (4, 1, 1, dict(lfil_extra=0)),                       # bcc, 128 rows, factors without fill
    (6, 0, 1, dict(block_threads=64)),                   # two warps
    (7, 0, 1, dict(block_threads=160, lfil_extra=40)),   # five warps, long rows
    (6, 0, 1, dict(trisolve_group=1)),                   # a step per level
    (7, 0, 1, dict(trisolve_group=0, block_threads=96)),
    (6, 0, 1, dict(trisolve_group=1, trisolve_warp_rows=8)),  # chunk streams
    (6, 0, 1, dict(trisolve=1)),                         # synchronisation-free
    (8, 0, 160, {}),                                     # two CTAs an SM
    (16, 0, 1, dict(lfil_extra=4)),                      # 4096 rows: larger blocks
]


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("K,lat,walkers,kw", CASES)
def test_apply_matches_dense_solves(vmc, prec, K, lat, walkers, kw):
    a, kappa, rc = (1.0, 2.0, 1.45) if lat == 0 else (2.031, 1.0, 3.39)
    s = O.system(K, lat, a, kappa, rc)
    R = O.initial_positions(s, 5, 0.2 * a)
    n = len(R)
    ctx = vmc.vmc_create([(K, lat, a, kappa, rc)] * walkers, vmc.params(precision=prec, **kw))
    try:
        vmc.vmc_set_positions(ctx, walkers - 1, R)
        L, U, perm = vmc.vmc_get_factors(ctx, walkers - 1)
        st = vmc.vmc_get_stats(ctx, walkers - 1)
        v = np.random.default_rng(K).standard_normal(n)
        z = vmc.vmc_apply_preconditioner(ctx, walkers - 1, v)
    finally:
        vmc.vmc_destroy(ctx)
    ref = np.zeros(n)
    ref[perm] = np.linalg.solve(U, np.linalg.solve(L, v))
    tol = 1e-12 if prec == 0 else 1e-5
    assert np.abs(z - ref).max() <= tol * np.abs(ref).max()
    if kw.get("trisolve_group", 8) > 1 and "trisolve" not in kw:
        assert st["groups_L"] <= 2 * -(-n // 16) and st["groups_U"] <= 2 * -(-n // 16)
    else:
        assert st["groups_L"] == st["levels_L"] and st["groups_U"] == st["levels_U"]


def test_more_walker_pairs_than_sms(vmc):
    """Background refactorisation asked for with more pairs than SMs (two CTAs an SM, two
    tasks or more a warp in half an SM's shared memory): the first moves of two walkers against
    the oracle's chains."""
    K, walkers, moves = 5, 160, 40
    seeds = list(range(1, walkers + 1))
    ctx = vmc.vmc_create([(K, 0, 1.0, 2.0, 1.5)] * walkers,
                         vmc.params(precision=1, refactor_lag=4, max_updates=8, sweep_moves=moves))
    try:
        vmc.vmc_init_positions(ctx, seeds, 0.1)
        acc, rat = vmc.vmc_sweep(ctx, 1, 0.2, seeds)
        st = vmc.vmc_get_stats(ctx, walkers - 1)
    finally:
        vmc.vmc_destroy(ctx)
    assert st["async_lag"] == 4 and st["refactors_async"] > 0
    s = O.system(K)
    for w in (0, walkers - 1):
        R0 = O.initial_positions(s, seeds[w], 0.1)
        _, r_ref, a_ref, _ = O.chain(s, seeds[w], 0.2, R0, 1, max_steps=moves, solver=O.SOLVER_SHERMAN_MORRISON)
        lo = w * K ** 3
        assert np.array_equal(acc[lo:lo + moves], a_ref[:moves])
        assert np.all(np.abs(rat[lo:lo + moves] - r_ref[:moves]) <= 1e-10 * np.maximum(np.abs(r_ref[:moves]), 1e-3))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("K,kw,B", [
    (13, {}, 128),                                      # 2197 = 17 x 128 + 21
    (13, dict(lfil_extra=0), 128),                      # shortest factor rows
    (13, dict(lfil_extra=0, trisolve_row_cap=64), 64),  # a caller's cap bounds the blocks
    (12, {}, 64),                                       # 1728: below the line
])
def test_rows_of_a_block(vmc, prec, K, kw, B):
    """The blocks have their full rows whatever the fill limit, and the streams hold them
    (the level-by-level fallback would take a step per level)."""
    from scipy.linalg import solve_triangular
    s = O.system(K, 0, 1.0, 2.0, 1.45)
    n = K ** 3
    ctx = vmc.vmc_create([(K, 0, 1.0, 2.0, 1.45)], vmc.params(precision=prec, **kw))
    try:
        vmc.vmc_set_positions(ctx, 0, O.initial_positions(s, 5, 0.2))
        L, U, perm = vmc.vmc_get_factors(ctx, 0)
        st = vmc.vmc_get_stats(ctx, 0)
        v = np.random.default_rng(K).standard_normal(n)
        z = vmc.vmc_apply_preconditioner(ctx, 0, v)
    finally:
        vmc.vmc_destroy(ctx)
    ref = np.zeros(n)
    ref[perm] = solve_triangular(U, solve_triangular(L, v, lower=True))  # substitution: the factors may be near singular
    assert np.abs(z - ref).max() <= (1e-12 if prec == 0 else 1e-5) * np.abs(ref).max()
    nb = -(-n // B)
    assert nb <= st["groups_U"] <= 2 * nb and st["groups_L"] <= 2 * nb
