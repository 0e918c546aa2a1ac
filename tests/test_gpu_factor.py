"""The reordering's cell search and the ILUTP with rows in flight against their definitions.

- Reordering: the pairing equals the oracle's literal greedy rule, exactly, on lattices too
  small for any cell search, on both lattices, for electrons near their sites, far from them,
  anywhere in the box and in one corner of it (most searches then end in a scan).
- ILUTP: the factors of the rows-in-flight variant equal, bit for bit, those of the one-warp
  hashed variant, which keeps its row by label and finishes a row before the next: sizes with
  one and several warps' rows per SM, values beyond a warp's shared part (n > 1024), exact LU,
  no fill, heavy fill, and every precision."""
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


def _system(K, lat):
    return (K, lat, 1.0, 2.0, 1.45) if lat == 0 else (K, lat, 2.031, 1.0, 3.39)


def _positions(s, sysd, how):
    K, _, a = sysd[:3]
    n = O.sites(s).shape[0]
    rng = np.random.default_rng(K)
    if how == "anywhere":
        return rng.uniform(0, K * a, (n, 3))
    if how == "corner":
        return rng.uniform(0, 0.6 * K * a, (n, 3))
    return O.initial_positions(s, 11, how * a)


@pytest.mark.parametrize("K,lat,how", [(3, 0, 0.3), (5, 0, 0.4), (7, 0, "anywhere"), (8, 0, "corner"), (12, 0, 0.25),
                                       (4, 1, 0.2), (5, 1, "anywhere"), (7, 1, 0.3), (16, 0, "anywhere")])
def test_reordering_is_the_greedy_rule(vmc, K, lat, how):
    sysd = _system(K, lat)
    s = O.system(*sysd)
    Z = O.sites(s)
    R = _positions(s, sysd, how)
    ctx = vmc.vmc_create([sysd], vmc.params(precision=1))
    try:
        try:
            vmc.vmc_set_positions(ctx, 0, R)
        except vmc.VmcError:
            pass  # such a matrix may break down: the pairing comes before the factorisation
        _, por, ooc = vmc.vmc_get_matrix(ctx, 0)
    finally:
        vmc.vmc_destroy(ctx)
    P, Q = O.greedy_pairing(s, R, Z, ooc.astype(np.int32), ooc.astype(np.int32))
    partner = np.empty(len(Z), dtype=np.int64)
    partner[Q] = P
    assert np.array_equal(por, partner[ooc])


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("K,lat,walkers,kw", [
    (3, 0, 1, dict(drop_tol=0.0, lfil_extra=27)),
    (4, 0, 1, dict(block_threads=64)),
    (6, 0, 160, {}),
    (7, 0, 1, dict(lfil_extra=0)),
    (5, 1, 2, dict(drop_tol=0.01, permtol=0.05)),
    (9, 0, 1, dict(lfil_extra=60, drop_tol=1e-6)),
    (11, 0, 1, dict(lfil_extra=32)),
])
def test_rows_in_flight_give_the_one_warp_factors(vmc, prec, K, lat, walkers, kw):
    sysd = _system(K, lat)
    s = O.system(*sysd)
    R = O.initial_positions(s, 5, 0.25 * sysd[2])
    out = []
    for variant in (0, 2):
        ctx = vmc.vmc_create([sysd] * walkers, vmc.params(precision=prec, ilutp_variant=variant, **kw))
        try:
            vmc.vmc_set_positions(ctx, walkers - 1, R)
            st = vmc.vmc_get_stats(ctx, walkers - 1)
            out.append(vmc.vmc_get_factors(ctx, walkers - 1) + (st["pivots"], st["nnz_LU"], st["levels_L"],
                                                                st["levels_U"], st["ilu_elims"], st["ilu_cand"]))
        finally:
            vmc.vmc_destroy(ctx)
    a, b = out
    assert np.array_equal(a[2], b[2]) and a[3:] == b[3:]
    assert np.array_equal(a[0].view(np.uint64), b[0].view(np.uint64))
    assert np.array_equal(a[1].view(np.uint64), b[1].view(np.uint64))
