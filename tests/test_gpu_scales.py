"""The reordering's cell search compares distances in FP32: its pairing is the oracle's greedy
rule, exactly, whatever the unit of length (lattice constants whose squares FP32 does not hold
among them), and positions outside the box, which only the allocation-free call is given
unwrapped, reach the ratio of the same positions inside it."""
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


@pytest.mark.parametrize("a", [1.0, 3e-10, 1e-25, 1e25])
@pytest.mark.parametrize("K,lat", [(3, 0), (8, 0), (12, 0), (5, 1), (7, 1)])
def test_pairing_in_any_unit_of_length(vmc, a, K, lat):
    sysd = (K, 0, a, 2.0 / a ** 2, 1.45 * a) if lat == 0 else (K, 1, a, 4.0 / a ** 2, 1.6 * a)
    s = O.system(*sysd)
    Z = O.sites(s)
    R = np.random.default_rng(K).uniform(0, K, (len(Z), 3)) * a * (1 - 1e-12)
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


@pytest.mark.parametrize("prec", [0, 1])
def test_positions_outside_the_box(vmc, prec):
    import torch

    K = 7
    sysd = (K, 0, 1.0, 2.0, 1.5)
    s = O.system(*sysd)
    R = O.initial_positions(s, 4, 0.2)
    shift = K * np.random.default_rng(2).integers(-3, 4, R.shape)
    shift[::2] = 0
    r = R[11] + 0.15
    got = []
    for x in (R, R + shift):
        xyz = torch.as_tensor(x, device="cuda").contiguous()
        out = torch.zeros(1, dtype=torch.float64, device="cuda")
        vmc.vmc_ratio_noalloc(sysd, vmc.params(precision=prec), xyz, 11, r, out)
        got.append(out.item())
    # positions rounded at |x| <= 4 K: 3e-15 each, on a ratio whose solve is good to 1e-12
    assert abs(got[1] - got[0]) <= 1e-11 * max(1.0, abs(got[0]))
