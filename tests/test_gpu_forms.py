"""Each form of a computation is the one that runs where it is meant to, and gives what it should:
- level-by-level task streams take a step for every 128 rows of a level (the chunk streams report
  chunks of several levels instead);
- the dense engine's flat form, which serves systems whose vectors do not fit shared memory,
  gives the split form's logs bit for bit;
- the products with A from the slots themselves, for an allocation-free call whose workspace has
  no room for the transposed copy, give the ratio of a context."""
import ctypes as C

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


def _level_sizes(M, upper):
    """Rows a level of the solve with M (strict triangle)."""
    n = len(M)
    lev = np.zeros(n, dtype=int)
    for r in range(n - 1, -1, -1) if upper else range(n):
        c = np.nonzero(M[r, r + 1:])[0] + r + 1 if upper else np.nonzero(M[r, :r])[0]
        lev[r] = lev[c].max() + 1 if len(c) else 0
    return np.bincount(lev)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("K,threads,kw", [(6, 0, {}), (12, 0, {}), (11, 64, dict(lfil_extra=0))])
def test_level_tasks_take_a_step_per_128_rows(vmc, prec, K, threads, kw):
    s = O.system(K, 0, 1.0, 2.0, 1.45)
    ctx = vmc.vmc_create([(K, 0, 1.0, 2.0, 1.45)],
                         vmc.params(precision=prec, trisolve_group=1, block_threads=threads, **kw))
    try:
        vmc.vmc_set_positions(ctx, 0, O.initial_positions(s, 5, 0.2))
        L, U, _ = vmc.vmc_get_factors(ctx, 0)
        st = vmc.vmc_get_stats(ctx, 0)
    finally:
        vmc.vmc_destroy(ctx)
    for M, upper, side in ((L, False, "L"), (U, True, "U")):
        rows = _level_sizes(M, upper)
        assert st["levels_" + side] == len(rows)
        assert st["chunks_" + side] == int((-(-rows // 128)).sum())


@pytest.mark.parametrize("prec", [0, 1])
def test_warp_rows_leave_blocked_solves_alone(vmc, prec):
    """trisolve_warp_rows is for level-by-level solves: with blocks the steps and the apply are
    the same, bit for bit."""
    s = O.system(7, 0, 1.0, 2.0, 1.45)
    v = np.random.default_rng(3).standard_normal(343)
    out = []
    for rows in (0, 8, 32):
        ctx = vmc.vmc_create([(7, 0, 1.0, 2.0, 1.45)], vmc.params(precision=prec, trisolve_warp_rows=rows))
        try:
            vmc.vmc_set_positions(ctx, 0, O.initial_positions(s, 5, 0.2))
            st = vmc.vmc_get_stats(ctx, 0)
            out.append((st["groups_L"], st["groups_U"], vmc.vmc_apply_preconditioner(ctx, 0, v).tobytes()))
        finally:
            vmc.vmc_destroy(ctx)
    assert out[0][0] <= 12 and out[0] == out[1] == out[2]


@pytest.mark.parametrize("K,threads", [(4, 0), (5, 64), (6, 96), (7, 0)])
def test_dense_kernels_agree(vmc, K, threads):
    """The dense kernels for rows split over a cluster and not, for long rows and for short rows or
    more than two walkers an SM: the same walker's log and positions, bit for bit."""
    out = []
    for walkers in (1, 160, 310):
        ctx = vmc.vmc_create([(K, 0, 1.0, 2.0, 1.5)] * walkers,
                             vmc.params(precision=0, engine=vmc.ENGINE_DENSE_SM, block_threads=threads))
        try:
            vmc.vmc_init_positions(ctx, [5] * walkers, 0.1)
            acc, rat = vmc.vmc_sweep(ctx, 2, 0.2, [7] * walkers)
            out.append([(a.tobytes(), r.tobytes(), vmc.vmc_get_positions(ctx, w).tobytes())
                        for w, (a, r) in enumerate(zip(acc.reshape(walkers, -1), rat.reshape(walkers, -1)))])
        finally:
            vmc.vmc_destroy(ctx)
    assert all(x == out[0][0] for o in out for x in o)


def test_flat_dense_form_gives_the_split_forms_logs(vmc):
    """A context with one walker too large for the split form takes the flat form for all of
    them.  That walker's matrix is singular (no particle near its first site), so it is given up
    at once and only the small walkers move."""
    import torch

    small, seeds = [3, 5], [11, 12, 13]
    R = [O.initial_positions(O.system(K), 3, 0.1) for K in small]
    n = [K ** 3 for K in small]

    def logs(Ks):
        ctx = vmc.vmc_create([(K, 0, 1.0, 2.0, 1.45) for K in Ks],
                             vmc.params(precision=0, engine=vmc.ENGINE_DENSE_SM, sm_refresh=1))
        try:
            for w, x in enumerate(R):
                vmc.vmc_set_positions(ctx, w, x)
            if len(Ks) > len(small):
                with pytest.raises(vmc.VmcError) as e:
                    vmc.vmc_set_positions(ctx, len(small), np.full((Ks[-1] ** 3, 3), 0.5 * Ks[-1]))
                assert e.value.status == 5
            total = sum(K ** 3 for K in Ks)
            sd = torch.as_tensor(seeds[:len(Ks)], dtype=torch.int64, device="cuda")
            rat = torch.zeros(2 * total, dtype=torch.float64, device="cuda")
            acc = torch.zeros(2 * total, dtype=torch.uint8, device="cuda")
            vmc.vmc_sweep_async(ctx, 2, 0.2, sd, acc, rat)
            torch.cuda.synchronize()
            m = 2 * sum(n)  # walker-major: the small walkers' entries come first
            return (acc[:m].cpu().numpy(), rat[:m].cpu().numpy(),
                    [vmc.vmc_get_positions(ctx, w) for w in range(len(small))])
        finally:
            vmc.vmc_destroy(ctx)

    split, flat = logs(small), logs(small + [19])  # 28 bytes x 6859 > the shared memory of an SM
    assert split[0].sum() > 50
    assert np.array_equal(split[0], flat[0])
    assert np.array_equal(split[1].view(np.uint64), flat[1].view(np.uint64))
    for a, b in zip(split[2], flat[2]):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", [0, 1])
def test_allocation_free_call_without_the_transposed_copy(vmc, prec):
    """The largest fill limit that the fixed workspace takes at n = 1000: there is no room for
    the copy of the slots beside it.  Both sides are solved to 1e-12; the bar is the parity
    tests' 1e-10."""
    import torch

    K, k = 10, 321
    sysd = (K, 0, 1.0, 2.0, 1.5)
    s = O.system(*sysd)
    R = O.initial_positions(s, 9, 0.2)
    r = R[k] + np.array([0.1, -0.2, 0.15])
    xyz = torch.as_tensor(R, device="cuda").contiguous()
    out = torch.zeros(1, dtype=torch.float64, device="cuda")
    lfil = None
    for cand in range(400, 20, -4):
        try:
            vmc.vmc_ratio_noalloc(sysd, vmc.params(precision=prec, lfil_extra=cand, gmres_m=40), xyz, k, r, out)
            lfil = cand
            break
        except vmc.VmcError as e:
            assert e.status in (1, 8)  # rows too long for a slot; workspace too large
    assert lfil is not None
    ctx = vmc.vmc_create([sysd], vmc.params(precision=prec, lfil_extra=lfil, gmres_m=40))
    try:
        vmc.vmc_set_positions(ctx, 0, R)
        want = vmc.vmc_ratio(ctx, 0, k, r)
    finally:
        vmc.vmc_destroy(ctx)
    assert abs(out.item() - want) <= 1e-10 * max(abs(want), 1e-3)
