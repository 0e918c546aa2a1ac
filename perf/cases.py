"""Performance cases: what a program that uses the engine has it do.

A case is one call pattern of the C ABI (through its binding ``vmc``) on walkers of one
size, or of several sizes:

* ``ratio``       single moves proposed by the caller: ``vmc_ratio_grad`` (ratio, drift,
                  Laplacian) on a walker that stays as it is;
* ``alloc_free``  ``vmc_ratio_noalloc``: set-up and one ratio of a new configuration;
* ``kinetic``     ``vmc_kinetic_energy``: one solve per particle of every walker;
* ``sweep``       a block of Metropolis moves from a saved configuration, as after a
                  checkpoint or a branching step: ``vmc_set_positions_all`` (rows,
                  reordering, factorisation), ``vmc_set_sweep_count``, ``vmc_sweep`` and
                  ``vmc_get_positions``, on any of the four engines.

The systems are those of ``paper_1008_5113_gb300.workloads``: the simple-cubic lattice
(a = 1, kappa = 2, r_c = 1.5) and the paper's body-centred one.  Chains start either from
the lattice sites plus the configured jitter ("sites": where every run begins) or from
configurations 20 sweeps into the chain ("equilibrated": where measurements are taken and
the matrices are hardest).  The equilibrated ones come from a plain dense chain in torch,
made once per lattice; a case's walkers are lattice translations of them drawn from the
seed, with Metropolis seeds of their own.
"""
from __future__ import annotations

import functools
import math
import random

import numpy as np
import torch

from paper_1008_5113_gb300 import vmc
from paper_1008_5113_gb300.workloads import BATCH_1000, PAPER_BCC, PAPER_SOLVER

EQUIL_SWEEPS = 20  # sweeps that the configurations are away from the lattice sites
BASE_WALKERS = 8   # independent equilibrated chains per lattice
PRECISIONS = {"fp64": vmc.PREC_FP64, "mixed": vmc.PREC_MIXED, "mixed_f32ilu": vmc.PREC_MIXED_F32ILU}
ENGINES = {"plain": vmc.ENGINE_PLAIN, "step": vmc.ENGINE_STEP, "persistent": vmc.ENGINE_PERSISTENT,
           "dense": vmc.ENGINE_DENSE_SM}


def _case(name, op, Ks, walkers, **kw):
    """Ks: lattice sizes as text ("8,10": `walkers` walkers of each)."""
    c = {"name": name, "op": op, "Ks": Ks, "lattice": "sc", "walkers": walkers, "precision": "mixed",
         "engine": "persistent", "start": "equilibrated", "moves": 0, "lfil": -1, "chain": -1, "lag": -1, "group": 8}
    c.update(kw)
    return c


def listed():
    return [
        # one proposal on one small walker: the latency of a single-move call
        _case("ratio_n216", "ratio", "6", 1, precision="fp64", moves=1),
        # proposals on one large walker early in its run, default solver
        _case("ratio_n4096", "ratio", "16", 1, start="sites", moves=4),
        # a caller that owns all memory: set-up and ratio of one configuration
        _case("alloc_free_n512", "alloc_free", "8", 1, moves=1),
        # the local-energy measurement between blocks of sweeps
        _case("kinetic_n343", "kinetic", "7", 12, lfil=32),
        # the plain reference path: one walker, one launch per move, a whole sweep
        _case("plain_n216_fp64", "sweep", "6", 1, precision="fp64", engine="plain"),
        # one launch per move for a batch, in-line refactorisation in FP32
        _case("step_n343_w96", "sweep", "7", 96, precision="mixed_f32ilu", engine="step", moves=48, lfil=16),
        # the configured batch, FP64: a CTA pair per walker, in the layout the autotuner picks
        _case("batch_n1000_w64_fp64", "sweep", "10", 64, precision="fp64", moves=48, lfil=32, chain=32, lag=16),
        # the same batch in mixed precision
        _case("batch_n1000_w64_mixed", "sweep", "10", 64, moves=80, lfil=32, chain=64, lag=32),
        # the paper's lattice and solver settings at its smallest size
        _case("paper_bcc_n686_w8", "sweep", "7", 8, lattice="bcc", moves=48),
        # two walker CTAs per SM, level-by-level solves, at the start of a run
        _case("batch_n4096_w256_mixed", "sweep", "16", 256, start="sites", moves=64, lfil=32, lag=0, group=1),
        # walkers of different sizes in one launch
        _case("uneven_w160_mixed", "sweep", "7,8,10,12,16", 32, start="sites", moves=80, lfil=32, group=1),
        # the standard algorithm: explicit inverse and Sherman-Morrison updates
        _case("dense_n729_w64_fp64", "sweep", "9", 64, precision="fp64", engine="dense"),
    ]


def draw(rng: random.Random):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("ratio", "ratio", "alloc_free", "kinetic", "plain", "step", "batch", "batch", "batch", "bcc",
                       "uneven", "dense"))
    prec = rng.choice(("fp64", "mixed", "mixed", "mixed_f32ilu"))
    if kind == "ratio":
        K = log_int(4, 15)
        c = _case("", "ratio", str(K), rng.randint(1, 3), precision=prec, moves=rng.randint(1, 4),
                  start="equilibrated" if K <= 10 else "sites", lfil=32 if K <= 10 else -1)
    elif kind == "alloc_free":
        c = _case("", "alloc_free", str(rng.randint(4, 9)), 1, precision=prec, moves=rng.randint(1, 2), lfil=24)
    elif kind == "kinetic":
        c = _case("", "kinetic", str(rng.randint(4, 7)), log_int(1, 40), precision=prec, lfil=32)
    elif kind == "plain":
        c = _case("", "sweep", str(rng.randint(5, 8)), 1, precision=prec, engine="plain", lfil=32,
                  moves=rng.randint(40, 120))
    elif kind == "step":
        c = _case("", "sweep", str(rng.randint(5, 9)), log_int(2, 100), precision=prec, engine="step", lfil=24,
                  moves=rng.randint(16, 48))
    elif kind == "bcc":
        c = _case("", "sweep", str(rng.randint(4, 7)), log_int(2, 60), precision=prec, lattice="bcc",
                  moves=rng.randint(16, 40), lag=rng.choice((-1, 0)))
    elif kind == "uneven":
        Ks = ",".join(str(K) for K in sorted(rng.sample(range(5, 15), 3)))
        c = _case("", "sweep", Ks, log_int(4, 60), precision=prec, start="sites", moves=rng.randint(8, 32), lfil=32,
                  group=rng.choice((1, 8)), lag=rng.choice((-1, 0)))
    elif kind == "dense":
        c = _case("", "sweep", str(rng.randint(5, 8)), log_int(1, 120), precision="fp64", engine="dense")
    else:
        K = log_int(5, 13)
        if K <= 10:
            c = _case("", "sweep", str(K), log_int(4, 120), precision=prec, moves=rng.randint(16, 48), lfil=32,
                      chain=rng.choice((16, 32, 64)), lag=rng.choice((-1, 0)))
        else:
            c = _case("", "sweep", str(K), log_int(16, 200), precision=prec, start="sites", moves=rng.randint(8, 24),
                      lfil=32, lag=rng.choice((-1, 0)), group=rng.choice((1, 8)))
    del c["name"]
    return c


# ---- systems and plain 64-bit mathematics (torch and numpy only) --------------------
def _wl(case):
    return PAPER_BCC if case["lattice"] == "bcc" else BATCH_1000


def _systems(case):
    w = _wl(case)
    return [(int(K), w.lattice, w.a, w.kappa, w.r_c) for K in case["Ks"].split(",") for _ in range(case["walkers"])]


def _n(system):
    return system[0] ** 3 * (2 if system[1] == 1 else 1)


def _row_entries(lattice):
    """Mean orbitals within r_c of a point: density times the ball's volume."""
    w = PAPER_BCC if lattice == "bcc" else BATCH_1000
    return (2 if lattice == "bcc" else 1) / w.a ** 3 * 4.0 / 3.0 * math.pi * w.r_c ** 3


def _sites(system):
    K, lat, a = system[:3]
    g = np.arange(K)
    z, y, x = np.meshgrid(g, g, g, indexing="ij")
    c = np.stack([x, y, z], -1).reshape(-1, 1, 3).astype(np.float64)
    off = np.array([0.0, 0.5]) if lat == 1 else np.array([0.0])
    return (a * (c + off[None, :, None])).reshape(-1, 3)


def _rows(system, R, Z=None):
    """Slater rows phi_j(r) of positions R (..., 3): (..., n), torch float64."""
    K, _, a, kappa, rc = system
    Z = torch.as_tensor(_sites(system), device=R.device) if Z is None else Z
    L = K * a
    d = R[..., None, :] - Z
    d = d - L * torch.round(d / L)
    d2 = (d * d).sum(-1)
    return torch.where(d2 <= rc * rc, torch.exp(-kappa * d2), torch.zeros_like(d2))


def _wrap(x, L):
    y = x - L * np.floor(x / L)
    return np.where(y >= L, y - L, y)


@functools.lru_cache(maxsize=None)
def _equilibrated(K, lattice):
    """BASE_WALKERS configurations after EQUIL_SWEEPS sweeps of Metropolis moves on
    |det A|^2: explicit inverses with Sherman-Morrison updates, fresh ones every sweep."""
    wl = PAPER_BCC if lattice == "bcc" else BATCH_1000
    system = (K, wl.lattice, wl.a, wl.kappa, wl.r_c)
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev).manual_seed(20 + 7 * K + wl.lattice)
    Z = torch.as_tensor(_sites(system), device=dev)
    n, L = Z.shape[0], K * wl.a
    rand = lambda *s: torch.randn(*s, generator=gen, device=dev, dtype=torch.float64)  # noqa: E731
    R = torch.remainder(Z + wl.jitter * rand(BASE_WALKERS, n, 3), L)
    for _ in range(EQUIL_SWEEPS):
        A = _rows(system, R, Z)
        B = torch.linalg.inv(A)
        new = torch.remainder(R + wl.sigma * rand(BASE_WALKERS, n, 3), L)
        u = _rows(system, new, Z) - A
        uni = torch.rand(BASE_WALKERS, n, generator=gen, device=dev, dtype=torch.float64)
        took = torch.zeros(BASE_WALKERS, n, dtype=torch.bool, device=dev)
        for k in range(n):
            col, uk = B[:, :, k], u[:, k]
            ratio = 1.0 + (uk * col).sum(1)
            acc = ratio * ratio > uni[:, k]
            took[:, k] = acc
            f = torch.where(acc, -1.0 / ratio, torch.zeros_like(ratio))
            B.baddbmm_((col * f[:, None])[:, :, None], torch.bmm(uk[:, None, :], B))
        R = torch.where(took[..., None], new, R)
    return R.cpu().numpy()


def _configurations(case, rng):
    """Every walker's start positions, in [0, L)."""
    wl = _wl(case)
    out = []
    for system in _systems(case):
        K, a = system[0], system[2]
        L, per = K * a, _n(system) // K ** 3
        if case["start"] == "sites":
            out.append(_wrap(_sites(system) + wl.jitter * rng.standard_normal((_n(system), 3)), L))
            continue
        base = _equilibrated(K, case["lattice"])
        t = rng.integers(0, K, 3)
        R = base[rng.integers(len(base))].reshape(K, K, K, per, 3)  # particles by home site (z, y, x)
        R = np.roll(R, (t[2], t[1], t[0]), (0, 1, 2)).reshape(-1, 3) + a * t
        out.append(_wrap(R, L))
    return out


def _inputs(case, seed):
    rng = np.random.default_rng([seed, 11])
    R = _configurations(case, rng)
    seeds = rng.integers(1, 1 << 62, len(R)).astype(np.uint64)
    return rng, R, seeds


def _proposals(case, rng, R):
    """Caller-proposed single moves: (walker, particle, new position)."""
    sigma = _wl(case).sigma
    out = []
    for w, r in enumerate(R):
        for k in rng.choice(len(r), size=max(1, case["moves"]), replace=False):
            out.append((w, int(k), r[k] + sigma * rng.standard_normal(3)))
    return out


# ---- the passes ---------------------------------------------------------------------
class _State:
    def __init__(self, case, ctx):
        self.case, self.ctx = case, ctx

    def __del__(self):
        if self.ctx is not None:
            vmc.vmc_destroy(self.ctx)


def _params(case):
    kw = dict(PAPER_SOLVER) if case["lattice"] == "bcc" else {}
    return vmc.params(precision=PRECISIONS[case["precision"]], engine=ENGINES[case["engine"]],
                      lfil_extra=case["lfil"], max_updates=case["chain"], refactor_lag=case["lag"],
                      trisolve_group=case["group"], sweep_moves=case["moves"] if case["op"] == "sweep" else 0, **kw)


def prepare(case, seed):
    rng, R, seeds = _inputs(case, seed)
    systems = _systems(case)
    if case["op"] == "alloc_free":
        s = _State(case, None)
        s.system, s.params = systems[0], _params(case)
        s.xyz = torch.as_tensor(R[0], device="cuda").contiguous()
        s.moves = _proposals(case, rng, R)
        s.out = torch.zeros(len(s.moves), dtype=torch.float64, device="cuda")
        return s
    s = _State(case, vmc.vmc_create(systems, _params(case), stream=torch.cuda.current_stream()))
    s.R, s.seeds = np.concatenate(R), seeds
    s.n = [_n(x) for x in systems]
    if case["op"] == "ratio":
        s.moves = _proposals(case, rng, R)
    if case["op"] != "sweep":
        vmc.vmc_set_positions_all(s.ctx, s.R)
    return s


def run(s):
    case, ctx = s.case, s.ctx
    if case["op"] == "ratio":
        got = [vmc.vmc_ratio_grad(ctx, w, k, r) for w, k, r in s.moves]
        return {"ratio": np.array([g[0] for g in got]), "grad": np.stack([g[1] for g in got]),
                "lap": np.array([g[2] for g in got])}
    if case["op"] == "alloc_free":
        for i, (_, k, r) in enumerate(s.moves):
            vmc.vmc_ratio_noalloc(s.system, s.params, s.xyz, k, r, s.out[i:i + 1])
        return s.out
    if case["op"] == "kinetic":
        return vmc.vmc_kinetic_energy(ctx, len(s.n))
    vmc.vmc_set_positions_all(ctx, s.R)
    vmc.vmc_set_sweep_count(ctx, EQUIL_SWEEPS)
    acc, rat = vmc.vmc_sweep(ctx, 1, _wl(case).sigma, s.seeds)
    made, lo = [], 0
    for n in s.n:  # the log entries of particles that were not moved are not written
        m = min(n, case["moves"]) if case["moves"] and case["engine"] != "dense" else n
        made.append(np.arange(lo, lo + m))
        lo += n
    made = np.concatenate(made)
    return {"accepted": acc[made], "ratio": rat[made],
            "positions": np.concatenate([vmc.vmc_get_positions(ctx, w) for w in range(len(s.n))])}


def work(case):
    """Bytes and operations of one pass that no implementation of the path avoids: each
    solve reads its sparse matrix once (12 bytes an entry) and writes its solution; a
    set-up reads the positions and writes the matrix and a factorisation with as many
    entries; the dense engine's update reads and writes the inverse."""
    z = _row_entries(case["lattice"])
    b = f = 0.0
    for system in _systems(case):
        n = _n(system)
        solve_b, solve_f = n * (12 * z + 8), 4 * n * z
        setup_b, setup_f = n * (24 + 24 * z), 12 * n * z
        m = case["moves"] or n
        if case["op"] == "ratio":
            b, f = b + m * solve_b, f + m * solve_f
        elif case["op"] == "alloc_free":
            b, f = b + m * (setup_b + solve_b), f + m * (setup_f + solve_f)
        elif case["op"] == "kinetic":
            b, f = b + n * solve_b, f + n * solve_f
        elif case["engine"] == "dense":  # about half of the moves are accepted
            b, f = b + 8 * n * n + 8.0 * n * n * n, f + 2.0 * n ** 3 + 1.0 * n ** 3
        else:
            b, f = b + setup_b + min(m, n) * solve_b, f + setup_f + min(m, n) * solve_f
    return {"bytes": b, "flops": f}


# ---- the same results in plain 64-bit arithmetic --------------------------------------
def _philox(ctr, key):
    """Philox4x32-10 (Salmon et al., SC'11) on uint64 arrays holding 32-bit words."""
    c = [np.asarray(x, np.uint64) for x in ctr]
    k0, k1 = (np.asarray(x, np.uint64) for x in key)
    m32 = np.uint64(0xFFFFFFFF)
    s32 = np.uint64(32)
    for r in range(10):
        if r:
            k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m32, (k1 + np.uint64(0xBB67AE85)) & m32
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> s32) ^ c[1] ^ k0, p1 & m32, (p0 >> s32) ^ c[3] ^ k1, p0 & m32]
    return c


def _u01(hi, lo):
    return (((hi << np.uint64(32)) | lo) >> np.uint64(12)).astype(np.float64) * 2.0 ** -52 + 2.0 ** -53


def _metropolis_draws(seed, sweep, m):
    """Normals (m, 3) and acceptance uniforms (m,) of the first m particles."""
    p = np.arange(m, dtype=np.uint64)
    z0 = np.zeros(m, np.uint64)
    key = (np.uint64(int(seed) & 0xFFFFFFFF), np.uint64(int(seed) >> 32))
    sw = z0 + np.uint64(sweep)
    a = _philox((sw, p, z0 + np.uint64(1), z0), key)
    b = _philox((sw, p, z0 + np.uint64(1), z0 + np.uint64(1)), key)
    u = _philox((sw, p, z0 + np.uint64(2), z0), key)
    ra, pa = np.sqrt(-2.0 * np.log(_u01(a[0], a[1]))), 2.0 * math.pi * _u01(a[2], a[3])
    rb, pb = np.sqrt(-2.0 * np.log(_u01(b[0], b[1]))), 2.0 * math.pi * _u01(b[2], b[3])
    return np.stack([ra * np.cos(pa), ra * np.sin(pa), rb * np.cos(pb)], -1), _u01(u[0], u[1])


def _exact_chain(system, sigma, R, seed, m):
    """The first m moves of a sweep: C = I + U A^{-1} E; a ratio is the pivot that Gaussian
    elimination over the accepted moves has reached."""
    dev = torch.device("cuda")
    z, uni = _metropolis_draws(seed, EQUIL_SWEEPS, m)
    new = _wrap(R[:m] + sigma * z, system[0] * system[2])
    Rt = torch.as_tensor(R, device=dev)
    A = _rows(system, Rt)
    U = _rows(system, torch.as_tensor(new, device=dev)) - A[:m]
    E = torch.zeros(len(R), m, dtype=torch.float64, device=dev)
    E[torch.arange(m), torch.arange(m)] = 1.0
    C = (torch.eye(m, dtype=torch.float64, device=dev) + U @ torch.linalg.solve(A, E)).cpu().numpy()
    acc, rat, out = np.zeros(m, bool), np.zeros(m), R.copy()
    for k in range(m):
        rat[k] = C[k, k]
        if rat[k] * rat[k] > uni[k]:
            acc[k] = True
            out[k] = new[k]
            C[k + 1:, k + 1:] -= np.outer(C[k + 1:, k] / rat[k], C[k, k + 1:])
    return acc, rat, out


def exact(case, seed):
    rng, R, seeds = _inputs(case, seed)
    systems = _systems(case)
    if sum(1.3e-12 * _n(s) ** 3 for s in systems) > 12.0:  # seconds of dense 64-bit algebra
        return None
    dev = torch.device("cuda")
    if case["op"] in ("ratio", "alloc_free"):
        got = []
        lu = {}
        for w, k, r in _proposals(case, rng, R):
            K, _, a, kappa, rc = systems[w]
            Z = torch.as_tensor(_sites(systems[w]), device=dev)
            if w not in lu:
                A = _rows(systems[w], torch.as_tensor(R[w], device=dev))
                lu[w] = (A, torch.linalg.lu_factor(A))
            A, fac = lu[w]
            e = torch.zeros(len(R[w]), 1, dtype=torch.float64, device=dev)
            e[k] = 1.0
            x = torch.linalg.lu_solve(*fac, e)
            x = (x + torch.linalg.lu_solve(*fac, e - A @ x))[:, 0]
            L = K * a
            rt = torch.as_tensor(_wrap(r, L), device=dev)
            row = _rows(systems[w], rt)
            ratio = 1.0 + ((row - A[k]) * x).sum()
            d = rt - Z
            d = d - L * torch.round(d / L)
            px = row * x
            grad = (-2.0 * kappa * d * px[:, None]).sum(0) / ratio
            lap = ((4.0 * kappa * kappa * (d * d).sum(1) - 6.0 * kappa) * px).sum() / ratio
            got.append((ratio.item(), grad.cpu().numpy(), lap.item()))
        if case["op"] == "alloc_free":
            return np.array([g[0] for g in got])
        return {"ratio": np.array([g[0] for g in got]), "grad": np.stack([g[1] for g in got]),
                "lap": np.array([g[2] for g in got])}
    if case["op"] == "kinetic":
        out = []
        for system, r in zip(systems, R):
            K, _, a, kappa, _ = system
            rt, Z = torch.as_tensor(r, device=dev), torch.as_tensor(_sites(system), device=dev)
            A = _rows(system, rt, Z)
            d = rt[:, None, :] - Z
            d = d - K * a * torch.round(d / (K * a))
            f = 6.0 * kappa - 4.0 * kappa * kappa * (d * d).sum(-1)
            out.append(((f * A * torch.linalg.inv(A).T).sum() / (2.0 * len(r))).item())
        return np.array(out)
    acc, rat, pos = [], [], []
    for system, r, sd in zip(systems, R, seeds):
        n = _n(system)
        m = min(n, case["moves"]) if case["moves"] and case["engine"] != "dense" else n
        a, q, p = _exact_chain(system, _wl(case).sigma, r, sd, m)
        acc.append(a)
        rat.append(q)
        pos.append(p)
    return {"accepted": np.concatenate(acc), "ratio": np.concatenate(rat), "positions": np.concatenate(pos)}
