"""Walkers whose Krylov vectors do not fit the task ring (FP64 from about 12 000 particles, FP32
from 24 000): the product with A gathers from the solve area, or from global memory where not
even the solve vector fits shared memory.  Ratios against GMRES in plain 64-bit arithmetic on
the sparse matrix (scipy), at sizes on either side of both lines; the bar is that of the parity
tests, 1e-10 relative."""
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


def _phi(r, Z, L, kappa, rc):
    d = r[:, None, :] - Z[None, :, :]
    d -= L * np.round(d / L)
    d2 = (d * d).sum(-1)
    return np.where(d2 <= rc * rc, np.exp(-kappa * d2), 0.0)


@pytest.mark.parametrize("K,prec,threads", [(22, 0, 0), (24, 0, 0), (24, 0, 96), (28, 1, 0), (30, 1, 0), (30, 1, 64),
                                            (30, 0, 0)])
def test_ratios(vmc, K, prec, threads):
    from scipy.sparse import csr_matrix
    from scipy.sparse.linalg import gmres

    kappa, rc, L = 2.0, 1.5, float(K)
    rng = np.random.default_rng(K)
    g = np.arange(K, dtype=np.float64)
    Z = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)[:, ::-1]  # x fastest
    n = len(Z)
    R = np.mod(Z + 0.1 * rng.standard_normal((n, 3)), L)
    rows, cols, vals = [], [], []
    near = np.stack(np.meshgrid(*[np.arange(-2, 3)] * 3, indexing="ij"), -1).reshape(-1, 3)
    cell = np.floor(R + 0.5).astype(int)
    for off in near:  # every site within r_c of a particle is within two cells of the nearest site
        c = np.mod(cell + off, K)
        j = c[:, 0] + K * (c[:, 1] + K * c[:, 2])
        d = R - Z[j]
        d -= L * np.round(d / L)
        d2 = (d * d).sum(1)
        m = d2 <= rc * rc
        rows.append(np.nonzero(m)[0]); cols.append(j[m]); vals.append(np.exp(-kappa * d2[m]))
    A = csr_matrix((np.concatenate(vals), (np.concatenate(rows), np.concatenate(cols))), shape=(n, n))
    ctx = vmc.vmc_create([(K, 0, 1.0, kappa, rc)], vmc.params(precision=prec, block_threads=threads))
    try:
        vmc.vmc_set_positions(ctx, 0, R)
        for k in (0, n // 2, n - 1):
            r = np.mod(R[k] + 0.2 * rng.standard_normal(3), L)
            got = vmc.vmc_ratio(ctx, 0, k, r)
            e = np.zeros(n)
            e[k] = 1.0
            x, info = gmres(A, e, rtol=1e-14, atol=0.0, restart=80, maxiter=20)
            assert np.linalg.norm(A @ x - e) < 1e-13
            want = 1.0 + (_phi(r[None], Z, L, kappa, rc)[0] - A[k].toarray()[0]) @ x
            assert abs(got - want) <= 1e-10 * max(abs(want), 1e-3)
    finally:
        vmc.vmc_destroy(ctx)
