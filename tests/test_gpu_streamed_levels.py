"""Levels whose sweeps stream more than L2 holds (their entries are loaded past
L1): the V-cycle against the same cycle on the exported operators in FP64 on
the host."""
import numpy as np
import pytest
import scipy.sparse as sp

pytestmark = pytest.mark.gpu

thermo = pytest.importorskip("paper_1902_00095_gb300.thermo")

STREAM_BYTES = 180e6  # kStreamBytes of the V-cycle


def grid_operator(nx, ny, nz, seed):
    """7-point operator of an nx x ny x nz grid with log-normal face
    coefficients, vertical ones 30 times smaller, slightly diagonally dominant."""
    rng = np.random.default_rng(seed)
    n = nx * ny * nz
    cell = np.arange(n).reshape(nz, ny, nx)
    rows, cols, vals = [], [], []
    for axis, scale in ((0, 1.0 / 30.0), (1, 1.0), (2, 1.0)):
        lo = np.delete(cell, -1, axis).ravel()
        hi = np.delete(cell, 0, axis).ravel()
        t = scale * np.exp(rng.standard_normal(lo.size))
        rows += [lo, hi]
        cols += [hi, lo]
        vals += [-t, -t]
    off = sp.csr_matrix((np.concatenate(vals), (np.concatenate(rows), np.concatenate(cols))), (n, n))
    A = (off + sp.diags(1.001 * -np.asarray(off.sum(axis=1)).ravel())).tocsr()
    A.sort_indices()
    return A


def l1_diag(A):
    d = A.diagonal()
    return np.where(d >= 0.0, 1.0, -1.0) * np.asarray(abs(A).sum(axis=1)).ravel()


def host_cycle(levels, b, l, nu_pre, nu_post):
    A, P, dinv = levels[l]
    if P is None:
        return np.linalg.solve(A.toarray(), b)
    x = dinv * b
    for _ in range(1, nu_pre):
        x = x + dinv * (b - A @ x)
    x = x + P @ host_cycle(levels, P.T @ (b - A @ x), l + 1, nu_pre, nu_post)
    for _ in range(nu_post):
        x = x + dinv * (b - A @ x)
    return x


# FP32: 12 levels of 9 passes over rows of some 30 entries, 2^-24 each
@pytest.mark.parametrize("precision,tol", [(0, 1e-11), (1, 2e-4)])
def test_vcycle_on_streamed_levels(precision, tol):
    A = grid_operator(151, 150, 149, seed=8)
    g = thermo.AMG(A.indptr, A.indices, A.data, precision=precision, seed=3, nu_pre=3, nu_post=4)
    n, nnz = g.info()
    size = 8 if precision == 0 else 4
    assert nnz[0] * (size + 4) > STREAM_BYTES
    if precision == 0:
        assert g.level_storage(1)[0] == 2 and nnz[1] * 12 > STREAM_BYTES
    levels = []
    for l in range(len(n)):
        e = g.export_level(l)
        M = sp.csr_matrix((e["A"][2], e["A"][1], e["A"][0]), (n[l], n[l]))
        P = e["P"] and sp.csr_matrix((e["P"][2], e["P"][1], e["P"][0]), (n[l], n[l + 1]))
        levels.append((M, P, 1.0 / l1_diag(M)))
    b = np.random.default_rng(9).standard_normal(A.shape[0])
    x, ref = g.vcycle(b), host_cycle(levels, b, 0, 3, 4)
    assert np.max(np.abs(x - ref)) <= tol * np.max(np.abs(ref))
    g.close()
