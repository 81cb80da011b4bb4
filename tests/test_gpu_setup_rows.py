"""AMG setup kernels at the edges of their row classes: every level's operator,
C/F split and interpolation bit for bit against the oracle, on matrices whose
rows reach past each class's capacities (row length, strong neighbours, set
size, products), and with and without truncation."""
import numpy as np
import pytest

from oracle import amg as oamg

pytestmark = pytest.mark.gpu

thermo = pytest.importorskip("paper_1902_00095_gb300.thermo")


def graph_matrix(n, degree, seed, hubs=0, positive=0.0):
    """Diagonally dominant matrix on a random symmetric graph of mean degree
    `degree`, non-symmetric values, a share `positive` of them positive;
    `hubs` rows connected to every other row."""
    rng = np.random.default_rng(seed)
    m = n * degree // 2
    i, j = rng.integers(0, n, m), rng.integers(0, n, m)
    near = rng.random(m) < 0.7  # most edges short, so that sets overlap
    j = np.where(near, (i + rng.integers(1, 2 + 2 * degree, m)) % n, j)
    pairs = {(min(a, b), max(a, b)) for a, b in zip(i, j) if a != b}
    for h in range(hubs):
        pairs |= {(min(h, b), max(h, b)) for b in range(n) if b != h}
    pairs = np.array(sorted(pairs))
    rows = np.concatenate([pairs[:, 0], pairs[:, 1], np.arange(n)])
    cols = np.concatenate([pairs[:, 1], pairs[:, 0], np.arange(n)])
    vals = -10.0 ** rng.uniform(-2.0, 0.0, rows.size)
    vals[rng.random(rows.size) < positive] *= -0.1
    order = np.lexsort((cols, rows))
    rows, cols, vals = rows[order], cols[order].astype(np.int32), vals[order]
    rowptr = np.zeros(n + 1, np.int64)
    rowptr[1:] = np.cumsum(np.bincount(rows, minlength=n))
    off = np.where(rows != cols, np.abs(vals), 0.0)
    diag = rows == cols
    vals[diag] = 1.02 * np.add.reduceat(off, rowptr[:-1]) + 1e-3
    return rowptr, cols, vals


def compare(A, interp, pmax, levels):
    g = thermo.AMG(*A, interp=interp, pmax=pmax, max_levels=levels, coarse_size=20, seed=3)
    h = oamg.setup(A, seed=3, coarse_size=20, max_levels=levels, pmax=pmax,
                   interp="ext+i" if interp else "classical")
    n, nnz = g.info()
    assert list(n) == [lev["n"] for lev in h["levels"]]
    for l, lev in enumerate(h["levels"]):
        e = g.export_level(l)
        for a, b in zip(e["A"], lev["A"]):
            assert np.array_equal(a, b), l
        if "P" in lev:
            assert np.array_equal(e["cf"], lev["cf"]), l
            for a, b in zip(e["P"], lev["P"]):
                assert np.array_equal(a, b), l
    g.close()


# degree 6: rows of the 8-lane class and a few past it; 40: the 16-lane class;
# 110 and 220: past its row length, neighbours and lists; 30 with hub rows of
# 1500 entries: past the one-pass kernels' last capacities
@pytest.mark.parametrize("n,degree,hubs", [(900, 6, 0), (25, 6, 0), (700, 40, 0), (900, 110, 0),
                                           (1000, 220, 0), (1500, 30, 2)])
@pytest.mark.parametrize("interp", [0, 1])
def test_interpolation_and_galerkin_rows_are_bit_exact(n, degree, hubs, interp):
    compare(graph_matrix(n, degree, seed=n + degree, hubs=hubs, positive=0.1), interp, 4, 3)


@pytest.mark.parametrize("pmax", [1, 3, 16, 0])
@pytest.mark.parametrize("interp", [0, 1])
def test_interpolation_widths_are_bit_exact(pmax, interp):
    compare(graph_matrix(600, 14, seed=pmax, positive=0.2), interp, pmax, 2)


# rows of R (A P) with 236 columns on average and up to 505 out of 2842 (past
# the dense-row kernel), from fewer and from more than 1024 products
def test_products_past_the_group_kernels_are_bit_exact():
    compare(graph_matrix(12000, 24, seed=12024, positive=0.1), 0, 4, 3)


def test_refreshed_galerkin_values_are_the_products_of_their_factors():
    """Newton with structure reuse refreshes the Galerkin values on known
    patterns: every operator below the first Galerkin level equals R (A P) of
    the level above it in the oracle's order, bit for bit (level 0's own values
    have moved on to the next state by the time they can be read)."""
    from synthetic import make_problem
    prob = make_problem("tiny", shape=(40, 36, 12), seed=11, dt_days=0.5)
    s = thermo.Solver.from_problem(prob)
    s.newton_step(prob["p_n"], prob["T_n"], prob["dt"], max_newton=2, tol_f=0.0, tol_dx=0.0,
                  rtol=1e-12, reuse=True)
    for w in (0, 1):
        n, _ = s.hierarchy_info(w)
        assert n.size > 2
        levels = [s.export_level(w, l) for l in range(n.size)]
        for fine, coarse in zip(levels[1:], levels[2:]):
            P = fine["P"]
            C = oamg.galerkin(fine["A"], P, oamg.transpose(P, coarse["cf"].size))
            for a, b in zip(C, coarse["A"]):
                assert np.array_equal(a, b), w
    s.close()


# block widths and fall-backs of the vertical-line step: few and many columns,
# odd columns per block, one and two layers past the middle, columns past the
# shared-memory share (nz 150: 8 columns of FP64 take 37.5 KB) and past its
# limit (nz 900: 225 KB)
@pytest.mark.parametrize("shape", [(5, 3, 2), (7, 6, 3), (13, 11, 17), (52, 51, 9), (21, 3, 150),
                                   (141, 140, 70), (3, 2, 900)])
@pytest.mark.parametrize("precision", [0, 1])
def test_line_step_by_blocks_matches_banded_solves(shape, precision):
    """One V-cycle of the Schur hierarchy (variant 1 with a zero pressure
    right-hand side applies it alone) against the same cycle from the exported
    levels with LAPACK's banded solver for the columns. FP64 rounding through
    recurrences and residuals of these diagonally dominant systems stays below
    1e-10; FP32 hierarchies below 2e-3."""
    import scipy.linalg
    import scipy.sparse as sp
    from synthetic import make_problem
    nx, ny, nz = shape
    prob = make_problem("tiny", shape=shape, seed=3)
    s = thermo.Solver.from_problem(prob)
    s.assemble(prob["p_k"], prob["T_k"], prob["p_n"], prob["T_n"], prob["dt"])
    s.build(variant=1, precision=precision)
    n, nxy = s.N, nx * ny
    csr = lambda a, shape=None: sp.csr_matrix((a[2], a[1], a[0]), shape=shape)
    sizes = s.hierarchy_info(1)[0]
    ex = [s.export_level(1, l) for l in range(sizes.size)]
    A = [csr(e["A"], (m, m)) for e, m in zip(ex, sizes)]
    P = [csr(e["P"], (m, k)) for e, m, k in zip(ex, sizes, sizes[1:])]
    d, up, lo = A[0].diagonal(), A[0].diagonal(nxy), A[0].diagonal(-nxy)

    def columns(r):
        out = np.empty(n)
        for c in range(nxy):
            k = c + nxy * np.arange(nz)
            ab = np.zeros((3, nz))
            ab[0, 1:], ab[1], ab[2, :-1] = up[k[:-1]], d[k], lo[k[:-1]]
            out[k] = scipy.linalg.solve_banded((1, 1), ab, r[k])
        return out

    def cycle(l, b):
        if l + 1 == sizes.size:
            return np.linalg.solve(A[l].toarray(), b)
        if l == 0 and sizes.size > 1:
            step = columns
        else:
            dg = A[l].diagonal()
            l1 = np.asarray(abs(A[l]).sum(axis=1)).ravel()
            step = lambda r: r / np.where(dg >= 0, l1, -l1)
        x = step(b)
        x = x + P[l] @ cycle(l + 1, P[l].T @ (b - A[l] @ x))
        return x + step(b - A[l] @ x)

    v = np.random.default_rng(7).standard_normal(n)
    _, z = s.apply_preconditioner(np.zeros(n), v)
    x = cycle(0, v)
    tol = 1e-10 if precision == 0 else 2e-3
    assert np.linalg.norm(z - x) <= tol * np.linalg.norm(x)
    s.close()
