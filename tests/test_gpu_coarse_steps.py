"""Coarsest inverse at the edges of its split over CTAs and lanes: fewer rows
than CTAs, one row more than a multiple, rows past one warp's lanes, the
largest size that stays in shared memory and one past it; with equal pivot
candidates and pivots spread over all CTAs."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

thermo = pytest.importorskip("paper_1902_00095_gb300.thermo")


@pytest.mark.parametrize("n", [3, 15, 16, 17, 33, 127, 511, 513, 528, 650, 651])
@pytest.mark.parametrize("kind", ["signs", "spread"])
def test_coarse_inverse_at_split_edges(n, kind):
    rng = np.random.default_rng(n)
    if kind == "signs":  # every candidate of the first column has the same magnitude
        A = rng.choice([-1.0, 1.0], (n, n))
        A[np.arange(n), rng.permutation(n)] *= n
        A[:, 0] = rng.choice([-1.0, 1.0], n)
    else:
        A = 0.1 * rng.standard_normal((n, n)) / np.sqrt(n)
        A[rng.permutation(n), np.arange(n)] += 1.0 + rng.random(n)
        A[np.arange(n), np.arange(n)] += 1e-9
    rp = np.arange(n + 1, dtype=np.int32) * n
    g = thermo.AMG(rp, np.tile(np.arange(n, dtype=np.int32), n), A.ravel(), max_levels=1)
    b = rng.standard_normal(n)
    x, ref = g.vcycle(b), np.linalg.solve(A, b)
    # growth of partial pivoting with tied candidates stays far below 1e4 here
    assert np.linalg.norm(x - ref) <= 1e-12 * np.linalg.cond(A) * np.linalg.norm(ref)
    g.close()
