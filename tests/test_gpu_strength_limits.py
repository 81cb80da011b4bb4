"""Strength of connection where the threshold theta * max underflows to zero:
zeros are strong, positive entries are not, bit for bit with the oracle."""
import numpy as np
import pytest

from oracle import amg as oamg

pytestmark = pytest.mark.gpu

thermo = pytest.importorskip("paper_1902_00095_gb300.thermo")


@pytest.mark.parametrize("degree", [6, 40])  # 8 lanes a row, a warp a row
def test_strength_with_a_threshold_of_zero(degree):
    n, rng = 600, np.random.default_rng(degree)
    m = n * degree // 2
    i, j = rng.integers(0, n, m), rng.integers(0, n, m)
    key = np.unique(np.minimum(i, j)[i != j].astype(np.int64) * n + np.maximum(i, j)[i != j])
    a, b = key // n, key % n
    rows, cols = np.concatenate([a, b, np.arange(n)]), np.concatenate([b, a, np.arange(n)])
    tiny = 5e-324
    v = -10.0 ** rng.uniform(-2, 0, rows.size)
    # every third row: the smallest magnitude, zeros and positives; no row depends
    # on those (sums of the smallest magnitudes have no finite reciprocal)
    limit = rows % 3 == 1
    v[limit] = rng.choice([-tiny, -tiny, 0.0, -0.0, tiny, 1e-300, 1e-3], rows.size)[limit]
    v[cols % 3 == 1] = 1e-3
    v[rows == cols] = 1e3
    order = np.lexsort((cols, rows))
    rows, cols, v = rows[order], cols[order].astype(np.int32), v[order]
    rp = np.zeros(n + 1, np.int64)
    rp[1:] = np.cumsum(np.bincount(rows, minlength=n))
    theta, limit_sorted = 0.25, (rows % 3 == 1) & (cols % 3 != 1)
    want = oamg.strength((rp, cols, v), theta)
    has = np.zeros(n, bool)
    has[rows[limit_sorted & (v == -tiny)]] = True
    assert has.any() and want[limit_sorted & has[rows] & (v <= 0.0)].all()
    g = thermo.AMG(rp, cols, v, theta=theta, max_levels=2, coarse_size=20, seed=3)
    assert np.array_equal(g.export_level(0)["strong"], want)
    g.close()
