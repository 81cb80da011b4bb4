"""Interpolation rows past the capacities of the one-pass kernels: F rows with
far more strong neighbours than the level's others, and levels of long rows
throughout, bit for bit against the oracle on every level."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

pytest.importorskip("paper_1902_00095_gb300.thermo")
from test_gpu_setup_rows import compare, graph_matrix  # noqa: E402


def with_long_f_rows(n, degree, hubs):
    """`hubs` rows connected to every other row which no other row strongly
    depends on: they become F points (and stay diagonally dominant)."""
    rowptr, cols, vals = graph_matrix(n, degree, seed=n + hubs, hubs=hubs, positive=0.1)
    rows = np.repeat(np.arange(n), np.diff(rowptr))
    vals[(cols < hubs) & (rows >= hubs)] *= 1e-4
    return rowptr, cols, vals


# 300: rows the last class takes; 900: more than 128 strong F neighbours; 1500 and
# 3000: more than 1024 entries; degree 6 lists them through all three classes,
# 30 through two, 110 sends the level to the untruncated kernels
@pytest.mark.parametrize("n,degree,hubs", [(300, 6, 2), (900, 6, 1), (900, 30, 3), (1500, 6, 2),
                                           (3000, 30, 2), (1100, 110, 1)])
@pytest.mark.parametrize("interp", [0, 1])
def test_long_f_rows_are_bit_exact(n, degree, hubs, interp):
    compare(with_long_f_rows(n, degree, hubs), interp, 4, 3)


@pytest.mark.parametrize("pmax", [1, 16])
@pytest.mark.parametrize("interp", [0, 1])
def test_long_f_rows_and_widths_are_bit_exact(pmax, interp):
    compare(with_long_f_rows(1200, 8, 2), interp, pmax, 2)


# rows of 650 entries on average, most with more than 128 strong F neighbours
def test_a_level_of_long_rows_is_bit_exact():
    A = graph_matrix(1000, 1050, seed=3, positive=0.1)
    compare(A, 0, 4, 2)
