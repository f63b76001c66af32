"""The operation counts of bench.py's FP64 rooflines against counts of the elimination itself."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def _lu_operations(m, n):
    """Multiply-adds (two operations each) of the trailing updates of one m x n LU."""
    return sum(2 * (m - j - 1) * (n - j - 1) for j in range(n))


@pytest.mark.parametrize("m,n", [(1600, 700), (700, 700), (2304, 1152)])
def test_lu_count(m, n):
    import bench

    assert bench.lu_flop(m, n) == pytest.approx(_lu_operations(m, n), rel=2.0 / n)


@pytest.mark.parametrize("Ns,n_e", [(576, 576), (400, 200)])
def test_spin_coupled_recompute_is_counted_once_per_walker(Ns, n_e):
    import bench

    got = bench.soc_recompute_flop(Ns, n_e)
    assert got["elim"] == pytest.approx(_lu_operations(4 * Ns, 2 * n_e), rel=2.0 / n_e)
    assert got["lu_o"] == pytest.approx(_lu_operations(2 * n_e, 2 * n_e), rel=2.0 / n_e)
    assert got["solve"] == 2 * (2 * n_e) ** 2 * (2 * Ns)  # a multiply-add per entry of L and U and column
