"""fh_footprint counts what a context holds: synthesis tables once per distinct J, the LU's row moves per solve."""
import numpy as np
import pytest

from paper_1807_02718_gb300 import fh as F


@pytest.mark.parametrize("precision", [F.FH_FP64, F.FH_MIXED_BF16])
def test_shared_tables_are_counted_once(precision):
    from paper_1807_02718_gb300 import build
    build.build()
    N = {J: np.full(J, 16) for J in (128, 129)}
    one, other = (F.fh_footprint([J], [N[J]], precision) for J in (128, 129))
    both, twice = F.fh_footprint([128, 129], [N[128], N[129]], precision), F.fh_footprint([128] * 2, [N[128]] * 2, precision)
    assert both == one + other
    h, J = 127, 128                              # half the period, frequencies
    rows = 2 * (int(np.ceil(2.5 * h)) + 24) + 1  # half-integer samples of the near sums
    assert 2 * one - twice == 16 * (64 * J + 2 * (J - 1) + rows * J)


def test_row_moves_are_counted():
    """A panel of 16 columns moves at most 32 rows: two lists of 32 indices and their length for every solve."""
    from paper_1807_02718_gb300 import build
    build.build()
    small, large = (F.fh_footprint([J], [np.full(J, 8)], F.FH_FP64) for J in (2000, 2001))   # no near table past J = 1025
    n = 8
    assert large - small >= 16 * n * n + 16 * n * 4 + (2 * 32 + 1) * 4 + 16 * 64
