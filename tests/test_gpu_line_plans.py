"""Radices that the grids of test_gpu_lines.py leave out (the plan of a length
changes with the size of its grid), by the same comparison with the oracle; the
plans of FP64 boxes of 2^20 sites against the 2D solve."""
import pytest

import paper_1804_02883_gb300 as P
from test_gpu_lines import test_box_with_more_rows_than_partials as _box
from test_gpu_lines import test_solve_on_every_plan as _solve

MORE = [(8, 64), (144, 8), (90, 200), (108, 320), (40, 900), (64, 540)]
BOX = (128, 90, 96)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED_FP32])
@pytest.mark.parametrize("ny,nx", MORE)
def test_solve_on_the_other_plans(ny, nx, precision):
    _solve(ny, nx, precision)


@pytest.mark.gpu
@pytest.mark.parametrize("precision", [P.PLAIN_FP64, P.MIXED_FP32])
def test_large_box(precision):
    _box(*BOX, precision)
