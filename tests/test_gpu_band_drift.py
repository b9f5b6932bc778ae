"""Accuracy of the parallel banded QR in plain float where a row of R meets many reflectors (12 and 40 rows per
column): the squared residual of 20 instances against the FP64 oracle (Sec. 4.4)."""
import numpy as np
import pytest

from tests.test_gpu_band_parallel import solve
from tests.test_gpu_banded import oracle_solutions

pytestmark = pytest.mark.gpu


# The residual's entries carry a relative rounding error of some ten operations, 6e-7, of either sign; over the
# 800 and more rows that are left it averages to 2e-8 of their squared sum.  Twice that for the mean of the instances:
# a factor or an inverse off in one direction, by one unit in the last place, adds up instead.
@pytest.mark.parametrize("cols,rpc", [(200, 12), (120, 40)])
def test_squared_residual_has_no_drift(cols, rpc):
    _, res2, inst = solve([cols] * 20, rpc, 8, "fp32", 1e-3, refine_steps=0)
    _, _, want = oracle_solutions(inst, 1e-3)
    assert np.mean(np.abs(res2 - want) / want) <= 4e-8
