"""A non-physical cell ends a call with an error and leaves the grid's speed bound (and
with it the next time step) to the other cells, in both forms, also where both cells
that the mixed form's packed cell phase takes together (four layers apart) are
non-physical."""
import numpy as np
import pytest

from paper_2501_06717_gb300 import bats
from paper_2501_06717_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [bats.BATS_FP64, bats.BATS_MIXED])
@pytest.mark.parametrize("layers", [(1,), (1, 5)])
def test_time_step_after_a_non_physical_cell(layers, precision):
    root = (2, 2, 2)
    q = W.Problem("bound", (-1.0,) * 3, (1.0,) * 3, root, W.as_leaf_array(W.uniform_leaves(root)), (W.BC_PERIODIC,) * 6)
    x, y, z = W.cell_centres(q.lo, q.hi, root, q.leaves)
    one = np.ones_like(x)
    q = W.with_state(q, [one + 0.1 * np.sin(np.pi * x), 0.1 * one, 0 * one, 0 * one, 0.3 * one, 0.2 * one, 0 * one, one])
    with bats.Solver(q, precision=precision) as s:
        s.set_state(0, q.U0)
        dt = s.dt(0, 0.8)
        U0 = q.U0.copy()
        for k in layers:
            U0[7, 3, k, 4, 4] = np.nan
        s.set_state(0, U0)
        with pytest.raises(bats.BatsError) as e:
            s.step_dt(1, 1e-4)
        assert e.value.code == bats.BATS_ERR_NONPHYSICAL
        assert abs(s.dt(0, 0.8) / dt - 1) < 0.1
