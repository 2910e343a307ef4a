"""A dipole B0 is singular at its centre: a grid with a face or a cell centre exactly
there (and no inner body around it) is non-physical in both forms, as in the CPU
oracle, not a grid whose field happens to be 0 at that point."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2501_06717_gb300 import bats
from paper_2501_06717_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _grid(lo, hi):
    root = (1, 1, 1)
    q = W.Problem("origin", lo, hi, root, W.as_leaf_array(W.uniform_leaves(root)), (W.BC_OUTFLOW,) * 6,
                  b0=W.B0_DIPOLE, b0_param=np.array([0.0, 0.0, 0.05] + [0.0] * 9))
    one = np.ones_like(W.cell_centres(lo, hi, root, q.leaves)[0])
    return W.with_state(q, [one, 0.1 * one, 0.2 * one, 0.1 * one, 0.1 * one, 0.2 * one, 0.3 * one, one])


@pytest.mark.parametrize("precision", [bats.BATS_FP64, bats.BATS_MIXED])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_face_centre_at_the_dipole(axis, precision):
    lo, hi = [-3.5] * 3, [4.5] * 3
    lo[axis], hi[axis] = -4.0, 4.0
    q = _grid(tuple(lo), tuple(hi))
    Uo, _, _ = O.run(q, q.U0, 1, dt=1e-3)
    assert not np.all(np.isfinite(Uo))
    with bats.Solver(q, precision=precision) as s:
        s.set_state(0, q.U0)
        with pytest.raises(bats.BatsError) as e:
            s.step_dt(1, 1e-3)
    assert e.value.code == bats.BATS_ERR_NONPHYSICAL


@pytest.mark.parametrize("precision", [bats.BATS_FP64, bats.BATS_MIXED])
def test_cell_centre_at_the_dipole(precision):
    q = _grid((-0.5,) * 3, (7.5,) * 3)
    q.powell = 1
    Uo, _, _ = O.run(q, q.U0, 1, dt=1e-3)
    with bats.Solver(q, precision=precision) as s:
        s.set_state(0, q.U0)
        code = 0
        try:
            s.step_dt(1, 1e-3)
        except bats.BatsError as e:
            code = e.code
    assert code == (0 if np.all(np.isfinite(Uo)) else bats.BATS_ERR_NONPHYSICAL)
