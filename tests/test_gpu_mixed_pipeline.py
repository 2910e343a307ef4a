"""The mixed stage kernel's block pipeline at its edges: one block in all, as many
blocks as the GPU's 152 SMs, one more, and two or three per CTA, on periodic
faces (copied slabs only) and outflow faces (slabs filled by threads), against
the CPU oracle at the mixed form's bound (1e-5 of a variable's largest value
after one step), and bit for bit equal over the blocks per work item and the
staging layouts."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2501_06717_gb300 import bats
from paper_2501_06717_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc", [W.BC_PERIODIC, W.BC_OUTFLOW])
@pytest.mark.parametrize("root", [(1, 1, 1), (4, 19, 2), (3, 3, 17), (5, 61, 1), (8, 57, 1)])
def test_blocks_per_cta_edges(root, bc):
    prob = W.Problem("pipeline", (0.0,) * 3, tuple(float(r) for r in root), root, W.as_leaf_array(W.uniform_leaves(root)),
                     (bc,) * 6)
    x, y, z = W.cell_centres(prob.lo, prob.hi, root, prob.leaves)
    s = [np.sin(2 * np.pi * (a + 0.1 * k)) for k, a in enumerate((x, y, z))]
    prob = W.with_state(prob, [1 + 0.3 * s[0] * s[1], 0.5 * s[1], 0.4 * s[2], 0.3 * s[0], 0.5 * s[2], 0.4 * s[0],
                               0.6 + 0.2 * s[1], 1 + 0.3 * s[2]])
    Uo, _, _ = O.run(prob, prob.U0, 1, cfl=0.8)
    scale = np.abs(Uo).reshape(8, -1).max(1)
    first = None
    for bpc, staging in ((1, 1), (4, 1), (1, 0)):
        with bats.Solver(prob, precision=bats.BATS_MIXED, blocks_per_cta=bpc) as h:
            h.set_staging(staging)
            h.set_state(0, prob.U0)
            h.step(1, 0.8)
            U = h.get_state(0)
        assert (np.abs(U - Uo).reshape(8, -1).max(1) / scale).max() <= 1e-5
        first = U if first is None else first
        assert np.array_equal(U, first), (bpc, staging)
