"""FP64 stage of small handles, whose blocks are shared by 8, 4 or 2 CTAs (by layers
of cells) when all of those fit the GPU's 152 SMs: a grid advanced alone and the
same grid advanced beside others that bring the handle past the limit of every
split give the same bits, on refined grids with every kind of face, the body, a
background field, local time steps and refluxing; and a split grid agrees with
the CPU oracle at the FP64 form's bound (1e-12 of a variable's largest value)."""
from dataclasses import replace

import numpy as np
import pytest

from oracle import oracle as O
from paper_2501_06717_gb300 import bats
from paper_2501_06717_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _grid(root, refine, bc, **more):
    leaves = W.uniform_leaves(root)
    if refine:
        leaves = W.balance(W.refine_where(leaves, lambda b0, b1: bool(np.all(b0 <= 0.0) and np.all(b1 >= 0.0)),
                                          (-1.0,) * 3, (1.0,) * 3, root, 1), root, (bc == W.BC_PERIODIC,) * 3)
    prob = W.Problem("split", (-1.0,) * 3, (1.0,) * 3, root, W.as_leaf_array(W.morton_sort(leaves)), (bc,) * 6, **more)
    x, y, z = W.cell_centres(prob.lo, prob.hi, root, prob.leaves)
    s = [np.sin(np.pi * (a + 0.1 * k)) for k, a in enumerate((x, y, z))]
    w = [1 + 0.3 * s[0] * s[1], 0.5 * s[1], 0.4 * s[2], 0.3 * s[0], 0.5 * s[2], 0.4 * s[0], 0.6 + 0.2 * s[1], 1 + 0.3 * s[2]]
    if prob.body_r:
        inside = x * x + y * y + z * z < prob.body_r ** 2
        w = [np.where(inside, prob.body[v], w[v]) for v in range(8)]
    return W.with_state(prob, w)


DIPOLE = np.array([0.0, 0.0, 0.05] + [0.0] * 9)
BODY = np.array([1.5, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 1.2])
CASES = [((1, 1, 1), False, W.BC_PERIODIC, {}),                                      # 1 block: 8 CTAs each
         ((3, 3, 2), False, W.BC_OUTFLOW, dict(limiter=W.LIM_MC, flux=W.FLUX_HLL)),  # 18: 8
         ((3, 3, 3), True, W.BC_OUTFLOW, dict(flux=W.FLUX_LINDE, reflux=1)),         # 34: 4
         ((3, 3, 3), True, W.BC_PERIODIC, dict(limiter=W.LIM_MC, rk=W.RK_SSP2)),     # 34: 4
         ((4, 4, 3), False, W.BC_OUTFLOW, dict(limiter=W.LIM_NONE, rk=W.RK_EULER)),  # 48: 2
         ((3, 3, 3), True, W.BC_OUTFLOW, dict(b0=W.B0_DIPOLE, b0_param=DIPOLE, powell=1, body_r=0.3, body=BODY,
                                              local_dt=1))]                          # 34: 4


@pytest.mark.parametrize("case", range(len(CASES)))
def test_split_equals_whole_blocks(case):
    root, refine, bc, more = CASES[case]
    q = _grid(root, refine, bc, **more)
    with bats.Solver(q) as h:
        h.set_state(0, q.U0)
        h.step(3, 0.5)
        alone = h.get_state(0)
    many = [q] + [replace(q) for _ in range(77 // q.nb + 1)]  # more than half the SMs: no split
    with bats.Solver(many) as h:
        for g in range(len(many)):
            h.set_state(g, q.U0)
        h.step(3, 0.5)
        beside = h.get_state(0)
    assert np.array_equal(alone, beside)
    Uo, _, _ = O.run(q, q.U0, 3, cfl=0.5)
    scale = np.abs(Uo).reshape(8, -1).max(1)
    for c in ((1, 2, 3), (4, 5, 6)):  # a component near zero against its vector's largest
        scale[list(c)] = scale[list(c)].max()
    assert (np.abs(alone - Uo).reshape(8, -1).max(1) / scale).max() <= 1e-12
