"""The mixed stage kernel's CTAs walk over items of several consecutive blocks, of at
most as many as leave a CTA eight items: grids large enough for items of 2 and 3
blocks with a partial last item give the same bits as single blocks, on slabs
filled by threads (outflow), resolution changes with refluxing, local time steps
and SSP-RK2, and with body cells and a dipole field (the general cell phase).
(Equal bits for two items of different lengths also need the walk over them to
cover every block once.)"""
import numpy as np
import pytest

from paper_2501_06717_gb300 import bats
from paper_2501_06717_gb300 import workloads as W

pytestmark = pytest.mark.gpu

BODY = np.array([1.5, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 1.2])
DIPOLE = np.array([0.0, 0.0, 0.05] + [0.0] * 9)


def _grid(root, radius, bc, **more):
    lo, hi = (-1.0,) * 3, (1.0,) * 3
    leaves = W.uniform_leaves(root)
    if radius:
        near = lambda b0, b1: bool(np.sum(np.maximum(0, np.maximum(b0, -b1)) ** 2) < radius ** 2)
        leaves = W.balance(W.refine_where(leaves, near, lo, hi, root, 1), root, (bc == W.BC_PERIODIC,) * 3)
    prob = W.Problem("items", lo, hi, root, W.as_leaf_array(W.morton_sort(leaves)), (bc,) * 6, **more)
    x = W.cell_centres(lo, hi, root, prob.leaves)
    s = [np.sin(np.pi * (a + 0.1 * k)) for k, a in enumerate(x)]
    w = [1 + 0.3 * s[0] * s[1], 0.5 * s[1], 0.4 * s[2], 0.3 * s[0], 0.5 * s[2], 0.4 * s[0], 0.6 + 0.2 * s[1], 1 + 0.3 * s[2]]
    if prob.body_r:
        inside = x[0] * x[0] + x[1] * x[1] + x[2] * x[2] < prob.body_r ** 2
        w = [np.where(inside, prob.body[v], w[v]) for v in range(8)]
    return W.with_state(prob, w)


@pytest.mark.parametrize("root,radius,bc,more,sizes", [
    ((5, 7, 109), 0.0, W.BC_OUTFLOW, {}, (2, 3, 16)),
    ((5, 7, 109), 0.0, W.BC_PERIODIC, dict(flux=W.FLUX_LINDE, rk=W.RK_SSP2, limiter=W.LIM_MC), (2, 3)),
    ((15, 13, 10), 0.4, W.BC_OUTFLOW, dict(reflux=1, powell=1), (2,)),
    ((15, 13, 10), 0.4, W.BC_PERIODIC, dict(local_dt=1, flux=W.FLUX_HLL), (2,)),
    ((15, 13, 10), 0.4, W.BC_OUTFLOW, dict(b0=W.B0_DIPOLE, b0_param=DIPOLE, powell=1, body_r=0.3, body=BODY), (2,))])
def test_items_of_several_blocks(root, radius, bc, more, sizes):
    import torch
    q = _grid(root, radius, bc, **more)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    first = None
    with bats.Solver(q, precision=bats.BATS_MIXED) as h:
        for size in (1,) + sizes:
            if size <= 3:  # items of `size` blocks, the last one partial
                assert q.nb >= size * 8 * sms and (size == 1 or q.nb % size)
            h.set_launch(0, size, 0, 0)
            h.set_state(0, q.U0)
            h.step(2, 0.5)
            U = h.get_state(0)
            first = U if first is None else first
            assert np.array_equal(U, first), size
