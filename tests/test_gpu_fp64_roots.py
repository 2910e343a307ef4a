"""FP64 form where the fast-speed roots are at their edges: B = 0 (the inner
root is exactly G), the degenerate sound = Alfven case along a field line (the
inner root of zero), and magnitudes far from one; against the CPU oracle.

Tolerance, per variable relative to its largest value after 3 steps (6 stages).
B = 0: about 50 dependent FP64 operations per cell and stage, each rounded once
(2^-53), 50 x 6 x 1.1e-16 = 3e-14 if all errors add up: 1e-13.  Degenerate: the
inner root's argument is a difference of equal terms, known to about 3 x 2^-53
of them, so the speed is known to sqrt(3.3e-16) = 2e-8 only, in the oracle as
here; it multiplies the jump of the two face states (at most 0.1 of a variable)
and enters with dt/dx c <= 0.8 over the directions, 6 stages: 6 x 0.8 x 0.1 x
2e-8 = 1e-8."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2501_06717_gb300 import bats
from paper_2501_06717_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flux", [W.FLUX_RUSANOV, W.FLUX_HLL, W.FLUX_LINDE])
@pytest.mark.parametrize("limiter", [W.LIM_MINMOD, W.LIM_MC])
@pytest.mark.parametrize("field,scale", [("none", 1.0), ("degenerate", 1.0), ("degenerate", 1e-12), ("degenerate", 1e15)])
def test_fast_speed_edges(field, scale, limiter, flux):
    root = (2, 2, 2)
    prob = W.Problem("edges", (0.0,) * 3, (1.0,) * 3, root, W.as_leaf_array(W.uniform_leaves(root)), (W.BC_PERIODIC,) * 6,
                     limiter=limiter, flux=flux)
    x, y, z = W.cell_centres(prob.lo, prob.hi, root, prob.leaves)
    g, s = prob.gamma, np.sin(2 * np.pi * (x + 2 * y))
    one = np.ones_like(x)
    rho = one + (0.0 if field == "degenerate" else 0.2) * s
    b = 0.0 if field == "none" else 1.0
    p = one / g + (0.0 if field == "degenerate" else 0.1) * np.cos(2 * np.pi * z)  # a^2 = 1 = B^2 / rho
    u = 0.1 * s
    # similarity scaling: rho, p and B^2 by the same factor leave u unchanged
    prob = W.with_state(prob, [scale * rho, u, 0.5 * u, 0 * one, np.sqrt(scale) * b * one, 0 * one, 0 * one, scale * p])
    Uo, _, _ = O.run(prob, prob.U0, 3, cfl=0.8)
    with bats.Solver(prob) as h:
        h.set_state(0, prob.U0)
        h.step(3, 0.8)
        Ug = h.get_state(0)
    vec = np.abs(Uo).reshape(8, -1).max(1)
    for c in ((1, 2, 3), (4, 5, 6)):  # a component near zero against its vector's largest
        vec[list(c)] = vec[list(c)].max()
    vec = np.where(vec > 0, vec, 1.0)
    assert (np.abs(Ug - Uo).reshape(8, -1).max(1) / vec).max() <= (1e-13 if field == "none" else 1e-8)
