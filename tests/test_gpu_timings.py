"""bats_get_timings over calls of any length: the stages' time is measured in every
step, eager and under graph replay, so the rest (two time-step kernels a step) is
what remains of the total, not nothing.

Bounds: a time-step kernel reads and writes device memory in a chain (speed bound,
dt), which takes at least 0.5 us; two a step.  The stages' mean time per step of a
replay does not depend on the length of the call beyond what the first steps differ
(cold caches, clocks): a factor of 1.5.  (Eager launches also wait for the host.)"""
import pytest

from paper_2501_06717_gb300 import bats
from paper_2501_06717_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [bats.BATS_FP64, bats.BATS_MIXED])
@pytest.mark.parametrize("graph", [0, 1])
def test_phases_of_long_calls(graph, precision):
    q = W.orszag_tang()
    mean = []
    with bats.Solver(q, precision=precision, use_graph=graph) as s:
        for n in (100, 4, 20, 100):  # the first call warms up
            s.set_state(0, q.U0)
            s.step(n, 0.1)
            stage, dt, total = s.timings()
            assert 0 < stage < total and abs(stage + dt - total) < 1e-6 * total
            assert dt >= n * 2 * 0.5e-3, (n, stage, dt, total)
            mean.append(stage / n)
        s.step(0, 0.1)
        assert s.timings()[0] == -1.0
    if graph:
        assert max(mean[1:]) < 1.5 * min(mean[1:]), mean
