"""The mixed stage's warp-wide wait has one answer per warp: all lanes are told the
same, also where the barrier completes at the moment the limit (1 s) runs out (the
code after the wait branches on the answer around warp collectives, where lanes
that disagree would wait for one another).  Every wait and delay here ends by
itself within 3 s."""
import pytest

from paper_2501_06717_gb300 import bats
from paper_2501_06717_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def test_all_lanes_of_a_warp_get_the_same_answer():
    q = W.orszag_tang()
    with bats.Solver(q, precision=bats.BATS_MIXED) as s:
        for delay in (0.0, 0.01, 2.0, 0.9999, 0.99999, 0.999999, 1.0, 1.000001, 1.00001, 1.0001):
            rc, lanes = bats.bats_debug_wait_warp(s.h, delay)
            assert lanes.min() == lanes.max(), (delay, lanes)
            assert rc == (bats.BATS_OK if lanes[0] else bats.BATS_ERR_TIMEOUT), (delay, rc)
            if delay <= 0.5 or delay >= 1.5:
                assert lanes[0] == (delay <= 0.5), delay
        # the handle stays usable
        s.set_state(0, q.U0)
        s.step(1, 0.8)
