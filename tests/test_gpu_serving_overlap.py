"""Runs that are served side by side, by the server's own count of running
runs: finished boxes that wait to be taken are not counted, and runs long
enough to overlap (each lasts many times the 3 ms between submissions) end in
the states of the same runs stepped alone, bit for bit."""
import time

import numpy as np
import pytest

from paper_2602_15939_gb300 import pic as P
from test_gpu_serving import _alone, _mix, _state


@pytest.mark.gpu
def test_kept_boxes_are_not_counted_as_running():
    specs = _mix()[:3]
    with P.Server(hbm_budget_bytes=1 << 36, max_active=8, steps_per_round=4) as srv:
        for s in specs:
            s.keep_state = 1
            srv.wait(srv.submit(s), 300)
        srv.wait(0, 300)
        assert srv.peak_concurrency() == 1
        assert srv.stats().active == 0 and srv.stats().peak_active == len(specs)


@pytest.mark.gpu
def test_states_of_runs_that_overlap_equal_the_runs_stepped_alone():
    specs = _mix()
    for s in specs:
        s.keep_state = 1
        s.nsteps *= 20
    with P.Server(hbm_budget_bytes=1 << 36, max_active=8, steps_per_round=4) as srv:
        tickets = []
        for s in specs:
            tickets.append(srv.submit(s))
            time.sleep(0.003)
        srv.wait(0, 300)
        assert srv.peak_concurrency() >= 2
        served = []
        for t, s in zip(tickets, specs):
            with srv.take(t) as b:
                served.append(_state(b, s.nspecies))
    for s, (parts, fields) in zip(specs, served):
        with _alone(s) as box:
            box.step(s.nsteps)
            parts_alone, fields_alone = _state(box, s.nspecies)
        for got, want in zip(parts, parts_alone):
            for g, w in zip(got, want):
                np.testing.assert_array_equal(g, w)
        for g, w in zip(fields, fields_alone):
            np.testing.assert_array_equal(g, w)
