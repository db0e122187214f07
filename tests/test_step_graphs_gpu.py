"""Which dg_step calls replay a graph: a step size that comes back does, also when
several take turns, and a graph that the handle holds is used; one that comes for
the first time runs directly, with the same states."""
import numpy as np
import pytest

from paper_2303_11767_gb300 import dgswe
from test_parity_gpu import case

pytestmark = pytest.mark.gpu


def _run(calls):
    _, u = case(24, 12, 2, 11)
    with dgswe.Solver(24, 12, 2, precision="fp32") as s:
        s.set_state(u)
        replays = []
        for n, dt, order in calls:
            s.set_option(dgswe.OPT_RK_ORDER, order)
            before = s.graph_replays()
            s.step(n, dt)
            replays.append(s.graph_replays() - before)
        return replays, s.get_state()


@pytest.mark.parametrize("calls,want", [
    ([(4, 1.0, 3)] * 3, [0, 1, 1]),
    ([(4, 1.0, 3), (4, 2.0, 3)] * 3, [0, 0, 1, 1, 1, 1]),                    # two step sizes in turn
    ([(4, 1.0, 3), (4, 1.0, 4)] * 3, [0, 0, 1, 1, 1, 1]),                    # two orders in turn
    ([(4, 1.0, 3), (4, 1.0, 3), (4, 2.0, 3), (4, 1.0, 3)], [0, 1, 0, 1]),    # back to a held graph
    ([(4, 1.0 + k, 3) for k in range(12)], [0] * 12),                        # a new size each time
    ([(33, 1.0, 3)], [2]),                                                   # two replays in the first call
])
def test_replays(calls, want):
    got, state = _run(calls)
    assert got == want
    _, u = case(24, 12, 2, 11)
    with dgswe.Solver(24, 12, 2, precision="fp32") as s:                     # one step at a time
        s.set_state(u)
        for n, dt, order in calls:
            s.set_option(dgswe.OPT_RK_ORDER, order)
            for _ in range(n):
                s.step(1, dt)
        assert np.array_equal(s.get_state(), state)
