"""The divergence counters of the kept-trial shower: lane_steps are the event's own
cycles, once each (those evaluated ahead of an emission and dropped do not count),
among the lanes that warp_steps counts."""
import numpy as np
import pytest

from tests.gpu_common import gaps, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,kw", [(20_011, {}), (20_011, {"max_cycles": 13}), (3001, {"nmax": 9}), (1, {})])
def test_lane_steps_are_committed_cycles(pdf, n, kw):
    G = gaps()
    g = run_gpu(G, 2, 13600.0, 7, n, pdf, precision=G.GAPS_MIXED, schedule=G.GAPS_SCHED_PERSISTENT, obs=False, **kw)
    st = g["stats"]
    # an event's last cycle has no trial above the cutoff, and nothing to evaluate
    done = int(np.sum(g["status"] == 1))
    assert st["lane_steps"] == st["steps"] - done
    assert st["lane_steps"] <= st["warp_steps"] and st["warp_steps"] % 32 == 0
