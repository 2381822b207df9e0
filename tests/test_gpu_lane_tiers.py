"""The lane kernel in its register tiers (blocks of an SM's 512, 768 and 1024
threads): the trial schemes that run in it give the same events in all of them."""
import numpy as np
import pytest

from tests.gpu_common import gaps, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["REDRAW", "SELECT", "VETOMAX"])
@pytest.mark.parametrize("block,per_sm", [(256, 3), (256, 4)])
def test_tiers_give_the_same_events(pdf, name, block, per_sm):
    G = gaps()
    mode = getattr(G, "GAPS_TRIALS_" + name)
    a, b = (run_gpu(G, 2, 13600.0, 77, 20_011, pdf, precision=G.GAPS_MIXED, schedule=G.GAPS_SCHED_PERSISTENT,
                    trial_mode=mode, obs=False, block_size=bs, blocks_per_sm=ps)
            for bs, ps in ((128, 2), (block, per_sm)))
    assert np.all(a["status"] == 1)
    for k in ("p", "flav", "col", "acol", "npart", "status", "n_emit", "weight", "t", "eta"):
        assert np.array_equal(a[k], b[k]), k
    for k in ("events", "steps", "trials", "isr_trials", "vetoes", "accepts", "rebuilds"):
        assert a["stats"][k] == b["stats"][k], k
