"""Blocks of the FP64 shower that find no part of the scratch free: their events
end with an error that the counters show, and the context stays usable."""
import numpy as np
import pytest

from tests.gpu_common import PROCESS, gaps

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 43])
def test_no_free_scratch_is_reported(pdf, n):
    import torch
    G = gaps()
    proc, sqrt_s = PROCESS["pp_lo"]
    ctx = G.gaps_init(G.make_config(proc, sqrt_s, pdf_grid=pdf, nmax=128))
    hold = G.library().gaps_test_hold_scratch
    try:
        buf = G.EventBuffers.allocate(n, 128)
        ev = buf.view()
        G.gaps_generate_hard(ctx, 0, n, ev)
        buf.status[-1:] = 1  # a record that is not to be showered keeps its status
        assert hold(ctx, 1) == 0
        G.gaps_shower(ctx, 0, n, ev)
        torch.cuda.synchronize()
        st = G.gaps_get_stats(ctx)
        status = buf.to_host(n)["status"]
        assert np.all(status[:-1] == G.GAPS_ERR_NUMERIC) and status[-1] == 1
        assert (st["events"], st["err_numeric"], st["steps"]) == (n, n - 1, 0)
        assert hold(ctx, 0) == 0
        G.gaps_generate_hard(ctx, 0, n, ev)
        G.gaps_shower(ctx, 0, n, ev)
        torch.cuda.synchronize()
        assert np.all(buf.to_host(n)["status"] == 1)
    finally:
        G.gaps_destroy(ctx)
