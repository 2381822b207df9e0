"""A context is ready when gaps_init returns, whatever stream its first call uses:
its counters and the flags of the FP64 scratch are cleared on the legacy stream,
for which a non-blocking stream does not wait."""
import threading

import numpy as np
import pytest

from tests.gpu_common import PROCESS, gaps

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    return gaps()


@pytest.mark.parametrize("precision", [0, 1])
def test_first_call_on_a_stream_that_does_not_wait_for_the_legacy_one(G, pdf, precision):
    import torch
    proc, sqrt_s = PROCESS["pp_lo"]
    n = 3001
    buf = G.EventBuffers.allocate(n, 128)
    ev = buf.view()
    a = torch.randn(4096, 4096, device="cuda")
    b = torch.empty_like(a)
    torch.cuda.synchronize()
    stop = threading.Event()

    def keep_busy():  # the legacy stream, always some milliseconds behind
        while not stop.is_set():
            for _ in range(8):
                torch.mm(a, a, out=b)
            torch.cuda.current_stream().synchronize()

    other = torch.cuda.Stream()  # (torch's streams are non-blocking)
    t = threading.Thread(target=keep_busy)
    t.start()
    try:
        for k in range(5):
            # memory that the context may get: not zero
            junk = torch.full((1 << 26,), -1, dtype=torch.int32, device="cuda")
            del junk
            torch.cuda.empty_cache()
            ctx = G.gaps_init(G.make_config(proc, sqrt_s, pdf_grid=pdf, nmax=128, precision=precision))
            try:
                G.gaps_generate_hard(ctx, 1000 * k, n, ev, other)
                G.gaps_shower(ctx, 1000 * k, n, ev, other)
                other.synchronize()
                st = G.gaps_get_stats(ctx, other)
            finally:
                G.gaps_destroy(ctx)
            assert np.all(buf.to_host(n)["status"] == 1)
            assert st["events"] == n and st["accepts"] == buf.to_host(n)["n_emit"].sum()
    finally:
        stop.set()
        t.join()
