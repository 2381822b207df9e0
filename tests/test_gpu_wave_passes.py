"""The wavefront's passes (end tables, veto cycles, emissions as kernels of their
own) against the persistent lane kernel, for the trial schemes that run in them:
redrawn trials and generate-select. Records and counters are compared exactly."""
import numpy as np
import pytest

from tests.gpu_common import gaps

pytestmark = pytest.mark.gpu

MIX = [(2, 13600.0, 1.0, 0.5), (0, 91.2, 0.5, 0.25), (0, 500.0, 4.0, 0.25)]
COUNTERS = ("events", "steps", "trials", "isr_trials", "vetoes", "accepts", "violations", "err_capacity",
            "err_iter_cap", "err_numeric", "rebuilds", "mlp_tiles")


@pytest.fixture(scope="module")
def G():
    return gaps()


def _run(G, pdf, schedule, mode, n, net=None, cap=None, mix=None, nmax=128, **kw):
    import torch
    ctx = G.gaps_init(G.make_config(0 if mix else 2, 91.2 if mix else 13600.0, pdf_grid=pdf, nmax=nmax, seed=1,
                                    precision=G.GAPS_MIXED, schedule=schedule, trial_mode=mode, mix=mix, **kw))
    try:
        if net is not None:
            G.gaps_set_learned_proposal(ctx, *net)
        buf = G.EventBuffers.allocate(cap or n, nmax)
        ev = buf.view()
        G.gaps_generate_hard(ctx, 99, n, ev)
        G.gaps_shower(ctx, 99, n, ev)
        torch.cuda.synchronize()
        out = buf.to_host(n)
        out["draw"] = buf.draw[:n].cpu().numpy()
        return out, G.gaps_get_stats(ctx)
    finally:
        G.gaps_destroy(ctx)


@pytest.mark.parametrize("mode", [0, 2])
@pytest.mark.parametrize("n,learned,kw", [
    (6000, False, {"wave_passes": 1}),
    (6000, False, {"wave_passes": 64}),
    (8000, True, {}),
    (8000, True, {"wave_passes": 3}),
    (9001, False, {"mix": MIX}),
    (3001, False, {"nmax": 8, "cap": 4096}),
    (2000, False, {"max_cycles": 3}),
    (1, True, {"cap": 16}),
])
def test_passes_equal_the_lane_kernel(G, pdf, mode, n, learned, kw):
    net = None
    if learned:
        from paper_2511_19633_gb300 import learned as L
        net = (L.init_params(5), np.zeros((G.GAPS_ISR_CLASSES, G.GAPS_ISR_ETA_BINS, G.GAPS_ISR_BINS),
                                          dtype=np.float32))
    a, sa = _run(G, pdf, G.GAPS_SCHED_PERSISTENT, mode, n, net,
                 **{k: v for k, v in kw.items() if k != "wave_passes"})
    b, sb = _run(G, pdf, G.GAPS_SCHED_WAVE, mode, n, net, **kw)
    if learned and n > 1:
        assert sa["violations"] > 0 and sa["mlp_tiles"] > 0
    if kw.get("nmax"):
        assert sa["err_capacity"] > 0
    if kw.get("max_cycles"):
        assert sa["err_iter_cap"] > 0
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    for k in COUNTERS:
        assert sa[k] == sb[k], k
