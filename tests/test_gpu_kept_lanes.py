"""The kept-trial shower against the lane kernel, which shares neither its phases
nor its lists with it: the learned proposal with a network whose heights fail
often (the violation and its plain-bound fallback) and with a trained one, the
heavy-quark measure, tables that depend on Q^2, the fitted PDF-ratio bound,
mixed batches, records that fill up and cycle caps. Both run through one context,
every record and every counter of the events is compared exactly."""
import ctypes

import numpy as np
import pytest

from tests.gpu_common import gaps

pytestmark = pytest.mark.gpu

MIX = [(2, 13600.0, 1.0, 0.5), (0, 91.2, 0.5, 0.25), (3, 13600.0, 4.0, 0.25)]
RECORD = ("p", "flav", "col", "acol", "npart", "status", "n_emit", "weight", "t", "eta", "draw")
COUNTERS = ("events", "steps", "trials", "isr_trials", "vetoes", "accepts", "violations", "err_capacity",
            "err_iter_cap", "err_numeric", "rebuilds", "mlp_tiles")


@pytest.fixture(scope="module")
def G():
    return gaps()


@pytest.fixture(scope="module")
def tables():
    from paper_2511_19633_gb300 import inputs
    flat = inputs.synthetic_pdf_grid()
    nq = flat.shape[2]
    return {"flat": flat, "thresholds": inputs.synthetic_pdf_grid(thresholds=True),
            # every density rises with Q^2, the gluon's the least
            "scale": flat * np.linspace(1.0, [[1.2]] + [[1.5]] * 10, nq, axis=2).astype(np.float32)}


@pytest.fixture(scope="module")
def nets(G, tables):
    """(parameters, margins): untrained with no margin, and trained"""
    from paper_2511_19633_gb300 import learned
    ctx = G.gaps_init(G.make_config(2, 13600.0, pdf_grid=tables["flat"], nmax=128, precision=G.GAPS_MIXED,
                                    schedule=G.GAPS_SCHED_PERSISTENT))
    try:
        r = learned.train_and_install(ctx, n_events=1 << 16, capacity=1 << 15, holdout_events=1 << 16,
                                      holdout_capacity=1 << 15, steps=2000, min_rows=256)
    finally:
        G.gaps_destroy(ctx)
    zero = np.zeros((G.GAPS_ISR_CLASSES, G.GAPS_ISR_ETA_BINS, G.GAPS_ISR_BINS), dtype=np.float32)
    return {"untrained": (learned.init_params(5), zero), "trained": (r["params"], r["log_margins"])}


def _pair(G, grid, process, n, net=None, fit=None, **kw):
    import torch
    nmax = kw.pop("nmax", 128)
    ctx = G.gaps_init(G.make_config(process, 91.2 if process == 0 else 13600.0, pdf_grid=grid, nmax=nmax, seed=3,
                                    precision=G.GAPS_MIXED, **kw))
    out = []
    try:
        if net is not None:
            G.gaps_set_learned_proposal(ctx, *net)
        if fit is not None:
            G.gaps_set_pdf_ratio_fit(ctx, fit)
        vlog = torch.zeros((1 << 18, 8), dtype=torch.float32, device="cuda")
        vcount = torch.zeros(1, dtype=torch.int64, device="cuda")
        G.gaps_set_violation_log(ctx, vlog, vcount)
        for lanes in (True, False):
            buf = G.EventBuffers.allocate(n, nmax)
            ev = buf.view()
            vcount.zero_()
            G.gaps_generate_hard(ctx, 1 << 33, n, ev)
            G.gaps_reset_stats(ctx)
            if lanes:
                stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
                assert G.library().gaps_test_shower_lanes(ctx, ctypes.c_uint64(1 << 33), ctypes.c_uint64(n),
                                                          ctypes.byref(ev), stream) == 0
            else:
                G.gaps_shower(ctx, 1 << 33, n, ev)
            torch.cuda.synchronize()
            rec = buf.to_host(n)
            rec["draw"] = buf.draw[:n].cpu().numpy()
            log = vlog[:int(vcount.item())].cpu().numpy()
            out.append((rec, G.gaps_get_stats(ctx), log[np.lexsort(log.T)]))
    finally:
        G.gaps_destroy(ctx)
    return out


def _same(a, b):
    for k in RECORD:
        assert np.array_equal(a[0][k], b[0][k]), k
    for k in COUNTERS:
        assert a[1][k] == b[1][k], k
    assert np.array_equal(a[2], b[2])


@pytest.mark.parametrize("schedule", [1, 3])
@pytest.mark.parametrize("table,process,net,kw", [
    ("flat", 2, "untrained", {}),
    ("flat", 2, "trained", {}),
    ("thresholds", 2, None, {}),
    ("thresholds", 2, "untrained", {}),
    ("scale", 2, None, {}),
    ("scale", 3, "untrained", {}),
    ("flat", 1, "untrained", {"t_cut": 0.5}),
    ("flat", 0, "untrained", {"mix": MIX}),
    ("thresholds", 0, "trained", {"mix": MIX}),
    ("flat", 2, "untrained", {"nmax": 9}),
    ("flat", 2, "untrained", {"max_cycles": 29}),
])
def test_kept_trials_equal_the_lane_kernel(G, tables, nets, schedule, table, process, net, kw):
    a, b = _pair(G, tables[table], process, 20_011, nets.get(net), schedule=schedule, **kw)
    if net == "untrained":
        assert a[1]["violations"] == len(a[2]) > 1000 and a[1]["mlp_tiles"] > 0
    if kw.get("nmax"):
        assert a[1]["err_capacity"] > 100
    if kw.get("max_cycles"):
        assert a[1]["err_iter_cap"] > 1000
    _same(a, b)


@pytest.mark.parametrize("net", [None, "untrained"])
def test_fitted_bound_equals_the_lane_kernel(G, tables, nets, net):
    fit = np.full((12, 12, 2), 1.3, dtype=np.float32)
    a, b = _pair(G, tables["flat"], 2, 20_011, nets.get(net), fit, schedule=G.GAPS_SCHED_WAVE)
    assert a[1]["violations"] == len(a[2]) > 1000
    _same(a, b)
