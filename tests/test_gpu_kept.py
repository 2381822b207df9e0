"""The kept-trial shower at the edges of its launch: numbers of events that
fill a block's slots or the grid exactly, or one less or more, events with more
ends than the phases keep in shared memory, records that fill up, records that
are not to be showered. The reference is the warp of events per launch that
gaps_collect_pdf_ratios runs (certified bounds, the same random numbers), so
every comparison is exact."""
import numpy as np
import pytest

from tests.gpu_common import gaps

pytestmark = pytest.mark.gpu

SLOTS = 192  # events in flight per SM


@pytest.fixture(scope="module")
def G():
    return gaps()


def _pair(G, pdf, process, sqrt_s, first, n, mark=None, **kw):
    import torch
    uses_pdf = process != 0 or any(r[0] for r in kw.get("mix") or [])
    nmax = kw.pop("nmax", 128)
    schedule = kw.pop("schedule", G.GAPS_SCHED_PERSISTENT)
    cfg = G.make_config(process, sqrt_s, pdf_grid=pdf if uses_pdf else None, nmax=nmax, seed=1,
                        precision=G.GAPS_MIXED, schedule=schedule, **kw)
    ctx = G.gaps_init(cfg)
    out = []
    try:
        for reference in (True, False):
            buf = G.EventBuffers.allocate(n, nmax)
            ev = buf.view()
            G.gaps_generate_hard(ctx, first, n, ev)
            if mark is not None:
                buf.status[mark] = 1
            G.gaps_reset_stats(ctx)
            if reference:
                samples = torch.empty((1, 4), dtype=torch.float32, device="cuda")
                count = torch.zeros(1, dtype=torch.int64, device="cuda")
                G.gaps_collect_pdf_ratios(ctx, first, n, ev, samples, count, keep_fraction=1e-9)
            else:
                G.gaps_shower(ctx, first, n, ev)
            torch.cuda.synchronize()
            rec = buf.to_host(n)
            rec["stats"] = G.gaps_get_stats(ctx)
            out.append(rec)
    finally:
        G.gaps_destroy(ctx)
    return out


def _same(a, b):
    for k in ("p", "flav", "col", "acol", "npart", "status", "n_emit", "weight", "t", "eta"):
        assert np.array_equal(a[k], b[k]), k
    for k in ("events", "steps", "trials", "isr_trials", "vetoes", "accepts", "violations", "err_capacity",
              "err_iter_cap", "err_numeric"):
        assert a["stats"][k] == b["stats"][k], k


@pytest.mark.parametrize("per_sm,more", [(0, 1), (1, -1), (1, 0), (1, 1), (2, 1), (SLOTS, -1), (SLOTS, 0),
                                         (SLOTS, 1), (2 * SLOTS, 3)])
def test_launch_sizes(G, pdf, per_sm, more):
    import torch
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + more
    a, b = _pair(G, pdf, 2, 13600.0, 4_000_000_007, n)
    _same(a, b)


@pytest.mark.parametrize("schedule", ["PERSISTENT", "WAVE"])
@pytest.mark.parametrize("process,sqrt_s,nmax,kw", [
    (2, 13600.0, 128, {"t_cut": 0.5}),  # more than 64 ends
    (2, 13600.0, 9, {}),                # records that fill up, an odd number of slots
    (0, 500.0, 17, {}),
    (3, 13600.0, 33, {"t_cut": 0.5}),
    (2, 13600.0, 128, {"max_cycles": 13}),  # a cap inside a round of eight cycles
    (0, 91.2, 128, {"mix": [(2, 13600.0, 1.0, 0.5), (0, 91.2, 0.5, 0.25), (3, 13600.0, 4.0, 0.25)]}),
])
def test_sizes_of_events(G, pdf, schedule, process, sqrt_s, nmax, kw):
    a, b = _pair(G, pdf, process, sqrt_s, 99, 30_011, nmax=nmax, schedule=getattr(G, "GAPS_SCHED_" + schedule), **kw)
    if kw.get("t_cut") and nmax > 64:
        assert int(a["npart"].max()) > 32
    _same(a, b)


def test_inactive_records(G, pdf):
    """records whose shower has already ended are passed over"""
    mark = slice(None, None, 3)
    a, b = _pair(G, pdf, 2, 13600.0, 5, 20_000, mark=mark)
    assert not a["n_emit"][mark].any()
    _same(a, b)
