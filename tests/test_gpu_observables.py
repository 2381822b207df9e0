"""Observables of events that share a warp against the same events one a warp:
launches of few events and of many, events with more pseudo-jets than a quarter
of a warp's shared memory holds, both precisions. An observable does not depend
on the launch, so the comparison is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MOST = 160_000


def _run(G, torch, ctx, first, n):
    buf = G.EventBuffers.allocate(n, 128)
    G.gaps_generate_hard(ctx, first, n, buf.view())
    G.gaps_shower(ctx, first, n, buf.view())
    obs = torch.full((G.GAPS_NOBS, n), float("nan"), dtype=torch.float64, device="cuda")
    G.gaps_observables(ctx, first, n, buf.view(), obs, None)
    return buf, obs


@pytest.fixture(scope="module", params=[("ee", 0), ("pp", 0), ("ee", 1), ("pp", 1), ("mix", 1)],
                ids=lambda p: f"{p[0]}-{'mixed' if p[1] else 'fp64'}")
def setup(request):
    torch = pytest.importorskip("torch")
    from paper_2511_19633_gb300 import gaps as G, inputs
    name, precision = request.param
    process, sqrt_s = (0, 500.0) if name == "ee" else (2, 13600.0)
    kw = {"mix": [(2, 13600.0, 1.0, 0.5), (0, 91.2, 0.5, 0.5)]} if name == "mix" else {}
    pdf = inputs.synthetic_pdf_grid()
    ctx = G.gaps_init(G.make_config(process, sqrt_s, pdf_grid=pdf, nmax=128, precision=precision,
                                    schedule=G.GAPS_SCHED_PERSISTENT, **kw))
    n = MOST if precision else 30_000
    buf, obs = _run(G, torch, ctx, 0, n)
    yield G, torch, ctx, int(buf.npart.max()), obs
    G.gaps_destroy(ctx)


@pytest.mark.parametrize("first,n", [(0, 1), (5, 31), (40, 1500), (2000, 12_001)])
def test_launch_sizes(setup, first, n):
    G, torch, ctx, largest, whole = setup
    assert not torch.isnan(whole[:4]).any()
    assert largest > 16
    _, got = _run(G, torch, ctx, first, n)
    assert torch.equal(torch.nan_to_num(got), torch.nan_to_num(whole[:, first:first + n]))
