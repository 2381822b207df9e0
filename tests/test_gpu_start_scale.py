"""Starting scales that bound nothing: a record whose t is infinite, above every
FP32 number or not a number showers from its dipoles' kinematic limits, in both
precisions, and one at or below the cutoff does not shower."""
import numpy as np
import pytest

from tests.gpu_common import gaps

pytestmark = pytest.mark.gpu


def _shower(G, pdf, precision, value, n=3000):
    import torch
    ctx = G.gaps_init(G.make_config(2, 13600.0, pdf_grid=pdf, nmax=128, precision=precision))
    try:
        buf = G.EventBuffers.allocate(n, 128)
        G.gaps_generate_hard(ctx, 0, n, buf.view())
        buf.t[:] = value
        G.gaps_shower(ctx, 0, n, buf.view())
        torch.cuda.synchronize()
        out = buf.to_host(n)
        out["draw"] = buf.draw[:n].cpu().numpy()
        return out
    finally:
        G.gaps_destroy(ctx)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), 1e300])
def test_scales_that_bound_nothing(pdf, precision, value):
    G = gaps()
    a, b = _shower(G, pdf, precision, 1e30), _shower(G, pdf, precision, value)
    assert a["n_emit"].mean() > 5 and np.all(a["status"] == 1)
    for k in a:
        assert np.array_equal(a[k], b[k]), k


@pytest.mark.parametrize("precision", [0, 1])
def test_cutoff_as_the_scale(pdf, precision):
    G = gaps()
    assert not _shower(G, pdf, precision, 0.5)["n_emit"].any()
