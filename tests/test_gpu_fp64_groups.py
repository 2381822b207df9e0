"""The FP64 shower's eight-lane groups at the edges of their launch: events that
fill a group, a warp, a block and a block's share exactly or with one left
over, two calls of one context at a time, and colour tags that do not fit a
byte. FP64 results do not depend on the launch, so every comparison is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

MOST = 100_000


def _events(G, torch, ctx, first, n, buf=None, stream=None):
    buf = buf or G.EventBuffers.allocate(n, 128)
    G.gaps_generate_hard(ctx, first, n, buf.view(), stream)
    G.gaps_shower(ctx, first, n, buf.view(), stream)
    return buf


def _same(a, b):
    for k in a:
        assert np.array_equal(a[k], b[k]), k


@pytest.fixture(scope="module")
def setup():
    torch = pytest.importorskip("torch")
    from paper_2511_19633_gb300 import gaps as G, inputs
    pdf = inputs.synthetic_pdf_grid()
    ctx = G.gaps_init(G.make_config(G.GAPS_PP_Z_LO, 13600.0, pdf_grid=pdf, nmax=128))
    whole = _events(G, torch, ctx, 0, MOST).to_host(MOST)
    yield G, torch, ctx, whole
    G.gaps_destroy(ctx)


@pytest.mark.parametrize("n", [1, 4, 5, 15, 16, 17, 609, 9728, 9729, 77825])
def test_launch_sizes(setup, n):
    """events first .. first + n - 1 of any launch are those of one large launch"""
    G, torch, ctx, whole = setup
    first = 7
    got = _events(G, torch, ctx, first, n).to_host(n)
    _same(got, {k: v[first:first + n] for k, v in whole.items()})


def test_two_streams(setup):
    """two calls of one context in flight at a time share the scratch pool"""
    G, torch, ctx, whole = setup
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    bufs = [G.EventBuffers.allocate(20_000, 128) for _ in streams]
    torch.cuda.synchronize()
    for k, s in enumerate(streams):
        _events(G, torch, ctx, 20_000 * k, 20_000, bufs[k], s)
    torch.cuda.synchronize()
    for k, b in enumerate(bufs):
        _same(b.to_host(20_000), {q: v[20_000 * k:20_000 * (k + 1)] for q, v in whole.items()})


def test_wide_colour_tags(setup):
    """tags beyond 255 only rename the colour lines of the hard event"""
    G, torch, ctx, whole = setup
    n = 2000
    buf = G.EventBuffers.allocate(n, 128)
    G.gaps_generate_hard(ctx, 0, n, buf.view())
    for t in (buf.col, buf.acol):
        t += 70_000 * (t != 0).int()
    G.gaps_shower(ctx, 0, n, buf.view())
    got = buf.to_host(n)
    for k in ("p", "flav", "npart", "status", "n_emit", "weight", "t", "eta"):
        assert np.array_equal(got[k], whole[k][:n]), k
    for k in ("col", "acol"):
        assert np.array_equal(np.where(got[k] > 70_000, got[k] - 70_000, got[k]), whole[k][:n]), k
