"""The targets of the learned bound at the edges of their launch: states in one
call, which fills the GPU with all bins of a channel in a warp, against the same
states in calls that take one bin a warp. A target does not depend on the
launch, so the comparison is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", params=[False, True], ids=["light", "thresholds"])
def setup(request):
    torch = pytest.importorskip("torch")
    from paper_2511_19633_gb300 import gaps as G, inputs
    pdf = inputs.synthetic_pdf_grid(thresholds=request.param)
    ctx = G.gaps_init(G.make_config(G.GAPS_PP_Z_NLO, 13600.0, pdf_grid=pdf, precision=G.GAPS_MIXED))
    n = 64 * torch.cuda.get_device_properties(0).multi_processor_count * 8
    rng = np.random.default_rng(3)
    eta = np.exp(rng.uniform(np.log(1e-5), np.log(0.99), n))
    s = np.exp(rng.uniform(np.log(0.5), np.log(1e7), n))
    states = np.stack([eta, s, rng.integers(2, 4, n), rng.integers(0, 11, n)], axis=1).astype(np.float32)
    states = torch.from_numpy(states).cuda()
    yield G, torch, ctx, states, _targets(G, torch, ctx, states)
    G.gaps_destroy(ctx)


def _targets(G, torch, ctx, states):
    n = len(states)
    feats = torch.full((16 * n, 4), float("nan"), dtype=torch.float32, device="cuda")
    targets = torch.full((16 * n,), float("nan"), dtype=torch.float32, device="cuda")
    G.gaps_isr_targets(ctx, states, n, feats, targets)
    return feats, targets


@pytest.mark.parametrize("n", [1, 2, 31, 607, 2000])
def test_targets_of_part_of_the_states(setup, n):
    G, torch, ctx, states, (feats, targets) = setup
    assert torch.isfinite(targets).all() and torch.isfinite(feats).all()
    first = 1001
    f, t = _targets(G, torch, ctx, states[first:first + n].contiguous())
    assert torch.equal(f, feats[16 * first:16 * (first + n)])
    assert torch.equal(t, targets[16 * first:16 * (first + n)])
