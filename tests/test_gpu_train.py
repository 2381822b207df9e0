"""One step of the network's training (gaps_mlp_train, a cluster of eight blocks
that share the batch's rows and the weights) against FP64: the batch is drawn
with replacement, so tables of one row, fewer rows than a batch and many rows
all fill it. The FP32 sums run over at most 256 rows, 64 inputs and three
layers: an entry's error is below 512 roundings (512 x 2^-24) of the sum of its
terms' magnitudes, and the moments add one more to their own magnitude."""
import numpy as np
import pytest

from tests.gpu_common import gaps

pytestmark = pytest.mark.gpu

EPS = 512 * 2.0 ** -24


def _philox(c0, c1, c2, c3, k0, k1):
    m, sh = np.uint64(0xFFFFFFFF), np.uint64(32)
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c0, np.uint64(0xCD9E8D57) * c2
        c0, c1, c2, c3 = (p1 >> sh) ^ c1 ^ np.uint64(k0), p1 & m, (p0 >> sh) ^ c3 ^ np.uint64(k1), p0 & m
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c0, c1


def _batch(n, seed):
    z, tid = np.zeros(256, dtype=np.uint64), np.arange(256, dtype=np.uint64)
    lo, hi = _philox(z, z, tid, z + np.uint64(0x5EED), seed & 0xFFFFFFFF, seed >> 32)
    return (((hi << np.uint64(32)) | lo) % np.uint64(n)).astype(np.int64)


def _gradient(p, x, t, tau):
    """FP64 gradient of the batch's loss, and the sums of the terms' magnitudes"""
    w1, b1, w2, b2, w3, b3 = np.split(p, np.cumsum([256, 64, 4096, 64, 64]))
    w1, w2 = w1.reshape(64, 4), w2.reshape(64, 64)
    h1 = np.maximum(x @ w1.T + b1, 0.0)
    h2 = np.maximum(h1 @ w2.T + b2, 0.0)
    r = h2 @ w3 + b3[0] - t
    w = np.where(r < 0.0, tau, 1.0 - tau)
    dy = 2.0 * w * r / 256
    mag = 2.0 * w * (np.abs(h2) @ np.abs(w3) + np.abs(b3[0]) + np.abs(t)) / 256  # of dy's terms
    on1, on2 = h1 > 0.0, h2 > 0.0
    d2, m2 = on2 * dy[:, None] * w3, on2 * mag[:, None] * np.abs(w3)
    d1, m1 = on1 * (d2 @ w2), on1 * (m2 @ np.abs(w2))
    cat = lambda a, b, e, f: np.concatenate([(a.T @ f(x)).ravel(), a.sum(0), (b.T @ h1).ravel(), b.sum(0), e @ h2, [e.sum()]])
    return cat(d1, d2, dy, lambda v: v), cat(m1, m2, mag, np.abs), np.sum(w * r * r) / 256


@pytest.mark.parametrize("n,resume", [(1, False), (31, True), (257, False), (70001, True)])
def test_one_step(n, resume):
    import torch
    from paper_2511_19633_gb300 import learned
    G = gaps()
    rng = np.random.default_rng(n)
    seed, tau, lr = (5 << 32) + 9, 0.9, 2e-3
    p = learned.init_params(3)
    x = rng.uniform(-1, 1, (n, 4)).astype(np.float32)
    t = rng.normal(-2, 1, n).astype(np.float32)
    m0 = (0.01 * rng.normal(size=p.size) if resume else np.zeros(p.size)).astype(np.float32)
    v0 = (0.01 * rng.uniform(0.5, 1, p.size) if resume else np.zeros(p.size)).astype(np.float32)
    P, m, v = (torch.from_numpy(a.copy()).cuda() for a in (p, m0, v0))
    loss = torch.zeros(1, device="cuda")
    G.gaps_mlp_train(P, m, v, torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), 1, lr, tau, seed, loss, 1)
    rows = _batch(n, seed)
    g, mag, ref = _gradient(p.astype(np.float64), x[rows].astype(np.float64), t[rows].astype(np.float64),
                            float(np.float32(tau)))
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    m1, v1 = b1 * m0 + (1 - b1) * g, b2 * v0 + (1 - b2) * g * g
    em = (1 - b1) * EPS * mag + 2.0 ** -22 * (np.abs(m0) + np.abs(g))
    ev = (1 - b2) * (2 * np.abs(g) * EPS * mag + (EPS * mag) ** 2) + 2.0 ** -22 * (np.abs(v0) + g * g)
    gm, gv, gp = (a.cpu().numpy().astype(np.float64) for a in (m, v, P))
    assert np.all(np.abs(gm - m1) <= em)
    assert np.all(np.abs(gv - v1) <= ev)
    # the update from the moments that came out
    step = lr * (gm / (1 - b1)) / (np.sqrt(gv / (1 - b2)) + 1e-8)
    assert np.all(np.abs(gp - (p - step)) <= 2.0 ** -20 * (np.abs(step) + 2.0 ** -3 * np.abs(p)))
    assert abs(loss.item() - ref) <= 1e-4 * ref


def test_no_steps():
    import torch
    from paper_2511_19633_gb300 import learned
    G = gaps()
    p = torch.from_numpy(learned.init_params(3)).cuda()
    a, z = p.clone(), torch.zeros_like(p)
    G.gaps_mlp_train(a, z, z.clone(), torch.ones((4, 4), device="cuda"), torch.ones(4, device="cuda"), 0, 1e-3, 0.5, 1)
    assert torch.equal(a, p) and not z.any()
