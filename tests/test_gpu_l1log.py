"""The L1-log training loss against float64, over magnitudes, signs and ties.

The network's weights are zero, so its image is the last layer's bias and the
targets choose every pair (y, t).  A value's error is a few roundings of 1 + |x|
and of the running products (each 2^-53), whatever its size; where both
magnitudes are tiny the error is relative.
"""
import numpy as np
import pytest
import torch

import paper_2106_12802_gb300 as mrs
from oracle import rdn as ordn

pytestmark = pytest.mark.gpu
CLIP = 100.0


def _slog(x):
    return np.sign(x) * np.log1p(np.abs(x))


@pytest.mark.parametrize("N,h,w,bias,lo,hi", [
    (1, 1, 1, (1e-7, -0.37, 3.1e4), -12, 30),
    (1, 5, 7, (0.0, -2.0 ** -20, 2.0 ** -20), -9, -4),
    (3, 37, 29, (1e-9, -3e-8, 5e-7), -12, -6.1),
    (2, 96, 80, (0.6, -1e30, 2.0 ** -29), -12, 38),
])
def test_l1log_loss_and_gradient(N, h, w, bias, lo, hi):
    s = 4
    H, W = h * s, w * s
    rng = np.random.default_rng(N + h)
    t = (rng.choice([-1.0, 1.0], (N, H, W, 3)) * 10.0 ** rng.uniform(lo, hi, (N, H, W, 3))).astype(np.float32)
    b = np.asarray(bias, np.float32)
    kind = rng.integers(0, 8, t.shape)
    t = np.where(kind == 0, np.broadcast_to(b, t.shape), np.where(kind == 1, np.float32(0.0), t)).astype(np.float32)
    L = [(wt * 0.0, bs * 0.0) for wt, bs in ordn.unpack(ordn.kaiming(1, s), s)]
    L[-1] = (L[-1][0], b.astype(np.float64))
    net = mrs.RDN(ordn.pack(L).astype(np.float32), s)
    img = lambda *sh: torch.zeros(sh, device="cuda")
    y = torch.empty((N, H, W, 3), device="cuda")
    v = net.train_step(img(N, h, w, 3), img(N, H, W, 3), img(N, H, W, 3), img(N, H, W, 3),
                       torch.from_numpy(t).cuda(), lr=0.0, loss="l1log", out=y, precision="fp32")
    db = net.get_grads()[-3:].astype(np.float64)
    net.close()
    assert np.array_equal(y.cpu().numpy(), np.broadcast_to(b, t.shape))
    y64 = np.broadcast_to(b, t.shape).astype(np.float64)
    t64 = np.minimum(t, np.float32(CLIP)).astype(np.float64)
    d = _slog(y64) - _slog(t64)
    ref = np.abs(d).mean()
    tiny = max(np.abs(y64).max(), np.abs(t64).max()) < 2.0 ** -20
    assert abs(v - ref) <= 1e-12 * ref + (0.0 if tiny else 1e-15)
    g = np.sign(y64 - t64) / (1.0 + np.abs(y64)) / d.size
    assert np.all(np.abs(db - g.sum((0, 1, 2))) <= 1e-5 * np.abs(g).sum((0, 1, 2)))
