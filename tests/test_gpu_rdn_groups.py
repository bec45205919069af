"""The two-encoder network's BF16 step where its grouped launches are at their
edges: fewer tiles than CTAs a group, one-pixel images, widths around the point
where a tile holds one image or several, 5, 17 and 65 convolutions a launch.

Bounds as in test_gpu_rdn_train.py's BF16 step (the same comparison): a wrong
group, map, mask or weight row turns a layer's gradient."""
import numpy as np
import pytest

from oracle import rdn as ordn
from test_gpu_rdn_train import _batch, _cuda, _f64, _params, cnn, mrs  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("s,N,h,w", [(8, 1, 1, 1), (8, 3, 1, 2), (2, 1, 3, 63), (2, 2, 3, 62), (4, 3, 5, 21),
                                     (4, 1, 2, 130)])
def test_grouped_launches_at_their_edges(mrs, s, N, h, w):  # noqa: F811
    lr, hr, alb, nrm, _, tgt = _batch(300 + s * 10 + w, N, h, w, s, 9)
    p = _params(s + 1, s, 9)
    net = mrs.RDN(p, s, 9)
    v = net.train_step(*_cuda(lr, hr, alb, nrm, tgt), lr=0.0, loss="l1log", precision="bf16")
    g = net.get_grads().astype(np.float64)
    again = net.train_step(*_cuda(lr, hr, alb, nrm, tgt), lr=0.0, loss="l1log", precision="bf16")
    assert again == v and np.array_equal(net.get_grads().astype(np.float64), g)
    net.close()
    p64 = p.astype(np.float64)
    ry, tape = ordn.forward_tape(p64, *[_f64(a) for a in (lr, hr, alb, nrm)], s, None)
    rv, rdy = cnn.loss_fn(ry, np.minimum(_f64(tgt), 100.0), "l1log")
    rg = ordn.backward(p64, tape, rdy)
    assert abs(v - rv) <= 5e-2 * rv
    for name, wo, bo, k, ci, co in ordn.layer_offsets(s, 9):
        ref, got = rg[wo:bo], g[wo:bo]
        cos = got @ ref / (np.linalg.norm(got) * np.linalg.norm(ref) + 1e-30)
        rel = np.linalg.norm(got - ref) / (np.linalg.norm(ref) + 1e-30)
        assert cos > 0.95 and rel < 0.35, (name, cos, rel)
