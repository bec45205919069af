"""The L1-log training loss of dark images and of images against themselves: every
value's error is a few roundings of its own magnitude (8 x 2^-53 of |y| + |t|), however
close it is to its target, and an image equal to its target has loss 0.

Zero weights at scale 1 make the network's image its LRHS."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [1e-8, 1e-6, 1e-5, 2.0 ** -20, 9e-4])
@pytest.mark.parametrize("apart", [0.0, 1e-7, 1e-4, 1.0])
def test_dark_images(size, apart):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2106_12802_gb300 as mrs
    from paper_2106_12802_gb300 import fusion
    r = np.random.default_rng(1)
    y = (size * r.uniform(0.2, 1.0, (1, 120, 100, 3))).astype(np.float32)
    t = np.clip(y * (1 + apart * r.normal(size=y.shape)), -size, size).astype(np.float32)
    net = mrs.Net(np.zeros(fusion.NPARAMS, np.float32))
    im = [torch.from_numpy(a).cuda() for a in (y, y, y, y, t)]
    v = mrs.train_step(net, *im, 1, lr=0.0, precision="fp32", loss="l1log")
    y, t = y.astype(np.longdouble), t.astype(np.longdouble)
    ref = np.abs(np.sign(y) * np.log1p(np.abs(y)) - np.sign(t) * np.log1p(np.abs(t))).mean()
    if not apart:
        assert v == 0.0
    assert abs(v - ref) <= 8 * 2.0 ** -53 * (np.abs(y) + np.abs(t)).mean() + 1e-15 * ref
