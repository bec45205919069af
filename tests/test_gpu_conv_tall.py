"""The FP32 convolution on images of more rows of blocks than a grid's y and z
dimensions hold (65,535: of 4 pixel rows where more than 16 channels come out, of
16 elsewhere), and as wide ones, against the float64 convolution with the bound of
a chain of K = 9 cin fused multiply-adds and the bias: (K + 1) 2^-24 of the sum of
|terms|."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,cout", [(4 * 65535 + 1, 2, 64), (300000, 1, 17), (16 * 65535 + 1, 1, 3), (1, 300001, 64)])
def test_tall_and_wide_images(H, W, cout):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2106_12802_gb300 as mrs
    r = np.random.default_rng(H + W)
    cin = 4
    x = torch.from_numpy(r.normal(size=(1, H, W, cin)).astype(np.float32)).cuda()
    w = r.normal(size=(cout, 3, 3, cin)).astype(np.float32)
    b = r.normal(size=cout).astype(np.float32)
    y = mrs.conv3x3(x, w, b, False, "fp32").double()
    # the float64 convolution as a product of the nine shifted images
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1))
    cols = torch.cat([xp[:, i:i + H, j:j + W] for i in range(3) for j in range(3)], 3)
    wd, bd = (torch.from_numpy(a).cuda().double() for a in (w.reshape(cout, -1), b))
    ref = cols @ wd.T + bd
    terms = cols.abs() @ wd.abs().T + bd.abs()
    assert ((y - ref).abs() <= (9 * cin + 1) * 2.0 ** -24 * terms + 1e-30).all()
