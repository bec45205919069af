"""The BF16 weight gradient of one layer, whose launch deals the classes (or their
halves, up to half as many as SMs) to the CTAs: at numbers of jobs around 76 and 152,
at one and at several per class, with channels that fill the tile and not.
Operands are small whole numbers, so that every sum is exact in FP32."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,W", [(1, 1, 1), (1, 75, 64), (2, 38, 20), (7, 11, 64), (1, 151, 3), (4, 38, 64),
                                   (1, 153, 64), (3, 51, 65), (2, 152, 130)])
@pytest.mark.parametrize("cin,cout", [(64, 64), (5, 33)])
def test_classes_and_halves(N, H, W, cin, cout):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2106_12802_gb300 as mrs
    r = np.random.default_rng(H + W)
    x = torch.from_numpy(r.integers(-3, 4, (N, H, W, cin)).astype(np.float32)).cuda()
    dy = torch.from_numpy(r.integers(-3, 4, (N, H, W, cout)).astype(np.float32)).cuda()
    dw, db = mrs.conv3x3_wgrad(x, dy, precision="bf16")
    xp = torch.nn.functional.pad(x.double(), (0, 0, 1, 1, 1, 1))
    ref = torch.stack([torch.einsum("nhwo,nhwc->oc", dy.double(), xp[:, i:i + H, j:j + W])
                       for i in range(3) for j in range(3)], 1).reshape(cout, 3, 3, cin)
    assert np.array_equal(dw, ref.cpu().numpy())
    assert np.array_equal(db, dy.double().sum((0, 1, 2)).cpu().numpy())
