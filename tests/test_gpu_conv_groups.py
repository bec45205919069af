"""The FP32 convolution of 17 to 32 output channels, which large images compute in
groups of 16 and small ones in one of 64: on either side of the line (a block of 32 x 4
pixels an SM), each output bit for bit as the same channel of 64."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,W", [(1, 9, 40), (1, 128, 128), (1, 150, 131), (4, 152, 33), (3, 64, 260), (2, 611, 31)])
@pytest.mark.parametrize("cin,cout", [(64, 32), (21, 17), (6, 25)])
def test_groups_of_16_equal_groups_of_64(N, H, W, cin, cout):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2106_12802_gb300 as mrs
    r = np.random.default_rng(cin)
    x = torch.from_numpy(r.normal(size=(N, H, W, cin)).astype(np.float32)).cuda()
    w = r.normal(size=(64, 3, 3, cin)).astype(np.float32)
    b = r.normal(size=64).astype(np.float32)
    for relu in (False, True):
        whole = mrs.conv3x3(x, w, b, relu, "fp32")
        part = mrs.conv3x3(x, w[:cout], b[:cout], relu, "fp32")
        assert torch.equal(part, whole[..., :cout])
