"""The FP32 SIMT convolution at the edges of its tiles (32 x 4 or 32 x 16
pixels, 64 or 16 output channels, 4 input channels per stage; 16-byte and
single loads and stores), against the float64 convolution: the error of a chain
of K = 9 cin fused multiply-adds and the bias is at most (K + 1) 2^-24 of the sum of
|terms|.  Inputs that are not a number or infinite reach exactly the outputs
whose window holds them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mrs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2106_12802_gb300 as m
    m.load()
    return m


CASES = [(1, 1, 1, 1, 1), (2, 3, 5, 3, 3), (1, 4, 32, 4, 16), (1, 5, 33, 5, 17), (2, 15, 31, 9, 64),
         (1, 17, 65, 12, 64), (3, 16, 40, 64, 3), (1, 9, 100, 21, 65), (1, 8, 34, 64, 64), (1, 6, 37, 130, 128),
         (1, 7, 64, 18, 256)]


@pytest.mark.parametrize("N,H,W,cin,cout", CASES)
def test_tile_edges(mrs, N, H, W, cin, cout):
    r = np.random.default_rng(H * 1000 + W)
    x = torch.from_numpy(r.normal(size=(N, H, W, cin)).astype(np.float32)).cuda()
    w = r.normal(size=(cout, 3, 3, cin)).astype(np.float32)
    b = r.normal(size=cout).astype(np.float32)
    y = mrs.conv3x3(x, w, b, False, "fp32")
    xd, wd = x.double().permute(0, 3, 1, 2), torch.from_numpy(w).cuda().double().permute(0, 3, 1, 2)
    bd = torch.from_numpy(b).cuda().double()
    ref = torch.nn.functional.conv2d(xd, wd, bd, padding=1).permute(0, 2, 3, 1)
    terms = torch.nn.functional.conv2d(xd.abs(), wd.abs(), bd.abs(), padding=1).permute(0, 2, 3, 1)
    assert ((y.double() - ref).abs() <= (9 * cin + 1) * 2.0 ** -24 * terms + 1e-30).all()


def test_not_finite_inputs_stay_in_their_windows(mrs):
    r = np.random.default_rng(3)
    x = torch.from_numpy(r.normal(size=(1, 12, 70, 6)).astype(np.float32)).cuda()
    w = np.abs(r.normal(size=(20, 3, 3, 6))).astype(np.float32) + 0.1
    clean = mrs.conv3x3(x, w, np.zeros(20, np.float32), False, "fp32")
    x[0, 5, 33, 2] = float("nan")
    x[0, 9, 2, 5] = float("inf")
    y = mrs.conv3x3(x, w, np.zeros(20, np.float32), False, "fp32")
    nan, inf = torch.zeros_like(y, dtype=torch.bool), torch.zeros_like(y, dtype=torch.bool)
    nan[0, 4:7, 32:35] = True
    inf[0, 8:11, 1:4] = True
    assert torch.equal(y.isnan(), nan) and torch.equal(y == float("inf"), inf)
    assert torch.equal(y[~(nan | inf)], clean[~(nan | inf)])
