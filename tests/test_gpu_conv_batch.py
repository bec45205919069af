"""Tensor-core convolutions of a batch of narrow images, several to a tile,
against the same images one at a time (one to a tile): bit for bit, since a
pixel's accumulation order does not depend on its row of the tile.  Widths at
the edges of 1, 2, 3 and many images a tile, batches that leave the last tile
part empty."""
import numpy as np
import pytest
import torch

import paper_2106_12802_gb300 as mrs

pytestmark = pytest.mark.gpu
SHAPES = [(2, 5, 62), (3, 5, 62), (2, 5, 63), (5, 7, 41), (7, 3, 40), (16, 48, 48), (9, 4, 13), (50, 2, 1),
          (130, 1, 1), (3, 1, 2)]


def _images(seed, *shape):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda")


@pytest.mark.parametrize("N,H,W", SHAPES)
@pytest.mark.parametrize("precision,cin,cout", [("bf16", 64, 64), ("bf16", 9, 3), ("bf16", 200, 64), ("fp8", 64, 64),
                                                ("fp8", 64, 3)])
def test_conv_of_a_batch_is_each_images(N, H, W, precision, cin, cout):
    rng = np.random.default_rng(W)
    x = _images(1, N, H, W, cin)
    x[:, 0, 0, 0] = 7.0                                   # one FP8 scale for all
    w = rng.normal(size=(cout, 3, 3, cin)).astype(np.float32)
    b = rng.normal(size=cout).astype(np.float32)
    got = mrs.conv3x3(x, w, b, relu=True, precision=precision)
    for n in sorted({0, 1, N // 2, N - 2, N - 1}):
        assert torch.equal(got[n:n + 1], mrs.conv3x3(x[n:n + 1].contiguous(), w, b, relu=True, precision=precision))


@pytest.mark.parametrize("N,H,W", SHAPES)
@pytest.mark.parametrize("mode", ["linear", "relu_mask", "residual"])
def test_dgrad_of_a_batch_is_each_images(N, H, W, mode):
    rng = np.random.default_rng(H)
    dy, aux = _images(2, N, H, W, 64), _images(3, N, H, W, 64)
    w = rng.normal(size=(64, 3, 3, 64)).astype(np.float32)
    got = mrs.conv3x3_dgrad(dy, w, mode, None if mode == "linear" else aux, "bf16")
    for n in sorted({0, 1, N // 2, N - 2, N - 1}):
        one = mrs.conv3x3_dgrad(dy[n:n + 1].contiguous(), w, mode,
                                None if mode == "linear" else aux[n:n + 1].contiguous(), "bf16")
        assert torch.equal(got[n:n + 1], one)


@pytest.mark.parametrize("H", [1, 2, 455, 456, 457, 608, 1300])
@pytest.mark.parametrize("precision,cin,cout", [("bf16", 64, 64), ("bf16", 130, 64), ("fp8", 64, 64), ("bf16", 9, 3)])
def test_rows_do_not_depend_on_the_image_around_them(H, precision, cin, cout):
    # images of one strip, from one row to many a CTA (the epilogue's two
    # arrangements, odd and even counts): a row is that of the three-row image
    # around it
    rng = np.random.default_rng(H)
    x = _images(5, 1, H, 70, cin)
    x[:, :, 0, 0] = 7.0                                   # one FP8 scale for all
    w = rng.normal(size=(cout, 3, 3, cin)).astype(np.float32)
    b = rng.normal(size=cout).astype(np.float32)
    got = mrs.conv3x3(x, w, b, precision=precision)
    for y in sorted({0, 1 % H, H // 2, max(H - 2, 0), H - 1}):
        lo, hi = max(y - 1, 0), min(y + 2, H)
        one = mrs.conv3x3(x[:, lo:hi].contiguous(), w, b, precision=precision)
        assert torch.equal(got[:, y], one[:, y - lo])
