"""The BF16 weight gradient's work list at its edges, against the float64 oracle on
the same rounded operands (the bounds of test_gpu_wgrad.py): strips of
one to 64 pixels and a strip's remainder on either side of a K step of 16,
fewer jobs than SMs, runs that start within a row of strips; and the FP32
kernel's tiles of pixels and channels."""
import numpy as np
import pytest
import torch

from oracle import cnn

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mrs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2106_12802_gb300 as m
    m.load()
    return m


def _bf16(a):
    return torch.from_numpy(np.ascontiguousarray(a, np.float32)).to(torch.bfloat16).to(torch.float64).numpy()


def _check(mrs, prec, N, H, W, cin, cout):
    rng = np.random.default_rng(N * 1000 + W)
    x = rng.normal(size=(N, H, W, cin)).astype(np.float32)
    dy = (rng.normal(size=(N, H, W, cout)) * 0.01).astype(np.float32)
    dw, db = mrs.conv3x3_wgrad(torch.from_numpy(x).cuda(), torch.from_numpy(dy).cuda(), precision=prec)
    xr, dyr = (_bf16(x), _bf16(dy)) if prec == "bf16" else (x.astype(np.float64), dy.astype(np.float64))
    zero_w = np.zeros((cout, 3, 3, cin))
    _, rw, rb = cnn.conv3x3_backward(xr, zero_w, dyr)
    _, aw, ab = cnn.conv3x3_backward(np.abs(xr), zero_w, np.abs(dyr))
    assert (np.abs(dw - rw) <= 1e-4 * aw + 1e-9).all()
    assert (np.abs(db - rb) <= 1e-4 * ab + 1e-9).all()


# FP32: half-tiles of 32 pixels, fewer pixels than splits, rows that wrap within
# a thread's steps of 4 pixels, channels in fours and not
@pytest.mark.parametrize("N,H,W,cin,cout", [(1, 1, 1, 64, 64), (2, 5, 3, 3, 2), (1, 7, 31, 64, 3), (1, 40, 33, 21, 64),
                                            (2, 65, 64, 12, 60), (1, 90, 100, 64, 64), (5, 33, 2, 6, 64)])
def test_fp32_tiles(mrs, N, H, W, cin, cout):
    _check(mrs, "fp32", N, H, W, cin, cout)


@pytest.mark.parametrize("N,H,W,cin,cout", [(1, 1, 1, 64, 64), (1, 2, 15, 1, 64), (2, 3, 16, 64, 1), (1, 40, 17, 64, 64),
                                            (3, 48, 48, 64, 64), (2, 60, 63, 18, 64), (1, 200, 65, 64, 64),
                                            (1, 90, 129, 64, 3), (2, 33, 200, 64, 64)])
def test_strip_and_run_edges(mrs, N, H, W, cin, cout):
    _check(mrs, "bf16", N, H, W, cin, cout)
