"""BF16 training steps of one network over several batch shapes: in turn, more
shapes than the handle keeps plans for, on a side stream; and recorded in a CUDA
graph, also for a shape that no direct step had, with direct steps of other shapes
between the recording and its replays.  Every step's gradient has the bits of a
step of a network made anew with the same weights."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

S = 2
SHAPES = [(2, 24, 36), (1, 24, 36), (2, 36, 24), (1, 70, 130), (3, 8, 12), (1, 2, 2), (5, 16, 16), (1, 16, 80),
          (2, 40, 62), (4, 10, 128)]


@pytest.fixture(scope="module")
def mrs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2106_12802_gb300 as m
    m.load()
    return m


def _params(seed):
    from paper_2106_12802_gb300 import fusion
    return np.random.default_rng(seed).normal(0.0, 0.04, fusion.NPARAMS).astype(np.float32)


def _batch(shape):
    g = torch.Generator(device="cuda").manual_seed(sum(shape))
    N, H, W = shape
    return [torch.rand(N, H // k, W // k, 3, device="cuda", generator=g) for k in (S, 1, 1, 1, 1)]


def _step(mrs, net, im):
    mrs.train_step(net, *im, S, lr=1e-4, precision="bf16", sync_loss=False)


def _grads_anew(mrs, state, im):
    net = mrs.Net(_params(99))
    mrs.set_state(net, state)
    _step(mrs, net, im)
    torch.cuda.synchronize()
    return mrs.get_grads(net)


@pytest.mark.parametrize("n", [2, len(SHAPES)])
def test_shapes_in_turn(mrs, n):
    net = mrs.Net(_params(0))
    side = torch.cuda.Stream()
    for shape in 3 * SHAPES[:n]:
        im, before = _batch(shape), mrs.get_state(net)
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _step(mrs, net, im)
        torch.cuda.synchronize()
        assert np.array_equal(mrs.get_grads(net), _grads_anew(mrs, before, im)), shape


@pytest.mark.parametrize("met", [True, False])
def test_recorded_step_keeps_its_plan(mrs, met):
    net = mrs.Net(_params(0))
    batches = [_batch(s) for s in SHAPES]
    _step(mrs, net, _batch((1, 100, 200)))       # the workspace holds every shape below
    if met:
        _step(mrs, net, batches[0])
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        _step(mrs, net, batches[0])
    for im in [None] + batches + batches:
        if im is not None:
            _step(mrs, net, im)
        torch.cuda.synchronize()
        before = mrs.get_state(net)
        g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(mrs.get_grads(net), _grads_anew(mrs, before, batches[0]))
