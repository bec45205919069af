"""FP32 network calls recorded in a CUDA graph follow the weights: a replay
after the weights have changed gives the bits of a direct call with the new
ones, and so does a direct call after replays of a recorded training step,
whose weight updates the host does not see."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

S = 2


@pytest.fixture(scope="module")
def mrs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2106_12802_gb300 as m
    m.load()
    return m


def _net(mrs, kind, seed):
    from paper_2106_12802_gb300 import fusion, rdn
    if kind == "rdn":
        return mrs.RDN(rdn.kaiming_params(S, seed=seed), S)
    return mrs.Net(np.random.default_rng(seed).normal(0.0, 0.04, fusion.NPARAMS).astype(np.float32))


class _Calls:
    """The calls of either network on one seeded batch."""

    def __init__(self, mrs, kind):
        g = torch.Generator(device="cuda").manual_seed(3)
        N, H, W = 1, 20, 36
        self.mrs, self.kind = mrs, kind
        self.im = [torch.rand(N, H // k, W // k, 3, device="cuda", generator=g) for k in (S, 1, 1, 1, 1)]

    def fuse(self, net, out=None):
        scale = (S,) if self.kind == "net" else ()
        return net.fuse(*self.im[:4], *scale, precision="fp32", out=out)

    def step(self, net, precision):
        if self.kind == "net":
            self.mrs.train_step(net, *self.im, S, lr=1e-4, precision=precision, sync_loss=False)
        else:
            net.train_step(*self.im, lr=1e-4, precision=precision, sync_loss=False)

    def state(self, net):
        return self.mrs.get_state(net) if self.kind == "net" else net.get_state()

    def set_state(self, net, st):
        self.mrs.set_state(net, st) if self.kind == "net" else net.set_state(st)

    def again(self, net):
        """A direct call of a network made anew with net's weights."""
        torch.cuda.synchronize()
        fresh = _net(self.mrs, self.kind, 99)
        self.set_state(fresh, self.state(net))
        return self.fuse(fresh)


def _record(call):
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        call()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        call()
    return g


@pytest.mark.parametrize("kind", ["net", "rdn"])
def test_replayed_call_follows_the_weights(mrs, kind, tmp_path):
    c = _Calls(mrs, kind)
    net, other = _net(mrs, kind, 0), _net(mrs, kind, 1)
    out = torch.empty_like(c.im[1])
    g = _record(lambda: c.fuse(net, out))
    changes = [lambda: None, lambda: c.step(net, "fp32"), lambda: c.step(net, "bf16"),
               lambda: c.set_state(net, c.state(other))]
    if kind == "net":
        mrs.save_checkpoint(_net(mrs, kind, 2), tmp_path / "net")
        changes += [lambda: mrs.load_checkpoint(net, tmp_path / "net"),
                    lambda: net.set_params(_net(mrs, kind, 3).get_params())]
    seen = []
    for change in changes:
        change()
        torch.cuda.synchronize()
        out.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, c.again(net))
        assert torch.equal(out, c.fuse(net))
        assert not any(torch.equal(out, o) for o in seen)
        seen.append(out.clone())


@pytest.mark.parametrize("kind,precision", [("net", "fp32"), ("net", "bf16"), ("rdn", "fp32")])
def test_direct_call_follows_a_replayed_step(mrs, kind, precision):
    c = _Calls(mrs, kind)
    net = _net(mrs, kind, 0)
    g = _record(lambda: c.step(net, precision))
    seen = []
    for _ in range(3):
        a = c.fuse(net)
        assert torch.equal(a, c.again(net))
        assert not any(torch.equal(a, o) for o in seen)
        seen.append(a)
        g.replay()
        torch.cuda.synchronize()
