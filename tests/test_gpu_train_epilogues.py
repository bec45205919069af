"""Both networks' BF16 training steps against the same steps in float64 with every
tensor rounded to BF16 where the step rounds it (operands, activations, their
gradients after each accumulation; ReLU masks from the rounded activations): the groups
of convolutions in one launch, their masks and second results, at images that share
tiles, at tiles' last columns and images' last rows.

Weights are 0, 1 and -1 (a few for each output; 2^-32 in the last layer, so that I_SR is
next to 1 and dL/dI_SR one constant with two signs), images and biases multiples
of 1/8: every activation and gradient is a whole number of 1/8 or of that constant, below
2^24 of it, so FP32 sums are exact, both sides round the same values, and a mask or sum
that is wrong in one pixel is not lost in rounding.  What is left are the weight
gradients' FP32 sums over pixels: 1e-4 of the sum of |terms|, as in test_gpu_wgrad.py."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
F = torch.nn.functional
T2D = torch.nn.grad


@pytest.fixture(scope="module")
def mrs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2106_12802_gb300 as m
    m.load()
    return m


def _rb(t):
    return t.float().bfloat16().double()


def _nchw(t):
    return t.double().permute(0, 3, 1, 2)


def _split(params, layers):
    """(weight [co, ci, k, k], bias) of every layer of the flat parameters, in float64."""
    at, out = 0, []
    p = torch.from_numpy(params).cuda().double()
    for _, k, ci, co in layers:
        w = p[at:at + co * k * k * ci].view(co, k, k, ci).permute(0, 3, 1, 2)
        at += co * k * k * ci
        out.append((w, p[at:at + co]))
        at += co
    return out


def _params(layers, seed):
    r = np.random.default_rng(seed)
    out = []
    for name, k, ci, co in layers:
        some = {"fuse": 16, "H_rec": 16}.get(name, 1 if name.endswith("conv4") else 3)
        w = np.zeros((co, k * k * ci), np.float32)
        for o in range(co):
            w[o, r.choice(k * k * ci, some, replace=False)] = r.choice([-1.0, 1.0], some)
        if name == "H_rec":
            w *= 2.0 ** -32
        out += [w.ravel(), np.full(co, 1.0) if name == "H_rec" else r.integers(-4, 9, co) / 8.0]
    return np.concatenate(out).astype(np.float32)


class _Net:
    """A network's layers in float64, weights rounded, and their gradients."""

    def __init__(self, params, layers):
        self.L = [(_rb(w), b) for w, b in _split(params, layers)]
        self.grads = [None] * len(self.L)
        self.unit = 0.125

    def exact(self, t):
        assert 0 < float(t.abs().max()) < self.unit * 2.0 ** 24
        return t

    def conv(self, i, x):
        w, b = self.L[i]
        return self.exact(F.conv2d(x, w, b, padding=w.shape[2] // 2))

    def loss_grad(self, y, target):
        """dL/dy of the L1-log loss as the kernel forms it, one constant with two signs."""
        dy = _rb(_nchw(torch.sign(y - target) / (1.0 + y.abs()) * np.float32(1.0 / y.numel())))
        self.unit = float(dy.abs().min()) * 2.0 ** -32
        assert float(dy.abs().max()) * 2.0 ** -32 == self.unit
        return dy

    def back(self, i, x, dz):
        """Layer i's gradients (weight, sum of |terms|, bias, sum of |terms|) from its
        input and dz; dz through the layer."""
        w, _ = self.L[i]
        pad = w.shape[2] // 2
        self.grads[i] = (T2D.conv2d_weight(x, w.shape, dz, padding=pad),
                         T2D.conv2d_weight(x.abs(), w.shape, dz.abs(), padding=pad),
                         dz.sum((0, 2, 3)), dz.abs().sum((0, 2, 3)))
        return self.exact(T2D.conv2d_input(x.shape, w, dz, padding=pad))


def _fusion_step(net, im, y):
    lr, hr, alb, nrm, tgt = im
    up = torch.ones_like(_nchw(hr))               # the LRHS is 1
    x0 = _rb(torch.cat([up] + [_nchw(t) for t in (hr, alb, nrm)], 1))
    h, r = [_rb(F.relu(net.conv(0, x0)))], []
    for k in range(8):
        r.append(_rb(F.relu(net.conv(1 + 2 * k, h[k]))))
        h.append(_rb(h[k] + net.conv(2 + 2 * k, r[k])))
    dh = _rb(net.back(17, h[8], net.loss_grad(y, tgt)))
    for k in range(7, -1, -1):
        da = _rb(net.back(2 + 2 * k, r[k], dh) * (r[k] > 0))
        dh = dh + net.back(1 + 2 * k, h[k], da)
        dh = _rb(dh * (h[0] > 0) if k == 0 else dh)
    net.back(0, x0, dh)


def _rdn_step(net, im, y, s):
    conv, back, blocks, D = net.conv, net.back, 15, int(np.log2(s))
    lr, hr, alb, nrm, tgt = im
    inL, inH = _rb(_nchw(lr)), _rb(torch.cat([_nchw(t) for t in (hr, alb, nrm)], 1))
    flr, fh0 = _rb(F.relu(conv(0, inL))), _rb(F.relu(conv(1, inH)))
    deep = fh0
    for _ in range(D):
        deep = F.pixel_unshuffle(deep, 2)
    cat = torch.cat([flr, deep], 1)
    f0 = _rb(F.relu(conv(2, cat)))
    X, parts = [f0], []
    for k in range(blocks):
        p = [X[k]]
        for c in range(4):
            p.append(_rb(F.relu(conv(3 + 4 * k + c, torch.cat(p, 1)))))
        parts.append(p)
        x = X[k] + p[4]
        if k % 5 == 4:
            x = x + X[k - 4]
            if k == blocks - 1:
                x = x + f0
        X.append(_rb(x))
    U = [X[-1]]
    for d in range(D):
        U.append(F.pixel_shuffle(_rb(F.relu(conv(3 + 4 * blocks + d, U[d]))), 2))

    g = back(3 + 4 * blocks + D, U[D], net.loss_grad(y, tgt))
    for d in range(D, 0, -1):
        g = _rb(g * (U[d] > 0))
        g = back(3 + 4 * blocks + d - 1, U[d - 1], F.pixel_unshuffle(g, 2))
    G = gdf = _rb(g)
    for k in range(blocks - 1, -1, -1):
        p = parts[k]
        if k % 5 == 4:
            skip = G
        dp = [G, None, None, None]
        dz = G * (p[4] > 0)
        for c in range(4, 0, -1):
            full = back(3 + 4 * k + c - 1, torch.cat(p[:c], 1), dz).split(64, 1)
            for j in range(c):
                v = full[j] if dp[j] is None else dp[j] + full[j]
                if j == c - 1 and j > 0:          # complete: masked by F_j
                    v = v * (p[j] > 0)
                dp[j] = _rb(v)
            dz = dp[c - 1]
        G = dp[0]
        if k % 5 == 0:
            G = _rb(G + skip)
    full = back(2, cat, _rb((gdf + G) * (f0 > 0)))
    back(0, inL, _rb(full[:, :64] * (flr > 0)))
    dz1 = full[:, 64:]
    for _ in range(D):
        dz1 = F.pixel_shuffle(dz1, 2)
    back(1, inH, _rb(dz1 * (fh0 > 0)))


def _batch(N, H, W, s):
    g = torch.Generator(device="cuda").manual_seed(N + H + W)
    im = [torch.randint(0, 17, (N, H * k, W * k, 3), device="cuda", generator=g) / 8.0 for k in (1, s, s, s)]
    return im + [torch.randint(0, 2, (N, H * s, W * s, 3), device="cuda", generator=g) * 2.0]


def _check(layers, got, net):
    for (name, *_), (gw, gb), (rw, aw, rb, ab) in zip(layers, _split(got, layers), net.grads):
        assert ((gw - rw).abs() <= 1e-4 * aw).all(), name
        assert ((gb - rb).abs() <= 1e-4 * ab).all(), name


# LR images: several to a tile (62 pixels and less), one to a tile, two strips
@pytest.mark.parametrize("N,H,W,s", [(3, 7, 20, 2), (2, 9, 62, 2), (5, 4, 41, 4), (1, 11, 63, 2), (1, 5, 129, 2),
                                     (2, 2, 130, 4), (16, 12, 12, 4), (2, 6, 9, 8)])
def test_two_encoder_step(mrs, N, H, W, s):
    from paper_2106_12802_gb300 import rdn
    im, layers = _batch(N, H, W, s), rdn.layers(s)
    params = _params(layers, W)
    net, y = mrs.RDN(params, s), torch.empty_like(im[1])
    net.train_step(*im, lr=0.0, loss="l1log", precision="bf16", out=y)
    ref = _Net(params, layers)
    _rdn_step(ref, im, y, s)
    _check(layers, net.get_grads(), ref)


@pytest.mark.parametrize("N,H,W", [(3, 14, 40), (5, 6, 62), (2, 10, 64), (1, 22, 128), (1, 6, 130), (40, 2, 2)])
def test_fusion_step(mrs, N, H, W):
    im = _batch(N, H // 2, W // 2, 2)
    im[0].fill_(1.0)
    layers = [("head", 3, 12, 64)] + [(f"conv{i}", 3, 64, 64) for i in range(1, 17)] + [("H_rec", 3, 64, 3)]
    params = _params(layers, W)
    params[-3:] = 0.0                             # I_SR is next to the upsampled LRHS
    net = mrs.Net(params)
    y = net.fuse(*im[:4], 2, precision="bf16")    # the step's forward
    mrs.train_step(net, *im, 2, lr=0.0, precision="bf16")
    ref = _Net(params, layers)
    _fusion_step(ref, im, y)
    _check(layers, mrs.get_grads(net), ref)
