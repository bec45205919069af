"""The work that a user has this framework do, as cases that can be timed and compared.

Renders (scenes of 10k to 200k triangles, one sample to many, whole images,
windows, extra layers, a batch of frames, an animated mesh), the hybrid frame,
the fusion network and the method's own network (inference and training), each
through the package's public calls.  `listed()` holds one case of each kind of
use, `draw(rng)` others of the same ranges.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

import paper_2106_12802_gb300 as mrs
from paper_2106_12802_gb300 import rdn as mrs_rdn

DEPTH, RR = 8, 3      # scattering events, first bounce with roulette (the renders' usual setting)
LR_RATE = 1e-4        # Adam's rate in the training recipe


def listed():
    return [
        # the smallest call: a thumbnail of the Cornell box, where launches and latency count
        {"name": "render_cornell_48", "kind": "render", "scene": "cornell", "tree": "lbvh", "W": 48, "H": 48,
         "spp": 1, "layers": False, "wx": 0, "wy": 0, "ww": 48, "wh": 48},
        # a crop for the network's training data: a ragged window of a frame, every layer of it
        {"name": "render_window_layers", "kind": "render", "scene": "procedural", "tree": "cluster", "W": 1024,
         "H": 1024, "spp": 6, "layers": True, "wx": 301, "wy": 417, "ww": 331, "wh": 267},
        # the method's rival and its training target: a whole image by path tracing alone
        {"name": "render_plain_1024", "kind": "render", "scene": "procedural", "tree": "hcluster", "W": 1024,
         "H": 1024, "spp": 64, "layers": False, "wx": 0, "wy": 0, "ww": 1024, "wh": 1024},
        # serving: low- and high-resolution renders of several users' frames in one batch, fused in FP8
        {"name": "serve_batch_fp8", "kind": "serve", "frames": 4, "W": 640, "H": 360, "scale": 2, "spp_l": 16,
         "spp_h": 2, "precision": "fp8"},
        # an animated mesh: new vertices each frame, the tree rebuilt, a preview image
        {"name": "animate_mesh", "kind": "animate", "nx": 301, "ny": 257, "tree": "hcluster", "W": 480, "H": 270,
         "spp": 1},
        # the method's whole step: tree, both renders on two streams, fusion, gate
        {"name": "frame_hybrid", "kind": "frame", "W": 1024, "H": 1024, "scale": 4, "spp_l": 64, "spp_h": 4,
         "precision": "bf16"},
        # the fusion network alone, at the frame's size
        {"name": "fuse_bf16_1024", "kind": "fuse", "N": 1, "W": 1024, "H": 1024, "scale": 4, "extra": False,
         "precision": "bf16"},
        # reference precision, a ragged size, the extra layers as input (evaluation)
        {"name": "fuse_fp32_ragged", "kind": "fuse", "N": 1, "W": 486, "H": 330, "scale": 2, "extra": True,
         "precision": "fp32"},
        # the method's own two-encoder network
        {"name": "rdn_bf16_1024", "kind": "rdn", "N": 1, "W": 1024, "H": 1024, "scale": 4, "extra": False,
         "precision": "bf16"},
        # training the fusion network: the recipe's batch and precision, and the call's default precision
        {"name": "train_bf16", "kind": "train", "N": 16, "W": 128, "H": 128, "scale": 4, "extra": False,
         "precision": "bf16", "loss": "l1log"},
        {"name": "train_fp32", "kind": "train", "N": 6, "W": 128, "H": 128, "scale": 4, "extra": False,
         "precision": "fp32", "loss": "robust"},
        # training the method's own network at its batch
        {"name": "rdn_train_bf16", "kind": "rdn_train", "N": 16, "W": 192, "H": 192, "scale": 4, "extra": False,
         "precision": "bf16", "loss": "l1log"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng, scale, lo, hi, pixels):
    """A ragged W x H of multiples of `scale`, of at most `pixels` pixels."""
    while True:
        W, H = (max(1, _log(rng, lo, hi) // scale) * scale for _ in range(2))
        if W * H <= pixels:
            return W, H


def draw(rng):
    kind = rng.choice(["render", "render", "serve", "animate", "frame", "fuse", "fuse", "rdn", "train", "train",
                       "rdn_train"])
    tree = rng.choice(["lbvh", "cluster", "hcluster"])
    if kind == "render":
        W, H = _size(rng, 1, 32, 1600, 1 << 20)
        spp = _log(rng, 1, max(1, min(64, (1 << 24) // (W * H))))
        ww, wh = (W, H) if rng.random() < 0.6 else (rng.randint(1, W), rng.randint(1, H))
        return {"kind": kind, "scene": rng.choice(["cornell", "procedural"]), "tree": tree, "W": W, "H": H,
                "spp": spp, "layers": rng.random() < 0.4, "wx": rng.randint(0, W - ww), "wy": rng.randint(0, H - wh),
                "ww": ww, "wh": wh}
    if kind == "animate":
        W, H = _size(rng, 1, 64, 800, 1 << 19)
        return {"kind": kind, "nx": rng.randint(20, 320), "ny": rng.randint(20, 320), "tree": tree, "W": W, "H": H,
                "spp": rng.randint(1, 3)}
    scale = rng.choice([2, 4])
    if kind == "serve":
        W, H = _size(rng, scale, 96, 900, 300_000)
        return {"kind": kind, "frames": rng.randint(2, 6), "W": W, "H": H, "scale": scale,
                "spp_l": _log(rng, 8, 48), "spp_h": rng.randint(1, 4), "precision": rng.choice(["bf16", "fp8"])}
    if kind == "frame":
        W, H = _size(rng, scale, 200, 1200, 1 << 20)
        return {"kind": kind, "W": W, "H": H, "scale": scale, "spp_l": _log(rng, 8, 64), "spp_h": rng.randint(1, 6),
                "precision": rng.choice(["bf16", "bf16", "fp8"])}
    extra = rng.random() < 0.35
    if kind == "fuse":
        precision = rng.choice(["bf16", "fp8", "fp32"])
        N = rng.randint(1, 3)
        W, H = _size(rng, scale, 64, 1300, (300_000 if precision == "fp32" else 1_200_000) // N)
        return {"kind": kind, "N": N, "W": W, "H": H, "scale": scale, "extra": extra, "precision": precision}
    if kind == "rdn":
        precision = rng.choice(["bf16", "bf16", "fp32"])
        N = rng.randint(1, 2)
        W, H = _size(rng, scale, 96, 1200, (200_000 if precision == "fp32" else 1_000_000) // N)
        return {"kind": kind, "N": N, "W": W, "H": H, "scale": scale, "extra": extra, "precision": precision}
    if kind == "train":
        precision = rng.choice(["bf16", "fp32"])
        N = rng.randint(1, 16)
        W, H = _size(rng, scale, 48, 200, (100_000 if precision == "fp32" else 300_000) // N)
        return {"kind": kind, "N": N, "W": W, "H": H, "scale": scale, "extra": extra, "precision": precision,
                "loss": rng.choice(["l1log", "robust"])}
    N = rng.randint(1, 16)
    precision = rng.choice(["bf16", "bf16", "fp32"])
    W, H = _size(rng, scale, 64, 224, (100_000 if precision == "fp32" else 600_000 if scale == 4 else 200_000) // N)
    # untrained and in 16 bits, the robust loss hangs on the few pixels nearest their target
    loss = rng.choice(["l1log", "robust"]) if precision == "fp32" else "l1log"
    return {"kind": kind, "N": N, "W": W, "H": H, "scale": scale, "extra": extra, "precision": precision,
            "loss": loss}


# ---- inputs ------------------------------------------------------------------

def _field(g, N, C, H, W, cell):
    """A smooth random field in [0, 1], [N, C, H, W]."""
    coarse = torch.rand((N, C, H // cell + 2, W // cell + 2), device="cuda", generator=g)
    return F.interpolate(coarse, size=(H, W), mode="bilinear", align_corners=False)


def _images(seed, c):
    """What the renders hand the networks: an HDR radiance (most of it in [0, 10], a few fireflies) at low
    resolution with little noise and at high resolution with much, albedo, unit normals, the extra layers, and
    the clean image as the training target; [N, H, W, C] float32."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    N, H, W, s = c["N"], c["H"], c["W"], c["scale"]

    def noise(shape, sigma):
        return torch.exp(sigma * torch.randn(shape, device="cuda", generator=g))

    clean = 8.0 * _field(g, N, 3, H, W, 24) ** 3 * (0.5 + _field(g, N, 3, H, W, 5)) + 0.02
    low = F.avg_pool2d(clean, s)
    low = low * noise(low.shape, 0.1)
    high = clean * noise(clean.shape, 0.6)
    high = torch.where(torch.rand((N, 1, H, W), device="cuda", generator=g) < 1e-4, 40.0 * high, high)
    albedo = 0.1 + 0.8 * _field(g, N, 3, H, W, 9)
    normal = F.normalize(_field(g, N, 3, H, W, 13) - 0.5 + 1e-3, dim=1)
    share = _field(g, N, 1, H, W, 31)
    extra = torch.cat([high * share, high * (1.0 - share), (0.3 * high) ** 2], 1)

    def nhwc(t):
        return t.permute(0, 2, 3, 1).contiguous().float()

    d = {"lrhs": nhwc(low), "hrls": nhwc(high), "albedo": nhwc(albedo), "normal": nhwc(normal),
         "target": nhwc(clean)}
    d["extra"] = nhwc(extra) if c["extra"] else None
    return d


def _net_layers(extra):
    return [(21 if extra else 12, 64)] + [(64, 64)] * 16 + [(64, 3)]


def _net_params(seed, extra):
    """Weights of a network in training: Kaiming scale, the blocks' second convolutions and the head damped."""
    r = np.random.default_rng([17, int(seed)])
    parts = []
    for i, (ci, co) in enumerate(_net_layers(extra)):
        damp = 0.2 if i == 17 else 0.25 if i and i % 2 == 0 else 1.0
        parts += [r.normal(0.0, damp * math.sqrt(2.0 / (9 * ci)), co * 9 * ci), r.normal(0.0, 0.01, co)]
    return np.concatenate(parts).astype(np.float32)


def _rdn_layers(scale, extra):
    """(kernel, inputs, outputs) of each convolution in the order of the parameters."""
    dense = [(3, 64 * k, 64) for _ in range(15) for k in (1, 2, 3, 4)]
    ups = [(3, 64, 256)] * int(math.log2(scale))
    return [(3, 3, 64), (3, 18 if extra else 9, 64), (1, 64 + 64 * scale * scale, 64)] + dense + ups + [(3, 64, 3)]


def _rdn_params(seed, c):
    return mrs_rdn.kaiming_params(c["scale"], 18 if c["extra"] else 9, seed=int(seed))


def _mesh(seed, c):
    """A waving sheet of 2 (nx - 1) (ny - 1) triangles over a ground quad, lit by a quad and the sky; and the
    vertices of its next frame."""
    r = np.random.default_rng([23, int(seed)])
    nx, ny = c["nx"], c["ny"]
    ph = r.uniform(0, 2 * math.pi, 6)
    x, y = np.meshgrid(np.linspace(-3, 3, nx), np.linspace(-2.5, 2.5, ny), indexing="ij")

    def frame(t):
        z = 0.8 + sum(0.25 / (k + 1) * np.sin((k + 1) * (1.1 * x + 0.7 * y) + ph[k] + t) *
                      np.cos((k + 1) * 0.9 * y - ph[k + 3]) for k in range(3))
        p = np.stack([x, y, z], -1)
        a, b, cc, d = p[:-1, :-1], p[1:, :-1], p[1:, 1:], p[:-1, 1:]
        sheet = np.stack([np.stack([a, b, cc], 2), np.stack([a, cc, d], 2)], 2).reshape(-1, 3, 3)

        def quad(o, u, v):
            o, u, v = (np.array(q, float) for q in (o, u, v))
            return [[o, o + u, o + u + v], [o, o + u + v, o + v]]

        fixed = quad((-8, -8, -0.5), (16, 0, 0), (0, 16, 0)) + quad((-1, 1, 5), (0, 2, 0), (2, 0, 0))
        return np.ascontiguousarray(np.concatenate([sheet, np.array(fixed)]), np.float32)

    n = 2 * (nx - 1) * (ny - 1)
    eye, fwd = np.array([0, -7.0, 4.5]), np.array([0, 7.0, -3.9])
    fwd /= np.linalg.norm(fwd)
    right = np.array([1.0, 0, 0])
    up = np.cross(right, fwd)
    th = math.tan(math.radians(22.0))
    desc = {"V": frame(0.0), "tri_mat": np.r_[np.zeros(n), 1, 1, 2, 2].astype(np.int32),
            "tri_light": np.r_[np.full(n + 2, -1), 0, 0].astype(np.int32),
            "mats": np.array([[1, 0.7, 0.5, 0.4, 0.3, 0, 0, 0], [0, 0.5, 0.5, 0.5, 1, 0, 0, 0],
                              [0, 0, 0, 0, 1, 12, 12, 12]], np.float32),
            "lights": np.array([[-1, 1, 5, 0, 2, 0, 2, 0, 0, 12, 12, 12]], np.float32),
            "env": np.full(3, 0.4, np.float32),
            "cam": np.concatenate([eye, fwd, right * th * c["W"] / c["H"], up * th]).astype(np.float32)}
    return desc, torch.from_numpy(frame(0.3 + r.uniform(0, 1))).pin_memory()


def _scene(seed, kind, tree, W, H):
    sc = mrs.Scene.seeded(int(seed), kind, aspect=float(np.float32(min(16.0, W / H))))
    sc.set_tree(tree)
    return sc


def _planes(W, H, *names):
    return {k: torch.empty((H, W) if k == "depth" else (H, W, 3), device="cuda") for k in names}


AUX = ("radiance", "albedo", "normal", "depth")


def prepare(case, seed):
    c, kind = case, case["kind"]
    st = {"c": c, "seed": int(seed)}
    if kind == "render":
        st["scene"] = _scene(seed, c["scene"], c["tree"], c["W"], c["H"])
        st["out"] = _planes(c["ww"], c["wh"], *AUX, *(("diffuse", "specular", "variance") if c["layers"] else ()))
        st["out"].update({k: torch.zeros(DEPTH + 1, dtype=torch.int64, device="cuda")
                          for k in ("counts", "shadow_counts")})
        whole = (c["ww"], c["wh"]) == (c["W"], c["H"])
        st["window"] = None if whole else (c["wx"], c["wy"], c["ww"], c["wh"])
    elif kind == "animate":
        desc, st["V"] = _mesh(seed, c)
        st["scene"] = mrs.Scene(desc)
        st["scene"].set_tree(c["tree"])
        st["out"] = _planes(c["W"], c["H"], *AUX)
    elif kind == "serve":
        N, W, H, s = c["frames"], c["W"], c["H"], c["scale"]
        st["net"] = mrs.Net(_net_params(5, False))
        st["ctx"] = mrs.RenderContext()
        st["scenes"] = [_scene(seed * 64 + i, "procedural", "hcluster", W, H) for i in range(N)]
        st["low"] = torch.empty((N, H // s, W // s, 3), device="cuda")
        st["high"] = [torch.empty((N, H, W, 3), device="cuda") for _ in range(3)]
        st["depth"] = torch.empty((N, H, W), device="cuda")
        st["fused"] = torch.empty((N, H, W, 3), device="cuda")
        st["jobs"] = []
        for i, sc in enumerate(st["scenes"]):
            both = {"scene": sc, "max_depth": DEPTH, "rr_start": RR}
            st["jobs"] += [
                dict(both, W=W // s, H=H // s, spp=c["spp_l"], seed=seed + i, out={"radiance": st["low"][i]}),
                dict(both, W=W, H=H, spp=c["spp_h"], seed=seed + 1000 + i,
                     out=dict(zip(AUX, [t[i] for t in st["high"]] + [st["depth"][i]])))]
    elif kind == "frame":
        W, H, s = c["W"], c["H"], c["scale"]
        st["net"] = mrs.Net(_net_params(5, False))
        st["scene"] = _scene(seed, "procedural", "hcluster", W, H)
        st["ctx"] = [mrs.RenderContext() for _ in range(2)]
        st["streams"] = [torch.cuda.Stream() for _ in range(2)]
        st["low"] = _planes(W // s, H // s, "radiance")
        st["high"] = _planes(W, H, *AUX)
        st["fused"], st["out"] = (torch.empty((1, H, W, 3), device="cuda") for _ in range(2))
        st["used"] = torch.zeros(2, dtype=torch.int32, device="cuda")
        st["D"] = torch.zeros(1, dtype=torch.float64, device="cuda")
    else:
        st["im"] = _images(seed, c)
        if kind in ("fuse", "train"):
            st["net"] = mrs.Net(_net_params(seed, c["extra"]))
            if kind == "train":
                st["net"].set_loss(c["loss"], 0.1)
        else:
            st["net"] = mrs.RDN(_rdn_params(seed, c), c["scale"], 18 if c["extra"] else 9)
        if kind in ("fuse", "rdn"):
            st["out"] = torch.empty_like(st["im"]["hrls"])
    return st


def run(state):
    c, kind = state["c"], state["c"]["kind"]
    if kind == "render":
        return mrs.render(state["scene"], c["W"], c["H"], c["spp"], DEPTH, RR, state["seed"], out=state["out"],
                          layers=c["layers"], window=state["window"])
    if kind == "animate":
        state["scene"].update_vertices(state["V"])
        return mrs.render(state["scene"], c["W"], c["H"], c["spp"], DEPTH, RR, state["seed"], out=state["out"])
    if kind == "serve":
        mrs.render_batch(state["ctx"], state["jobs"])
        state["net"].fuse(state["low"], *state["high"], c["scale"], precision=c["precision"], out=state["fused"])
        return [state["low"], state["high"], state["depth"], state["fused"]]
    if kind == "frame":
        scene, (ctx_l, ctx_h), (s_l, s_h) = state["scene"], state["ctx"], state["streams"]
        low, high, main = state["low"], state["high"], torch.cuda.current_stream()
        scene.rebuild()
        for s in (s_h, s_l):
            s.wait_stream(main)
        with torch.cuda.stream(s_h):
            mrs.render(scene, c["W"], c["H"], c["spp_h"], DEPTH, RR, state["seed"] + 1, ctx=ctx_h, out=high)
        with torch.cuda.stream(s_l):
            mrs.render(scene, c["W"] // c["scale"], c["H"] // c["scale"], c["spp_l"], DEPTH, RR, state["seed"],
                       ctx=ctx_l, out=low)
        for s in (s_h, s_l):
            main.wait_stream(s)
        lrhs = low["radiance"][None]
        state["net"].fuse(lrhs, *(high[k][None] for k in AUX[:3]), c["scale"], precision=c["precision"],
                          out=state["fused"])
        mrs.gate_async(state["fused"], lrhs, None, c["scale"], 0.01, out=state["out"], used=state["used"],
                       D=state["D"])
        return [state["out"], state["used"], state["D"], low, high]
    im, net = state["im"], state["net"]
    four = (im["lrhs"], im["hrls"], im["albedo"], im["normal"])
    if kind == "fuse":
        return net.fuse(*four, c["scale"], precision=c["precision"], out=state["out"], extra=im["extra"])
    if kind == "rdn":
        return net.fuse(*four, precision=c["precision"], out=state["out"], extra=im["extra"])
    if kind == "train":
        loss = mrs.train_step(net, *four, im["target"], c["scale"], lr=LR_RATE, precision=c["precision"],
                              extra=im["extra"])
        return {"loss": loss, "grads": mrs.get_grads(net)}
    loss = net.train_step(*four, im["target"], lr=LR_RATE, loss=c["loss"], extra=im["extra"],
                          precision=c["precision"])
    return {"loss": loss, "grads": net.get_grads()}


# ---- what a pass cannot do without ---------------------------------------------

def _net_flops(c, pixels):
    return pixels * sum(18 * ci * co for ci, co in _net_layers(c.get("extra", False)))


def _rdn_flops(c, pixels):
    s, total, up = c["scale"], 0, 0
    for i, (k, ci, co) in enumerate(L := _rdn_layers(s, c["extra"])):
        f = 2 * k * k * ci * co
        if i == 1 or i == len(L) - 1:
            f *= s * s
        elif co == 256:
            f *= 4 ** up
            up += 1
        total += f
    return total * pixels // (s * s)


def _render_work(paths, pixels, floats, tris):
    """Bytes: the triangles, and the image.  Operations: two closest-hit rays and one and a half shadow rays for
    a path, each down a tree of depth log2 n (24 a node) to two triangles (27 each)."""
    return 4 * floats * pixels + 36 * tris, paths * 3.5 * (24 * math.log2(tris) + 54)


def work(case):
    c, kind = case, case["kind"]
    px = c.get("W", 1) * c.get("H", 1)
    if kind == "render":
        n = c["ww"] * c["wh"]
        b, f = _render_work(n * c["spp"], n, 19 if c["layers"] else 10, 10_252 if c["scene"] == "cornell" else 200_968)
    elif kind == "animate":
        n = 2 * (c["nx"] - 1) * (c["ny"] - 1) + 4
        b, f = _render_work(px * c["spp"], px, 10, 2 * n)
    elif kind in ("serve", "frame"):
        s, many = c["scale"], c.get("frames", 1)
        bl, fl = _render_work(px // (s * s) * c["spp_l"], px // (s * s), 3, 200_968)
        bh, fh = _render_work(px * c["spp_h"], px, 10, 200_968)
        b, f = many * (bl + bh + 12 * px), many * (fl + fh + _net_flops(c, px))
    else:
        px *= c["N"]
        inputs = 4 * px * (9 + 3 / c["scale"] ** 2 + (9 if c["extra"] else 0))
        own = kind.startswith("rdn")
        flops = _rdn_flops(c, px) if own else _net_flops(c, px)
        layers = [(k * k, ci, co) for k, ci, co in _rdn_layers(c["scale"], c["extra"])] if own else \
            [(9, ci, co) for ci, co in _net_layers(c["extra"])]
        params = 4 * sum(k * ci * co + co for k, ci, co in layers)
        training = "train" in kind
        b = inputs + 12 * px + params * (7 if training else 1)
        f = flops * (3 if training else 1)
    return {"bytes": float(b), "flops": float(f)}


# ---- the networks in 64 bits ------------------------------------------------------

def _nchw(t):
    return t.double().permute(0, 3, 1, 2)


def _convs(p, layers):
    """One callable for each convolution, over the flat parameters p."""
    at, made = 0, []
    for k, ci, co in layers:
        w = p[at:at + co * k * k * ci].view(co, k, k, ci).permute(0, 3, 1, 2)
        b = p[at + co * k * k * ci:at + co * k * k * ci + co]
        at += co * k * k * ci + co
        made.append(lambda x, w=w, b=b, k=k: F.conv2d(x, w, b, padding=k // 2))
    return made


def _net_exact(p, im, c, clip=None):
    convs = _convs(p, [(3, ci, co) for ci, co in _net_layers(c["extra"])])
    low, high = _nchw(im["lrhs"]), _nchw(im["hrls"])
    extra = None if im["extra"] is None else _nchw(im["extra"])
    if clip:
        low, high = low.clamp(max=clip), high.clamp(max=clip)
    up = F.interpolate(low, scale_factor=c["scale"], mode="bilinear", align_corners=False)
    x = [up, high, _nchw(im["albedo"]), _nchw(im["normal"])]
    if extra is not None:
        x += [extra[:, :6].clamp(max=clip) if clip else extra[:, :6], torch.log1p(extra[:, 6:].clamp(min=0))]
    h = F.relu(convs[0](torch.cat(x, 1)))
    for k in range(8):
        h = h + convs[2 + 2 * k](F.relu(convs[1 + 2 * k](h)))
    return convs[17](h) + up


def _rdn_exact(p, im, c):
    convs = iter(_convs(p, _rdn_layers(c["scale"], c["extra"])))
    depth = int(math.log2(c["scale"]))
    x = [_nchw(im["hrls"]), _nchw(im["albedo"]), _nchw(im["normal"])]
    if im["extra"] is not None:
        e = _nchw(im["extra"])
        x += [e[:, :6], torch.log1p(e[:, 6:].clamp(min=0))]
    low, high = F.relu(next(convs)(_nchw(im["lrhs"]))), F.relu(next(convs)(torch.cat(x, 1)))
    for _ in range(depth):
        high = F.pixel_unshuffle(high, 2)
    first = h = F.relu(next(convs)(torch.cat([low, high], 1)))
    for _ in range(3):
        group = h
        for _ in range(5):
            parts = [h]
            for _ in range(3):
                parts.append(F.relu(next(convs)(torch.cat(parts, 1))))
            h = h + F.relu(next(convs)(torch.cat(parts, 1)))
        h = h + group
    h = h + first
    for _ in range(depth):
        h = F.pixel_shuffle(F.relu(next(convs)(h)), 2)
    return next(convs)(h)


def _loss_exact(y, target, kind):
    t = target.clamp(max=100.0)
    if kind == "robust":
        e = (y - t).abs()
        return (e / (0.1 + e)).mean()
    return (y.sign() * y.abs().log1p() - t.sign() * t.abs().log1p()).abs().mean()


def exact(case, seed):
    """The networks' outputs, losses and gradients; a Monte Carlo image has no such value."""
    c, kind = case, case["kind"]
    if kind in ("render", "animate", "serve", "frame"):
        return None
    im, own = _images(seed, c), kind.startswith("rdn")
    p = torch.from_numpy(_rdn_params(seed, c) if own else _net_params(seed, c["extra"])).cuda().double()
    if kind == "fuse":
        with torch.no_grad():
            return _net_exact(p, im, c).permute(0, 2, 3, 1).contiguous()
    if kind == "rdn":
        with torch.no_grad():
            return _rdn_exact(p, im, c).permute(0, 2, 3, 1).contiguous()
    p.requires_grad_()
    y = _rdn_exact(p, im, c) if own else _net_exact(p, im, c, clip=100.0)
    loss = _loss_exact(y, _nchw(im["target"]), c["loss"])
    loss.backward()
    return {"loss": float(loss.detach()), "grads": p.grad}
