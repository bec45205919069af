"""The traversal's slab test over centre / half-extent nodes, at the rays and
boxes where it can go wrong: directions with zero components (of either
sign), origins in the planes of boxes' sides, flat boxes (axis-aligned
triangles), boxes far from the origin of coordinates, one- to three-leaf
trees.  The closest hit equals the oracle's bit for bit, over every tree.  Left
out are the rays for which the oracle's traversal and its loop over all
triangles differ (a few: a ray within the plane of a box's side does not meet
that box, so a triangle that touches the plane with an edge or corner is a hit
in the loop alone; a triangle of a scene's size is tested without a box)."""
import numpy as np
import pytest

from synth import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mrs():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2106_12802_gb300 as m
    m.load()
    return m


@pytest.fixture(scope="module")
def orc():
    import oracle
    oracle.build()
    return oracle


def _quads(n, shift):
    """n axis-aligned triangles (flat boxes) with corners on a grid of step 1/4."""
    r = np.random.default_rng(n)
    p = r.integers(-8, 8, (n, 1, 3)) * 0.25 + np.asarray(shift, float)
    e = np.zeros((n, 2, 3))
    axis = r.integers(0, 3, n)
    for k in range(2):
        e[np.arange(n), k, (axis + 1 + k) % 3] = r.choice([-0.5, 0.25, 0.75], n)
    return np.concatenate([p, p + e[:, :1], p + e[:, 1:]], 1).astype(np.float32)


def _rays(V, count):
    r = np.random.default_rng(7)
    lo, hi = V.reshape(-1, 3).min(0), V.reshape(-1, 3).max(0)
    o = r.uniform(lo - 1, hi + 1, (count, 3))
    # a third of the coordinates taken from vertices: origins in box sides' planes
    on = r.random((count, 3)) < 0.33
    o = np.where(on, V.reshape(-1, 3)[r.integers(0, V.shape[0] * 3, (count, 3)), np.arange(3)], o)
    d = r.normal(size=(count, 3))
    zero = r.random((count, 3)) < 0.5
    zero[np.arange(count), r.integers(0, 3, count)] = False
    d = np.where(zero, np.where(r.random((count, 3)) < 0.5, 0.0, -0.0), d)
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    return np.ascontiguousarray(o, np.float32), np.ascontiguousarray(d, np.float32)


@pytest.mark.parametrize("kind,n,shift", [("flat", 1, (0, 0, 0)), ("flat", 2, (0, 0, 0)), ("flat", 3, (0, 0, 0)),
                                          ("flat", 40, (0, 0, 0)), ("flat", 400, (64, -32, 128)),
                                          ("soup", 2, (0, 0, 0)), ("soup", 33, (0, 0, 0)),
                                          ("soup", 400, (100, 0, -50))])
def test_zero_direction_components_and_flat_boxes(mrs, orc, kind, n, shift):
    desc = scenes.random_triangles(5, n)
    if kind == "flat":
        V = _quads(n, shift)
    else:
        V = (desc["V"].reshape(n, 3, 3) + np.asarray(shift, np.float32)).astype(np.float32)
    desc["V"] = np.ascontiguousarray(V.reshape(desc["V"].shape))
    o, d = _rays(V, 20000)
    pb, tb = orc.cast(desc["V"], o, d, brute=True)
    pt, tt = orc.cast(desc["V"], o, d)
    clear = (pb == pt) & (tb == tt)
    assert clear.mean() > 0.9 and (pb[clear] >= 0).sum() > 0
    sc = mrs.Scene(desc)
    for tree in ("lbvh", "cluster", "hcluster"):
        sc.set_tree(tree)
        p, t = sc.cast(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda())
        assert np.array_equal(p.cpu().numpy()[clear], pb[clear])
        assert np.array_equal(t.cpu().numpy()[clear], tb[clear])


# around the sizes where the tail kernel's launch changes: one path per warp,
# less than a warp's lanes, 640k and 2M paths in the wave, and several waves
@pytest.mark.parametrize("W,H,spp,wave", [(1, 1, 1, None), (7, 5, 3, None), (97, 61, 2, None), (331, 97, 5, None),
                                          (512, 320, 4, None), (641, 256, 4, None), (1024, 512, 4, None),
                                          (1025, 512, 4, None), (257, 129, 6, 40000)])
def test_render_does_not_depend_on_the_tail_launch(mrs, W, H, spp, wave):
    sc = mrs.Scene.seeded(3, n_spheres=12, n_large=3)
    if wave:
        sc.set_wave(wave)
    a = mrs.render(sc, W, H, spp, 6, 2, seed=5, layers=True)
    sc.set_tail(40)       # no tail kernel: one launch per step
    b = mrs.render(sc, W, H, spp, 6, 2, seed=5, layers=True)
    for k in b:
        assert torch.equal(a[k], b[k]), k
