"""Rays with direction components that are zero, denormal, or so small that a
box's distance over them overflows, of either sign, from origins inside and outside
the boxes' slabs, also of a tiny direction as a whole: the closest hit over every
tree equals the oracle's bit for bit."""
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


@pytest.mark.parametrize("length", [1.0, 1e-20])
@pytest.mark.parametrize("extent", [0.5, 64.0, 20000.0])
def test_tiny_components(mrs, orc, extent, length):
    n, count = 400, 30000
    r = np.random.default_rng(int(extent * 2))
    desc = scenes.random_triangles(5, n)
    V = (extent * (r.uniform(-1, 1, (n, 1, 3)) + r.normal(0, 0.12, (n, 3, 3)))).astype(np.float32)
    desc["V"] = np.ascontiguousarray(V.reshape(desc["V"].shape))
    o = (extent * r.uniform(-1, 1, (count, 3))).astype(np.float32)
    d = r.normal(size=(count, 3))
    d *= length / np.linalg.norm(d, axis=1, keepdims=True)
    tiny = r.random((count, 3)) < 0.5
    tiny[np.arange(count), r.integers(0, 3, count)] = False
    size = r.choice([0.0, 1e-45, 1e-42, 1e-39, 4e-39, 1e-38, 3e-38, 1e-37, 1e-36, 1e-35, 1e-34, 1e-30, 1e-22], (count, 3))
    d = np.where(tiny, size * r.choice([-1.0, 1.0], (count, 3)), d).astype(np.float32)
    pr, tr = orc.cast(desc["V"], o, d)
    assert (pr >= 0).sum() > count // 10
    sc = mrs.Scene(desc)
    for tree in ("lbvh", "cluster", "hcluster"):
        sc.set_tree(tree)
        p, t = sc.cast(torch.from_numpy(o).cuda(), torch.from_numpy(d).cuda())
        assert np.array_equal(p.cpu().numpy(), pr)
        assert np.array_equal(t.cpu().numpy(), tr)
