"""A render's first bounce made in the trace and shading kernels (tail from
bounce 1 or later) against the one that reads every path's state from memory
(tail from bounce 0): the same bits, for sample counts that are multiples of 8,
of 4 and neither, windows, the extra layers, escaping rays, and batched jobs
that start at any path."""
import pytest
import torch

import paper_2106_12802_gb300 as mrs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def scenes():
    mrs.load()
    a, b = mrs.Scene.seeded(5), mrs.Scene.seeded(11)
    yield a, b
    a.close()
    b.close()


@pytest.mark.parametrize("spp", [1, 3, 4, 8, 12, 16, 24])
@pytest.mark.parametrize("depth", [0, 1, 5])
def test_render_does_not_depend_on_where_the_tail_starts(scenes, spp, depth):
    sc = scenes[0]
    out = []
    for tail in (0, 1, 3, 40):
        sc.set_tail(tail)
        out.append(mrs.render(sc, 37, 29, spp, depth, 3, 9))
    sc.set_tail(-1)
    for o in out[1:]:
        assert all(torch.equal(out[0][k], o[k]) for k in out[0])


@pytest.mark.parametrize("W,H,spp", [(1, 1, 1), (69, 71, 1), (278, 280, 1), (411, 379, 1), (556, 560, 1), (300, 277, 4)])
def test_pairs_of_lanes(scenes, W, H, spp):
    # a path a pair of lanes (tail from bounce 0): a warp part filled, filled, and
    # refilled from the queue; past the rule's end (the last) a path a lane
    for sc in scenes:
        sc.set_tail(0)
        a = mrs.render(sc, W, H, spp, 6, 3, 4)
        sc.set_tail(40)
        b = mrs.render(sc, W, H, spp, 6, 3, 4)
        sc.set_tail(-1)
        assert all(torch.equal(a[k], b[k]) for k in a)


@pytest.mark.parametrize("spp", [6, 8])
def test_layers_of_a_window(scenes, spp):
    res = []
    for tail in (0, 2):
        ctx = mrs.RenderContext()
        ctx.set_tail(tail)
        res.append(mrs.render(scenes[0], 64, 48, spp, 4, 3, 2, ctx=ctx, grid=2, layers=True, window=(5, 7, 31, 23)))
        ctx.close()
    assert all(torch.equal(res[0][k], res[1][k]) for k in res[0])


def test_batched_jobs(scenes):
    jobs = [{"scene": scenes[i % 2], "W": w, "H": h, "spp": spp, "max_depth": 3, "seed": i}
            for i, (w, h, spp) in enumerate([(16, 8, 8), (7, 5, 3), (9, 9, 16), (8, 8, 8), (5, 5, 1), (6, 6, 4)])]
    res = []
    for tail in (0, 2):
        ctx = mrs.RenderContext()
        ctx.set_tail(tail)
        res.append(mrs.render_batch(ctx, jobs))
        ctx.close()
    for a, b in zip(*res):
        assert all(torch.equal(a[k], b[k]) for k in a)
