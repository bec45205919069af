"""Grazing hits whose leaf passes its box test by rounding alone: the boxes above the
leaf, tested as centres and half extents, let them through too, so that the closest
hit is the oracle's.  Each ray was found by a search over hits near a side of a small
distant box, for those whose entry into the box as centre and half extent is more than
8 x 2^-24 behind its exit (3 in a million)."""
import numpy as np
import pytest

from synth import scenes

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# float32 bits: a triangle's three vertices, the ray's origin and direction
RAYS = [
    "3fc1a662 bee3e461 3ee1b518 3fc07252 bee3e461 3ee119fc 3fc1a662 bee892d7 3ee1ba27 42e50012 c2cb1e66 415ee105 bf3e039f 3f2a0c0e bdb57af6",
    "bfbf7c2b 3f14041e bfae554d bfc0288a 3f14041e bfae3383 bfbf7c2b 3f165e2a bfae6eba 43310d7e 42ca5c7a c209c7ed bf5c2ec6 bef81f3b 3e2330c6",
    "3fd6b5ea bfcc2317 3fc9348e 3fddd11c bfcc2317 3fc8ba0f 3fd6b5ea bfcd4a21 3fc8ccce c312afd4 c4828c80 c3b84bd1 3e08142d 3f6f1c92 3ea9c19c",
    "bfad0f69 3f424f07 3f874e30 bfa5503d 3f424f07 3f87b6cd bfad0f69 3f4073b6 3f86f55a 446ce445 44af54a9 43fe199c bf0976b9 bf4b150c be92eedb",
    "bfa4dbab bfeb45ff 3fd0e0b0 bfa5478e bfeb45ff 3fd1094a bfa4dbab bfe95db3 3fd0e085 4510deef c510f197 c4670dec bf2e47a4 3f2e21da 3e8b25c0",
    "bf7c945d 3fb8e68c bde5633e bf73abfa 3fb8e68c bde9979b bf7c945d 3fb7b6e9 bdebb23b c526188b 45821375 449d06bb 3f0580eb bf511bf0 be7c8b5d",
    "be96dcd4 beaa1ba2 bf9b2236 bea36afa beaa1ba2 bf9b1fb1 be96dcd4 beb40040 bf9b38f8 c58e0a6a 45fb40b8 438cd555 3efbd540 bf5ec12e bcfac86f",
    "3fc54fd3 3fcaf8d9 bf9c7458 3f9cbc62 3fcaf8d9 bf9f10c0 3fc54fd3 3fd82fb9 bf9e7e71 c584d41a c63bf0db 4511d165 3ea7d745 3f6d6ce8 be3848a9",
    "bf103a49 3f7a28aa 3ff2e395 bf0ea5bf 3f7a28aa 3ff2d75a bf103a49 3f765348 3ff2e2c2 46323bbd c64310f3 c4254b4d bf2c8bc3 3f3cd8e9 3d207891",
    "3f1329c1 3fa19de5 bf82aba8 3ebcb400 3fa19de5 bf80496f 3f1329c1 3fb3e43e bf7ecc8c 45dfd0bc 46a045c0 455a3c67 bea69dfe bf6ea18f be228633",
]


@pytest.mark.parametrize("k", range(len(RAYS)))
def test_grazing_hit_passes_the_tree(orc, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2106_12802_gb300 as mrs
    a = np.array([int(x, 16) for x in RAYS[k].split()], np.uint32).view(np.float32).reshape(5, 3)
    # the triangle among 63 small ones far apart (none of them in the way)
    n = 64
    desc = scenes.random_triangles(5, n)
    r = np.random.default_rng(k)
    V = (r.uniform(-3e4, 3e4, (n, 1, 3)) + r.uniform(-1, 1, (n, 3, 3))).astype(np.float32)
    V[0] = a[:3]
    desc["V"] = np.ascontiguousarray(V.reshape(desc["V"].shape))
    pr, tr = orc.cast(desc["V"], a[3:4], a[4:5])
    assert pr[0] == 0
    sc = mrs.Scene(desc)
    for tree in ("lbvh", "cluster", "hcluster"):
        sc.set_tree(tree)
        p, t = sc.cast(torch.from_numpy(a[3:4].copy()).cuda(), torch.from_numpy(a[4:5].copy()).cuda())
        assert int(p[0]) == 0 and float(t[0]) == float(tr[0])
