"""The tree builds' radix sort at the edges of its tiles and of its variants
(4 or 8 keys a thread, tile counts summed by the scatter blocks or scanned): the
exported order is the stable order of the Morton codes."""
import numpy as np
import pytest
import torch  # noqa: F401

import paper_2106_12802_gb300 as mrs
from test_gpu_render import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 1023, 1024, 1025, 2049, 262143, 262144, 262145, 2097152, 2097153])
def test_order_is_the_stable_order_of_the_codes(n):
    desc = scenes.random_triangles(7, min(n, 5000))
    if n > 5000:
        # many equal codes: copies of the same triangles
        desc["V"] = np.tile(desc["V"], (n // 5000 + 1, 1, 1))[:n].copy()
        desc["tri_mat"] = np.zeros(n, np.int32)
        desc["tri_light"] = np.full(n, -1, np.int32)
    sc = mrs.Scene(desc)
    g = sc.export_bvh()
    sc.close()
    assert np.array_equal(g["order"], np.argsort(g["morton"], kind="stable"))
