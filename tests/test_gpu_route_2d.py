"""Walks among segments do not depend on the search order, at sizes around the lines of the routed
order (3): 32 segments per lane that needs the tree, 256 in all, a wide node's 32 slots."""
import numpy as np
import pytest

from paper_2405_12964_gb300 import dwos, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [16, 31, 32, 33, 64, 97, 160, 255, 256, 257, 300])
@pytest.mark.parametrize("kind", ["disk", "star"])     # every lane needs the tree; few do
def test_orders_agree(kind, n):
    if kind == "disk":
        sc = scenes.disk_scene("mapped_cos", n_seg=n, n_query=23, seed=n)
    else:
        sc = scenes.star_box_scene(n_seg=n, n_modes=2, n_query=23, K=2, seed=n)
    rec = []
    for order in (0, 2, 3):
        s = dwos.Solver(0)
        s.load_scene(sc, traversal=order)
        # (in the disk: clear of the polygon's edges)
        r = s.walk_records(sc.query * (0.5 if kind == "disk" else 1.0), 300)["rec"].view(np.uint32)
        s.sync()
        rec.append(r)
    assert np.array_equal(rec[0], rec[1]) and np.array_equal(rec[0], rec[2])
