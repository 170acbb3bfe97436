"""The warp's search of triangles with few queries, whose groups of lanes take nodes from each
other's stacks: a push by one lane of a group follows every lane's read of the stack."""
import numpy as np
import pytest

from paper_2405_12964_gb300 import dwos, scenes

pytestmark = pytest.mark.gpu


# fewer queries than groups, one per group, more; a last warp of every fill
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 31, 33, 129])
def test_shared_stacks(n):
    v, e = scenes.icosphere(40)
    rng = np.random.default_rng(n)
    p = rng.normal(size=(n, 3))
    # near the centre almost every box is within the bound: the longest searches
    p *= (np.where(np.arange(n) % 3 == 0, 1e-3, 0.9) / np.linalg.norm(p, axis=1))[:, None]
    got = {}
    for order in (0, 2):
        s = dwos.Solver(0)
        s.set_options(traversal=order)
        s.set_boundary(v, e)
        got[order] = [o.cpu().numpy() for o in s.closest_point(p)[:2]]
        s.sync()
    assert np.array_equal(got[0][0], got[2][0]) and np.array_equal(got[0][1], got[2][1])
