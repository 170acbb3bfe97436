"""The caller's bound on a distance query's node visits, over triangles: a query within it passes,
one beyond it is reported, however many lanes work on it."""
import numpy as np
import pytest

from paper_2405_12964_gb300 import dwos, scenes

pytestmark = pytest.mark.gpu

STEP_LIMIT = 4


def _runs(s, q, walks, bound, differential=True):
    s.set_traversal_budget(bound)
    try:
        s.walk_records(q, walks, differential=differential)
        s.sync()
        return True
    except dwos.DwosError as err:
        assert err.status == STEP_LIMIT
        return False


def test_one_query_takes_no_more_visits_than_its_bound():
    # one walk of one step: one query, without an element to start from.  Under a bound its nodes
    # stay with one group of lanes, so what it needs is read from a run whose bound never binds
    sc = scenes.sh_sphere_scene(freq=24, lmax=3, n_query=1, K=1)
    q = np.array([[1.45, 0.2, -0.3]])
    s = dwos.Solver(0)
    s.load_scene(sc, traversal=2, max_steps=1)
    assert _runs(s, q, 1, 1 << 30, differential=False)
    st = s.stats()
    assert st["steps_main"] + st["steps_nested"] == 1
    units = st["wide_nodes_visited"]               # of 32 child slots: four nodes
    assert units > 3                               # above the nine nodes any bound allows
    for bound in range(1, 2 * units):
        # refused below what the query needs, which does not depend on the bound
        assert _runs(s, q, 1, bound, differential=False) == (bound >= units)
        assert s.stats()["wide_nodes_visited"] <= max(3, bound)


def test_one_wide_nodes_worth_of_triangles_passes_any_bound():
    # 32 elements fill one node of 32 slots: one visit
    sc = scenes.sh_sphere_scene(freq=1, lmax=1, n_query=16, K=1)
    s = dwos.Solver(0)
    s.load_scene(sc, traversal=2)
    assert s.bvh_info()["n_tree"] == 32
    for bound in (1, 2, 3):
        assert _runs(s, sc.query, 32, bound)


def test_a_deep_search_is_refused():
    sc = scenes.sh_sphere_scene(freq=24, n_query=16, K=1)
    for order in (2, 3):
        s = dwos.Solver(0)
        s.load_scene(sc, traversal=order)
        assert not _runs(s, sc.query, 32, 1)
        assert _runs(s, sc.query, 32, 0)
