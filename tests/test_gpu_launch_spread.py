"""Launches that cannot fill every lane put a few walks on each warp.  A walk is
fixed by its id, so the records of a small launch equal the first records of a
large one with full warps bit for bit, whatever the number of walks: one, around
a warp's 32 lanes, and around the number of warps of a launch with one block of
one warp on each of the 152 multiprocessors.
"""
import numpy as np
import pytest

from paper_2405_12964_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def Solver():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_12964_gb300 import build
    build.build()
    from paper_2405_12964_gb300.dwos import Solver as S
    return S


@pytest.mark.parametrize("which", ["star", "disk", "sphere", "thermal"])
def test_small_launches_run_the_same_walks(Solver, which):
    sc = {"star": lambda: scenes.star_box_scene(n_seg=512, n_query=1),
          "disk": lambda: scenes.disk_scene("screened_1", n_query=1),
          "sphere": lambda: scenes.sh_sphere_scene(freq=6, n_query=1),
          "thermal": lambda: scenes.thermal_scene(n_query=1)}[which]()
    s = Solver(0)
    s.load_scene(sc, block_size=32, blocks_per_sm=1)
    n = 152 * 32 + 5                              # more walks than one warp per multiprocessor has lanes
    ref = s.walk_records(sc.query, n)["rec"].view(np.uint32).reshape(n, -1)
    for shape in (dict(block_size=32, blocks_per_sm=1), dict(block_size=0, blocks_per_sm=0)):
        s.set_options(**shape)
        for w in (1, 2, 31, 32, 33, 151, 152, 153, 303, 305, n - 6, n):
            got = s.walk_records(sc.query, w)["rec"].view(np.uint32).reshape(w, -1)
            assert np.array_equal(got, ref[:w]), (shape, w)
    st = s.stats()
    assert st["steps_main"] > 0
