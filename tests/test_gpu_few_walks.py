"""3D launches below 4096 walks per multiprocessor run an instantiation of the walk kernel with more
registers and fewer blocks.  A walk is fixed by its id: the records of launches on both sides of the
line equal the first records of a larger one bit for bit."""
import numpy as np
import pytest
import torch

from paper_2405_12964_gb300 import dwos, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("freq, sigma", [(3, 1.0), (12, 0.0)])
def test_both_instantiations_run_the_same_walks(freq, sigma):
    sc = scenes.sh_sphere_scene(freq=freq, lmax=2, sigma=sigma, n_query=1)
    s = dwos.Solver(0)
    s.load_scene(sc)
    line = 4096 * torch.cuda.get_device_properties(0).multi_processor_count
    big = line + 1000

    def records(n):
        return s.walk_records(sc.query, n)["rec"].view(np.uint32).reshape(n, -1)

    ref = records(big)
    for n in (1, 5000, line - 1, line):
        assert np.array_equal(records(n), ref[:n]), n
