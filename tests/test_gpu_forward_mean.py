"""The mean of u and its standard error do not depend on whether derivatives are asked for."""
import numpy as np
import pytest
import torch

from paper_2405_12964_gb300 import dwos, scenes

pytestmark = pytest.mark.gpu


# clusters of one, two, four and eight blocks for the derivatives; walks of every remainder
@pytest.mark.parametrize("points, walks", [(1, 1), (3, 4096), (5, 63), (64, 1000), (150, 257), (300, 600), (700, 300)])
def test_same_bits_with_and_without_derivatives(points, walks):
    sc = scenes.disk_scene("mapped_cos", n_query=points, seed=points)
    s = dwos.Solver(0)
    s.load_scene(sc)
    x = torch.as_tensor(np.asarray(sc.query, np.float32)).cuda()
    plain, both = s.eval(x, walks), s.eval(x, walks, grad=True)
    s.sync()
    for k in ("u", "u_se"):
        assert torch.equal(plain[k], both[k])
