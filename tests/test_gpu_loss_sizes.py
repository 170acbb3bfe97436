"""The squared loss at point counts around its kernel's line between one block and a cluster."""
import numpy as np
import pytest
import torch

from paper_2405_12964_gb300 import dwos, scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 255, 256, 257, 1023, 1024, 1025, 2049, 16384])
def test_loss_equals_the_sum_over_the_walks(n):
    sc = scenes.disk_scene("mapped_cos", n_seg=64, n_query=n, seed=n)
    ref = np.random.default_rng(n).normal(size=n).astype(np.float32)
    s = dwos.Solver(0)
    s.load_scene(sc)
    walks = 8
    u = s.walk_records(sc.query, walks)["rec"]["u"].reshape(n, walks).astype(np.float64)
    mean = u.mean(1)
    want = 0.5 * ((mean - ref) ** 2).sum()
    # a warp's walks of one point are summed in FP32 (at most five roundings of 2^-24 of their
    # absolute sum), everything else in FP64
    d = 5 * 2.0 ** -24 * np.abs(u).mean(1) + 2.0 ** -50 * np.abs(mean)
    tol = (np.abs(mean - ref) * d + d * d).sum() + n * 2.0 ** -52 * want
    assert abs(float(s.grad_l2(sc.query, ref, walks)[0]) - want) <= tol
    b = dwos.Batch([(s, sc.query, walks, ref, 0)])
    b.run()
    b.synchronize()
    assert abs(float(b.out[0]["loss"]) - want) <= tol
    assert np.all(np.abs(b.out[0]["u_mean"].cpu().numpy() - mean) <= d)
