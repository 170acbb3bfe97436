"""The binary tree's boxes after a build and after a refit: searches from the root, which descend by
them alone, against every element measured in FP64, at sizes around the blocks of 8, 64 and 512 leaves
the boxes are made from."""
import numpy as np
import pytest
import torch

from paper_2405_12964_gb300 import dwos, scenes

pytestmark = pytest.mark.gpu


def _distances(p, v, e):
    """Distance of every point from the closest element, FP64."""
    a = v[e[:, 0]]
    out = []
    for x in p:
        if v.shape[1] == 2:
            d = v[e[:, 1]] - a
            t = np.clip(((x - a) * d).sum(1) / (d * d).sum(1), 0, 1)
            out.append(np.linalg.norm(a + t[:, None] * d - x, axis=1).min())
        else:
            out.append(_triangles(x, a, v[e[:, 1]], v[e[:, 2]]).min())
    return np.array(out)


def _triangles(x, a, b, c):
    n = np.cross(b - a, c - a)
    n2 = (n * n).sum(1)
    # inside the prism over the triangle: the plane's distance; else the closest edge
    inside = np.ones(len(a), bool)
    best = np.full(len(a), np.inf)
    for p, q in ((a, b), (b, c), (c, a)):
        inside &= (np.cross(q - p, x - p) * n).sum(1) >= 0
        d = q - p
        t = np.clip(((x - p) * d).sum(1) / (d * d).sum(1), 0, 1)
        best = np.minimum(best, np.linalg.norm(p + t[:, None] * d - x, axis=1))
    return np.where(inside, np.abs(((x - a) * n).sum(1)) / np.sqrt(n2), best)


@pytest.mark.parametrize("size", [3, 7, 8, 9, 63, 64, 65, 511, 512, 513, 1025, 4097])
def test_segments(size):
    rng = np.random.default_rng(size)
    ang = np.sort(rng.random(size)) * 2 * np.pi
    v = (1 + 0.2 * rng.random(size))[:, None] * np.stack([np.cos(ang), np.sin(ang)], 1)
    e = np.stack([np.arange(size), (np.arange(size) + 1) % size], 1).astype(np.int32)
    _check(rng, v, e, rng.normal(size=(size, 2, 1)) * 0.01)


@pytest.mark.parametrize("freq", [1, 2, 5, 6, 15])      # 20 to 4500 triangles
def test_triangles(freq):
    sc = scenes.sh_sphere_scene(freq=max(freq, 1), lmax=2, n_query=4)
    tri = np.asarray(sc.elem)
    _check(np.random.default_rng(freq), np.asarray(sc.vert, np.float64), tri, np.zeros((len(sc.vert), 3, 1)) + 0.01)


def _check(rng, v, e, jac):
    dim = v.shape[1]
    p = rng.uniform(-1.5, 1.5, size=(200, dim)).astype(np.float32)
    s = dwos.Solver(0)
    for traversal in (0, 3):
        s.set_options(traversal=traversal)
        s.set_boundary(v, e, jac)
        for theta in (None, 1.0, -3.0):
            if theta is not None:
                s.set_params(torch.tensor([theta], dtype=torch.float32).cuda())
            got = s.closest_point(p)[0]
            want = _distances(p.astype(np.float64), np.asarray(s.current_vertices(), np.float64), e)
            # FP32 differences of coordinates of size 2: a few units of 2^-23 absolute
            assert np.abs(got.double().cpu().numpy() - want).max() <= 16 * 2.0 ** -23


@pytest.mark.parametrize("size", [3, 31, 32, 33, 64, 65, 1025, 4097, 40000])
def test_inside(size):
    rng = np.random.default_rng(size)
    ang = np.arange(size) * 2 * np.pi / size
    v = (1 + 0.3 * np.cos(5 * ang))[:, None] * np.stack([np.cos(ang), np.sin(ang)], 1)
    v = v.astype(np.float32)
    e = np.stack([np.arange(size), (np.arange(size) + 1) % size], 1).astype(np.int32)
    p = rng.uniform(-1.5, 1.5, size=(300, 2)).astype(np.float32)
    s = dwos.Solver(0)
    s.set_boundary(v, e)
    got = s.inside(p).cpu().numpy()
    v, p = v.astype(np.float64), p.astype(np.float64)
    a, b = v, np.roll(v, -1, 0)
    want = np.zeros(len(p), int)
    for i, x in enumerate(p):      # crossings of the ray towards +x
        up = (a[:, 1] > x[1]) != (b[:, 1] > x[1])
        cross = a[up, 0] + (x[1] - a[up, 1]) * (b[up, 0] - a[up, 0]) / (b[up, 1] - a[up, 1])
        want[i] = (cross > x[0]).sum() & 1
    clear = _distances(p, v, e) > 1e-5       # away from the boundary both are exact
    assert (got[clear] == want[clear]).all()
