"""Searches over thin triangles: the warp's search (order 2, oriented boxes) against the search of
one query per lane (order 0, axis-aligned boxes), which measure elements with the same arithmetic.

Copies of a triangle lie close together, so that a box that exceeds its triangle's distance by a
few parts in a million prunes the closest one.  Queries keep half an element's length or more away:
an element is then measured with an error of a few 2^-24 of its distance, below the searches'
allowance, and both orders find the same minimum bit for bit.
"""
import numpy as np
import pytest
import torch

from paper_2405_12964_gb300 import dwos

pytestmark = pytest.mark.gpu


def _triangles(kind, ratio, rng, groups=64, copies=8):
    """(n, 3, 3) triangles of length about 1 and height/length `ratio`: needles (one sharp corner)
    or caps (one obtuse corner), the corner at any of the three vertices."""
    n = groups * copies

    def each(x):
        return np.repeat(x, copies, 0)

    u = each(rng.normal(size=(groups, 3)))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    w = np.cross(u, each(rng.normal(size=(groups, 3))))
    w /= np.linalg.norm(w, axis=1, keepdims=True)
    shift = rng.normal(size=(n, 3))
    shift *= (10 ** rng.uniform(-6, -2, size=n) / np.linalg.norm(shift, axis=1))[:, None]
    a = each(rng.uniform(-3, 3, size=(groups, 3))) + shift
    if kind == "needle":
        ln = rng.uniform(0.5, 1.5, size=(2, n, 1))
        t = [a, a + ln[0] * u, a + ln[1] * (u + ratio * w)]
    else:
        t = [a + rng.uniform(0.3, 0.7, size=(n, 1)) * u + ratio * w, a, a + u]
    t = np.stack(t, 1)
    roll = rng.integers(0, 3, n)
    return t[np.arange(n)[:, None], (np.arange(3) + roll[:, None]) % 3].astype(np.float32)


def _proper(t):
    """Without those whose cross product FP32 coordinates have flattened."""
    t64 = t.astype(np.float64)
    return t[(np.cross(t64[:, 1] - t64[:, 0], t64[:, 2] - t64[:, 0]) ** 2).sum(1) > 1e-18]


def _queries(t, rng, n=20000):
    d = rng.normal(size=(n, 3))
    d *= (10 ** rng.uniform(0, 2, size=n) / np.linalg.norm(d, axis=1))[:, None]
    return (t.mean(1)[rng.integers(0, len(t), n)] + d).astype(np.float32)


def _elements(n):
    return np.arange(3 * n, dtype=np.int32).reshape(n, 3)


@pytest.mark.parametrize("scale", [1.0, 1e-6, 1e6])
@pytest.mark.parametrize("ratio", [1e-2, 1e-3, 1e-4, 1e-5, 1e-6])
@pytest.mark.parametrize("kind", ["needle", "cap"])
def test_thin_triangles(kind, ratio, scale):
    rng = np.random.default_rng(5)
    t = _proper(_triangles(kind, ratio, rng))
    p = _queries(t, rng) * np.float32(scale)
    t = t * np.float32(scale)
    d = {}
    for order in (0, 2):
        s = dwos.Solver(0)
        s.set_options(traversal=order)
        s.set_boundary(t.reshape(-1, 3), _elements(len(t)))
        d[order] = s.closest_point(p)[0].cpu().numpy()
        s.sync()
    assert np.array_equal(d[0], d[2])


@pytest.mark.parametrize("ratio", [1e-3, 1e-5, 1e-6])
def test_triangles_flattened_by_a_refit(ratio):
    rng = np.random.default_rng(6)
    thin = _triangles("cap", ratio, rng)
    wide = _triangles("cap", 0.5, np.random.default_rng(6))
    p = _queries(thin, rng)
    d = {}
    for order in (0, 2):
        s = dwos.Solver(0)
        s.set_options(traversal=order)
        s.set_boundary(wide.reshape(-1, 3), _elements(len(wide)), (thin - wide).reshape(-1, 3, 1))
        s.set_params(torch.ones(1, device="cuda"))
        d[order] = s.closest_point(p)[0].cpu().numpy()
        s.sync()
    assert np.array_equal(d[0], d[2])


@pytest.mark.parametrize("n", [2000, 60000])          # sharp corners of 3e-3 and 1e-4
def test_walks_in_a_double_fan(n):
    # two fans of triangles with a common rim, closed; the walks start inside
    a = 2 * np.pi * np.arange(n) / n
    v = np.concatenate([np.stack([np.cos(a), np.sin(a), 0 * a], 1), [[0, 0, 0.7], [0, 0, -0.6]]])
    i, j = np.arange(n), (np.arange(n) + 1) % n
    e = np.concatenate([np.stack([i * 0 + n, i, j], 1), np.stack([i, i * 0 + n + 1, j], 1)]).astype(np.int32)
    rng = np.random.default_rng(n)
    q = rng.uniform(-0.3, 0.3, size=(64, 3))
    rec = []
    for order in (0, 2, 3):
        s = dwos.Solver(0)
        s.set_options(traversal=order, K=1, eps=0.1, h=0.15, check_inside=0)
        s.set_boundary(v, e, np.ones((len(v), 3, 1)))
        s.set_dirichlet_mapped(v[:, 0])
        s.set_pde(1.0, 0.5)
        rec.append(s.walk_records(q, 64)["rec"].view(np.uint32))
        s.sync()
    assert np.array_equal(rec[0], rec[1]) and np.array_equal(rec[0], rec[2])
