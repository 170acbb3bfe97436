"""The tree searches at the sizes and shapes where they can go wrong: element
counts around a wide node's slots (32 segments, 8 triangles) and their powers,
one element, outsized elements beside the tree, patches from flat to closed,
clusters that make the tree deep, surfaces far from the origin, coincident
elements.  Search orders 0 (one query per lane, binary tree), 2 and 3 (the
warp's search of the wide tree) measure the same elements with the same
arithmetic, so distances agree bit for bit; they equal brute force in 64 bits
up to FP32 rounding: a distance is formed from coordinate differences (two
roundings of up to |p| 2^-24 each per axis) and some ten operations.
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


def _brute(v, e, p):
    """Distance of each point to the closest element, in 64 bits."""
    out = np.full(len(p), np.inf)
    v, p = v.astype(np.float32).astype(np.float64), p.astype(np.float32).astype(np.float64)
    for el in e:
        a, b = v[el[0]], v[el[1]]
        seg = [(a, b)] if len(el) == 2 else [(a, b), (b, v[el[2]]), (v[el[2]], a)]
        for s, t in seg:
            u = np.clip(((p - s) @ (t - s)) / ((t - s) @ (t - s)), 0, 1)
            out = np.minimum(out, np.linalg.norm(p - s - u[:, None] * (t - s), axis=1))
        if len(el) == 3:                          # inside the prism over the face
            c = v[el[2]]
            n = np.cross(b - a, c - a)
            n /= np.linalg.norm(n)
            h = (p - a) @ n
            q = p - h[:, None] * n
            m = np.stack([np.cross(t - s, q - s) @ n for s, t in seg], 1)
            out = np.where((m >= 0).all(1) | (m <= 0).all(1), np.minimum(out, np.abs(h)), out)
    return out


def _soup(dim, n, rng, size=0.02, spread=1.0, c=None):
    """Segments, or equilateral triangles, of half length / radius `size`, turned at random."""
    c = rng.uniform(-spread, spread, size=(n, 1, dim)) if c is None else c
    r = np.linalg.qr(rng.normal(size=(n, dim, dim)))[0]
    a = 2 * np.pi * np.arange(dim) / dim
    v = np.einsum("vk,nkd->nvd", np.stack([np.cos(a), np.sin(a)], 1), r[:, :2])
    return (c + size * v).reshape(-1, dim), np.arange(n * dim, dtype=np.int32).reshape(n, dim)


def _case(name, dim, rng):
    if name.startswith("n"):
        return _soup(dim, int(name[1:]), rng)
    if name == "outsized":                        # 3 elements much larger than the other 200
        v, e = _soup(dim, 200, rng, size=0.002, spread=0.3)
        w, f = _soup(dim, 3, rng, size=2.0)
        return np.concatenate([v, w]), np.concatenate([e, f + len(v)]).astype(np.int32)
    if name == "deep":                            # elements at 0.85^k of sizes in proportion: a chain of splits
        c = np.zeros((40, 1, dim))
        c[:, 0, 0] = 0.85 ** np.arange(40)
        return _soup(dim, 40, rng, size=0.05 * c[:, :, :1], c=c)
    if name == "coincident":                      # equal keys: the tree splits by index
        v, e = _soup(dim, 1, rng, size=0.3)
        return v, np.repeat(e, 100, axis=0)
    if name == "far":                             # a patch a thousand sizes from the origin
        v, e = _soup(dim, 300, rng)
        return v + 1000.0, e
    v, e = scenes.icosphere(9) if dim == 3 else scenes.radial_polygon(900, lambda t: 1 + 0.2 * np.cos(5 * t))[1:]
    return v, e


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("name", ["n1", "n2", "n7", "n8", "n9", "n31", "n32", "n33", "n63", "n64", "n65", "n256",
                                  "n257", "n513", "n1025", "outsized", "deep", "coincident", "far", "closed"])
def test_search_orders_agree_with_brute_force(Solver, dim, name):
    rng = np.random.default_rng(7 * dim + len(name))
    v, e = _case(name, dim, rng)
    at, span = v.mean(0), np.abs(v - v.mean(0)).max() + 0.1
    p = np.concatenate([at + rng.uniform(-1.5, 1.5, size=(997, dim)) * span,
                        v[e].mean(1)[rng.integers(0, len(e), 200)] + rng.normal(0, 1e-3, size=(200, dim)),
                        at + rng.normal(size=(3, dim)) * 100 * span]).astype(np.float32)
    want = _brute(v, e, p)
    d = {}
    for order in (0, 2):
        s = Solver(0)
        s.set_options(traversal=order)
        s.set_boundary(v, e)
        d[order] = s.closest_point(p)[0].cpu().numpy()
        s.sync()
    assert np.array_equal(d[0], d[2])
    scale = np.abs(p).max(1) + np.abs(v).max()
    assert np.all(np.abs(d[0] - want) <= 2 ** -24 * (4 * np.sqrt(dim) * scale + 10 * want) + 1e-7)


@pytest.mark.parametrize("freq", [1, 2, 6, 17])
def test_walks_over_triangles_do_not_depend_on_the_search(Solver, freq):
    # the box's triangles outsized or not, a source, nested walks; after a refit too
    sc = scenes.sh_sphere_scene(freq=freq, lmax=3, n_query=37)
    rec = []
    for order in (0, 2, 3):
        s = Solver(0)
        s.load_scene(sc, traversal=order)
        a = s.walk_records(sc.query, 48)["rec"].view(np.uint32)
        s.set_boundary(sc.reference_vertices(), sc.elem, sc.jac)
        s.set_dirichlet_mapped(sc.g_vert)
        s.set_params(sc.theta0 * 1.1)
        b = s.walk_records(sc.query, 48)["rec"].view(np.uint32)
        s.sync()
        rec.append(np.concatenate([a, b]))
    assert np.array_equal(rec[0], rec[1]) and np.array_equal(rec[0], rec[2])
