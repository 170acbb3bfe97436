"""Per-point means, derivatives and standard errors against the walks' own records in FP64."""
import numpy as np
import pytest
import torch

from paper_2405_12964_gb300 import dwos, scenes

pytestmark = pytest.mark.gpu


# one column of derivatives, a warp's width, the columns of one block and one more; clusters of
# one, two, four and eight blocks; walks that leave every remainder of a block's chunk
@pytest.mark.parametrize("n_param, points, walks", [(1, 3, 1), (17, 5, 63), (17, 64, 1000), (32, 700, 130), (128, 2, 257),
                                                    (129, 9, 128), (300, 1, 777)])
def test_forward_derivatives(n_param, points, walks):
    sc = scenes.disk_scene("mapped_cos", n_seg=96, n_query=points, seed=3)
    rng = np.random.default_rng(n_param)
    n_vert = len(sc.vert)
    jac = rng.normal(size=(n_vert, 2, n_param)).astype(np.float32)
    dg = rng.normal(size=(n_vert, n_param)).astype(np.float32)
    s = dwos.Solver(0)
    s.load_scene(sc)
    s.set_boundary(sc.vert, sc.elem, jac)
    s.set_dirichlet_mapped(sc.g_vert, dg)
    out = {k: v.double().cpu().numpy() for k, v in s.eval(sc.query, walks, grad=True).items()}
    rec = s.walk_records(sc.query, walks)["rec"].reshape(points, walks)
    u = rec["u"].astype(np.float64)
    du = np.zeros((points, walks, n_param))
    hit = rec["elem"] >= 0
    vid = np.asarray(sc.elem)[np.where(hit, rec["elem"], 0)]
    bary = np.stack([np.float32(1) - rec["b1"] - rec["b2"], rec["b1"]], -1).astype(np.float64)
    for i in range(2):
        for j in range(0, n_param, 32):
            c = slice(j, min(j + 32, n_param))
            cj = np.einsum("pwk,pwkn->pwn", rec["c"][..., :2].astype(np.float64), jac[vid[..., i]][..., c].astype(np.float64))
            du[..., c] += bary[..., i, None] * (cj + dg[vid[..., i]][..., c])
    du[~hit] = 0.0

    def check(name, values, tol):
        m = values.mean(1)
        se = values.std(1, ddof=1) / np.sqrt(walks) if walks > 1 else 0.0 * m
        scale = np.abs(values).max() + 1e-30
        # the FP64 sums; the variance is a difference of sums of squares, hence the square root
        assert np.abs(out[name] - m).max() <= tol * scale
        assert np.abs(out[name + "_se"] - se).max() <= (tol + 1e-7) * scale

    check("u", u, 1e-13)
    # a walk's derivative is two FP32 fused products and a sum: 3 x 2^-24 of its terms' size, which
    # is at most (|c_x| + |c_y|) |J| + |dg|; relative to the largest term
    size = np.abs(rec["c"][..., :2]).sum(-1).max() * np.abs(jac).max() + np.abs(dg).max()
    check("du", du, 3 * 2.0 ** -24 * size / (np.abs(du).max() + 1e-30) + 1e-13)
    plain = s.eval(sc.query, walks)
    assert np.abs(plain["u"].double().cpu().numpy() - out["u"]).max() <= 1e-13 * np.abs(u).max()
