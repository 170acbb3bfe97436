"""The work that users of this library have it do, as cases whose passes can be timed.

A case names a workload (`kind`) and its sizes.  The kinds are the calls of the
library's own optimisation loops, examples and benchmark:

  opt      an optimisation iteration: new parameters (tree refit) and the gradient of the squared loss
  disk     forward mode: u, du/dtheta and their standard errors on a disk
  star     the gradient of the squared loss on the 2D shape-from-diffusion geometry
  sphere   the same on the 3D thermal-design geometry (triangles, a source term)
  fit      the autograd function in 3D: forward value and backward pass through a torch loss
  thermal  walks on stars in 2D (a wire under an insulating slab), reflecting or with Neumann data
  cube     walks on stars in 3D (two Dirichlet and four Neumann faces)
  batch    many problems of uneven size in one captured graph
  cvgrad   a gradient with the learned control variate: the network's inference and corrected walks
  cvtrain  one training step of the control-variate network

Walk counts per point are multiples of the U-statistic batch size where a
gradient of the squared loss is asked for; point counts and meshes are any size.
"""
import math
import random

import numpy as np
import torch

from paper_2405_12964_gb300 import dwos, scenes


def listed():
    return [
        # the noisy-gradient study's cheapest iteration: 2 walks per point, all launch and walk latency
        dict(name="opt_noisy", kind="opt", n_seg=4096, points=256, walks=2),
        # the same study with its many-point profile, at the walk count its annealing ends with
        dict(name="opt_profile", kind="opt", n_seg=4096, points=16384, walks=128),
        # a closed-form disk as examples and the smoke run use it, screened
        dict(name="disk_forward", kind="disk", variant="screened_1", n_seg=128, points=64, walks=1024),
        # the benchmark's headline workload
        dict(name="star_grad", kind="star", n_seg=4096, modes=32, points=256, walks=4096, K=2, sigma=10.0),
        # the 3D workload: a 200k-triangle surface, many observation points
        dict(name="sphere_grad", kind="sphere", freq=100, lmax=8, points=4096, walks=1024, K=2),
        # a coarser surface fitted through torch autograd, odd sizes
        dict(name="sphere_fit", kind="fit", freq=23, lmax=3, points=333, walks=500, K=1),
        # the 2D thermal design read on the slab, reflecting
        dict(name="thermal_grad", kind="thermal", n_wire=64, n_slab=40, points=32, walks=8192, flux=0.0),
        # the same with a heat flux through the slab's surface
        dict(name="thermal_flux_grad", kind="thermal", n_wire=64, n_slab=40, points=32, walks=4096, flux=0.5),
        # a 3D mixed boundary
        dict(name="cube_grad", kind="cube", m=4, points=64, walks=4096, sigma=0.0, f=0.0),
        # independent problems, 2D and 3D in turn, as one graph
        dict(name="batch_mixed", kind="batch", problems=8, max_elems=50000, layout=1),
        # an iteration's estimate in the control-variate loop, middle of its annealing
        dict(name="cv_grad", kind="cvgrad", n_seg=4096, points=256, walks=512),
        # an iteration's training on the thinned walks
        dict(name="cv_train", kind="cvtrain", rows=65536),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _split(rng, most, p_lo, p_hi, w_lo, w_hi, step):
    """Points and walks per point, the walks a multiple of `step`, at most about `most` walks in all."""
    p = _log(rng, p_lo, p_hi)
    return dict(points=p, walks=max(step, _log(rng, w_lo, max(w_lo, min(w_hi, most // p))) // step * step))


def _batch_sizes(case):
    """The problems of a batch: 2D and 3D in turn, 1000 elements or more, uneven in every size."""
    rng = random.Random(case["layout"])
    return [dict(dim=2 + i % 2, elems=_log(rng, 1000, case["max_elems"]),
                 sigma=math.exp(rng.uniform(math.log(0.01), math.log(100.0))),
                 **_split(rng, 1 << 20, 16, 2048, 256, 4096, 8)) for i in range(case["problems"])]


def draw(rng):
    kind = rng.choice(["opt", "disk", "star", "sphere", "fit", "thermal", "cube", "batch", "cvgrad", "cvtrain"])

    def split(*a):
        return _split(rng, *a)

    if kind == "opt":
        return dict(kind=kind, n_seg=_log(rng, 64, 4096), **split(1 << 21, 16, 16384, 2, 1024, 2))
    if kind == "disk":
        return dict(kind=kind, variant=rng.choice(["screened_1", "mapped_cos", "mapped_data"]),
                    n_seg=_log(rng, 16, 1024), **split(1 << 18, 8, 512, 64, 4096, 1))
    if kind == "star":
        return dict(kind=kind, n_seg=_log(rng, 64, 44436), modes=rng.choice([8, 32]), K=rng.choice([1, 2, 4]),
                    sigma=round(math.exp(rng.uniform(math.log(0.01), math.log(100.0))), 3),
                    **split(1 << 20, 16, 4096, 256, 4096, 8))
    if kind == "sphere":
        return dict(kind=kind, freq=_log(rng, 7, 100), lmax=rng.choice([3, 8]), K=rng.choice([1, 2]),
                    **split(1 << 21, 16, 4096, 64, 2048, 8))
    if kind == "fit":
        return dict(kind=kind, freq=_log(rng, 7, 50), lmax=rng.choice([2, 3, 8]), K=rng.choice([1, 2]),
                    **split(1 << 19, 8, 1024, 64, 2048, 1))
    if kind == "thermal":
        return dict(kind=kind, n_wire=_log(rng, 16, 200), n_slab=_log(rng, 10, 100), flux=rng.choice([0.0, 0.0, 0.5]),
                    **split(1 << 17, 4, 64, 128, 16384, 8))
    if kind == "cube":
        sigma = rng.choice([0.0, 2.25])
        return dict(kind=kind, m=rng.randint(2, 8), sigma=sigma, f=rng.choice([0.0, 1.0]),
                    **split(1 << 17, 4, 64, 128, 4096, 8))
    if kind == "batch":
        return dict(kind=kind, problems=rng.randint(2, 12), max_elems=_log(rng, 2000, 50000),
                    layout=rng.randrange(1 << 20))
    if kind == "cvgrad":
        return dict(kind=kind, n_seg=_log(rng, 256, 4096), **split(1 << 20, 16, 1024, 64, 4096, 8))
    return dict(kind="cvtrain", rows=_log(rng, 64, 262144))


# ------------------------------------------------------------------ inputs


def _scene(case, seed):
    """The case's geometry, data and query points, from the seed alone."""
    kind, rng = case["kind"], np.random.default_rng(seed)
    if kind == "opt":
        sc = scenes.translated_star_scene(n_seg=case["n_seg"], n_query=case["points"], seed=seed)
        sc.meta["theta"] = rng.uniform(-0.1, 0.1, 2)
    elif kind == "disk":
        sc = scenes.disk_scene(case["variant"], n_seg=case["n_seg"], n_query=case["points"], seed=seed)
    elif kind in ("star", "cvgrad"):
        sc = scenes.star_box_scene(n_seg=case["n_seg"], n_modes=case.get("modes", 32), sigma=case.get("sigma", 10.0),
                                   n_query=case["points"], K=case.get("K", 2), seed=seed)
    elif kind in ("sphere", "fit"):
        sc = scenes.sh_sphere_scene(freq=case["freq"], lmax=case["lmax"], n_query=case["points"], K=case["K"],
                                    seed=seed)
        sc.u_ref = np.zeros(case["points"])
        sc.meta["theta"] = sc.theta0 + rng.normal(0.0, 0.003, sc.n_param)
    elif kind == "thermal":
        sc = scenes.thermal_scene(offset=rng.uniform(-0.1, 0.1, 2), n_wire=case["n_wire"], n_slab=case["n_slab"],
                                  n_query=case["points"])
        if case["flux"]:
            sc.neumann_h = np.where(sc.neumann == 1, case["flux"], 0.0)
        sc.u_ref = 0.1 + 0.05 * rng.random(case["points"])
    else:
        sc = scenes.cube_neumann_scene(m=case["m"], n_query=case["points"], K=2, sigma=case["sigma"], f=case["f"],
                                       seed=seed)
        sc.u_ref = sc.query[:, 0] + 0.1 * rng.normal(size=case["points"])
    sc.seed = seed * 2654435761 % (1 << 62) + 1
    return sc


def _cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a, dtype=np.float32)).cuda()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "cvtrain":
        g = torch.Generator().manual_seed(seed)
        n = case["rows"]
        x = (2 * torch.rand(n, 2, generator=g) - 1)
        u = torch.exp(-3 * (x ** 2).sum(1)) + 0.05 * torch.randn(n, generator=g)
        q = -2.0 + torch.randn(n, generator=g)
        head = torch.arange(n) % 2 == 0            # u rows and du/dn rows, as the walks give them
        t = torch.stack([torch.where(head, u, torch.zeros(())), torch.where(head, torch.zeros(()), q)], 1)
        m = torch.stack([head.float(), (~head).float() * 0.3 * torch.rand(n, generator=g)], 1)
        return dict(kind=kind, net=dwos.ControlVariateNet(0, seed=seed), x=x.cuda(), t=t.cuda(), m=m.cuda())
    if kind == "batch":
        jobs = []
        for i, z in enumerate(_batch_sizes(case)):
            if z["dim"] == 2:
                sc = scenes.star_box_scene(n_seg=z["elems"] - 4, n_modes=8, sigma=z["sigma"], n_query=z["points"],
                                           walks=z["walks"], seed=seed + i)
            else:
                sc = scenes.sh_sphere_scene(freq=max(7, round(math.sqrt(z["elems"] / 20))), lmax=3, coef_std=0.02,
                                            sigma=z["sigma"], n_query=z["points"], walks=z["walks"], seed=seed + i)
                sc.u_ref = np.zeros(z["points"])
            sc.seed = seed * 2654435761 % (1 << 62) + 1
            s = dwos.Solver(0)
            s.load_scene(sc)
            jobs.append((s, _cuda(sc.query), sc.walks, _cuda(sc.u_ref), 0))
        b = dwos.Batch(jobs)
        b.capture()
        return dict(kind=kind, batch=b)
    sc = _scene(case, seed)
    s = dwos.Solver(0)
    # about one walk in four million over the slab runs into the step limit; 1024 steps (a phase
    # takes 13 on average) keep it from holding up the call for the default limit's 16384
    s.load_scene(sc, **(dict(max_steps=1024) if kind == "thermal" else {}))
    st = dict(kind=kind, solver=s, xq=_cuda(sc.query), walks=case["walks"],
              uref=None if sc.u_ref is None else _cuda(sc.u_ref))
    if kind in ("opt", "fit"):                     # parameters move the reference geometry
        s.set_boundary(sc.reference_vertices(), sc.elem, sc.jac)
        s.set_dirichlet_mapped(sc.g_vert, sc.dg_vert)
        st["theta"] = _cuda(sc.meta["theta"])
    if kind == "fit":
        st["target"] = _cuda(np.random.default_rng(seed + 1).random(case["points"]))
    if kind == "cvgrad":
        st["net"] = dwos.ControlVariateNet(0, seed=seed)
    return st


def run(st):
    kind = st["kind"]
    if kind == "cvtrain":
        loss = st["net"].train_step(st["x"], st["t"], st["m"], lr=2e-3)
        return {"loss": loss, "params": st["net"].params()}
    if kind == "batch":
        st["batch"].launch()
        return [(o["loss"], o["grad"], o["u_mean"]) for o in st["batch"].out]
    s = st["solver"]
    if kind == "disk":
        return s.eval(st["xq"], st["walks"], grad=True)
    if kind == "fit":
        theta = st["theta"].clone().requires_grad_(True)
        u = dwos.solve(theta, s, st["xq"], st["walks"])
        loss = 0.5 * ((u - st["target"]) ** 2).sum()
        loss.backward()
        return {"u": u.detach(), "loss": loss.detach(), "grad": theta.grad}
    if kind == "cvgrad":
        _, cv_grad, _ = st["net"].eval(st["xq"])
        out = s.grad_l2_cv(st["xq"], st["uref"], st["walks"], cv_grad=cv_grad, whole_walk=True,
                           cv_elem=s.cv_table(st["net"]))
        return {k: out[k] for k in ("loss", "grad", "u_se", "u_se_cv")}
    if kind == "opt":
        s.set_params(st["theta"])
    return s.grad_l2(st["xq"], st["uref"], st["walks"])


# ------------------------------------------------------------------ what a pass cannot do without

# Distance queries of one walk phase (measured averages) and the operations of one step: a Philox
# block (10 rounds of two 32 x 32 -> 64 products and four xors), a direction, the distance to the
# closest element and the move.
_STEPS = dict(opt=6, disk=8, star=6, sphere=9, fit=9, thermal=13, cube=16, cvgrad=6)
_STEP_OPS = {2: 130.0, 3: 170.0}
_MLP = 16 * 64 + 3 * 64 * 64 + 64 * 8              # products of one network row


def work(case):
    kind = case["kind"]
    if kind == "cvtrain":
        n = case["rows"]
        return dict(bytes=24.0 * n + 8 * 4 * dwos.MLP_NPARAM, flops=2.0 * 3 * _MLP * n)
    if kind == "batch":
        by = fl = 0.0
        for z in _batch_sizes(case):
            d, n, verts = z["dim"], z["points"], z["elems"] / (z["dim"] - 1)
            by += verts * 4 * (d + 1 + d * 16) + 4 * d * z["elems"] + n * (4 * d + 12)
            fl += n * z["walks"] * 3 * (6 if d == 2 else 9) * _STEP_OPS[d]
        return dict(bytes=by, flops=fl)
    d = 3 if kind in ("sphere", "fit", "cube") else 2
    if kind in ("sphere", "fit"):
        elems, params = 20 * case["freq"] ** 2 + 12, (case["lmax"] + 1) ** 2
        verts = 10 * case["freq"] ** 2 + 10
    elif kind == "cube":
        elems, params = 12 * case["m"] ** 2, 1
        verts = elems // 2 + 2
    else:
        elems = (case["n_wire"] + 2 * case["n_slab"] + 12) if kind == "thermal" else case["n_seg"] + 4 * (kind != "disk")
        verts = elems
        params = {"opt": 2, "thermal": 2, "disk": 19 if case.get("variant") == "mapped_data" else 17,
                  "star": 2 * case.get("modes", 32), "cvgrad": 64}[kind]
    n, K = case["points"], case.get("K", 2 if kind not in ("disk",) else 1)
    walks = n * case["walks"]
    phases = 1 + K
    if kind == "fit":
        phases = 2 + K                             # the forward values, then differential walks
    by = 4.0 * verts * (d + 1 + d * params) + 4.0 * d * elems + n * (4.0 * d + 4)
    by += 8.0 * (n * 2 * (1 + params) if kind == "disk" else params + 1)
    fl = float(walks) * phases * _STEPS[kind] * _STEP_OPS[d]
    if kind == "cvgrad":
        fl += 2.0 * 2 * _MLP * (n + elems)
    return dict(bytes=by, flops=fl)


# ------------------------------------------------------------------ the 2D walks in 64 bits
#
# The walks of a call are fixed by its Philox seed, so what a 2D call returns can be restated in
# 64 bits: brute-force closest segment, the same random numbers, the estimators' sums.  A few walks
# in a thousand take another branch in 32 bits.


def _philox(c, k0, k1):
    lo32 = 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = 0xD2511F53 * c[0], 0xCD9E8D57 * c[2]
        c = [((p1 >> 32) & lo32) ^ c[1] ^ k0, p1 & lo32, ((p0 >> 32) & lo32) ^ c[3] ^ k1, p0 & lo32]
        k0, k1 = (k0 + 0x9E3779B9) & lo32, (k1 + 0xBB67AE85) & lo32
    return [((w >> 9) * 2 + 1).double() * 2.0 ** -24 for w in c]


def _closest(x, a, b):
    """Index, parameter and distance of the closest segment of each point (ties to the lower index)."""
    idx, best = [], []
    e = b - a
    l2 = (e * e).sum(1)
    for p in x.split(max(1, (1 << 25) // len(a))):
        t = ((p[:, None, 0] - a[:, 0]) * e[:, 0] + (p[:, None, 1] - a[:, 1]) * e[:, 1]).div_(l2).clamp_(0, 1)
        d2 = (p[:, None, 0] - a[:, 0] - t * e[:, 0]).square_() + (p[:, None, 1] - a[:, 1] - t * e[:, 1]).square_()
        m = d2.min(1)
        idx.append(m.indices)
        best.append(t.gather(1, m.indices[:, None])[:, 0])
    i, t = torch.cat(idx), torch.cat(best)
    d = (x - a[i] - t[:, None] * e[i]).norm(dim=1)
    return i, t, d


def _phase64(sc, geo, x, wid, phase):
    """One walk phase from each point: (value, segment or -1, parameter, last point)."""
    a, b, g0, g1 = geo
    n, k, dev = len(x), math.sqrt(sc["sigma"]), x.device
    x, u = x.clone(), torch.zeros(n, dtype=torch.float64, device=dev)
    seg, par = torch.full((n,), -1, device=dev), torch.zeros(n, dtype=torch.float64, device=dev)
    live, step = torch.arange(n, device=dev), 0
    while len(live):
        i, t, d = _closest(x[live], a, b)
        step += 1
        end = (d < sc["eps"]) if step < 16384 else torch.ones_like(d, dtype=torch.bool)
        j = live[end]
        seg[j], par[j] = i[end], t[end]
        u[j] = g0[i[end]] + t[end] * (g1 - g0)[i[end]]
        live, r = live[~end], (d - 1e-3 * sc["eps"])[~end]
        w = wid[live]
        z = torch.zeros_like(w)
        r0 = _philox([w & 0xFFFFFFFF, w >> 32, z + step - 1, z + (phase << 8)], sc["seed"] & 0xFFFFFFFF, sc["seed"] >> 32)
        go = r0[2] <= 1.0 / torch.special.i0(k * r)
        ang = 2 * math.pi * r0[0]
        x[live[go]] += (r[:, None] * torch.stack([ang.cos(), ang.sin()], 1))[go]
        live = live[go]
    return u, seg, par, x


def _walks64(case, seed):
    """Per walk: u, du/dtheta (walks x parameters); and the scene."""
    sc = _scene(case, seed)
    s = dict(sigma=float(np.float32(sc.sigma)), eps=float(np.float32(sc.eps)), seed=sc.seed)
    f64 = lambda v: torch.as_tensor(np.asarray(v, np.float32).astype(np.float64)).cuda()  # noqa: E731
    jac = f64(sc.jac)
    vert = f64(sc.vert)
    if "theta" in sc.meta:
        vert = f64(sc.reference_vertices()) + torch.einsum("vkp,p->vk", jac, f64(sc.meta["theta"]))
    ev = torch.as_tensor(sc.elem.astype(np.int64)).cuda()
    g = f64(sc.g_vert)
    a, b = vert[ev[:, 0]], vert[ev[:, 1]]
    geo = (a, b, g[ev[:, 0]], g[ev[:, 1]])
    n, W = len(sc.query), case["walks"]
    x0 = f64(sc.query).repeat_interleave(W, 0)
    wid = torch.arange(n * W, device=x0.device)
    u, seg, par, xe = _phase64(s, geo, x0, wid, 0)
    ud = torch.zeros(n * W, jac.shape[2], dtype=torch.float64, device=x0.device)
    hit = (seg >= 0).nonzero()[:, 0]
    i, t = seg[hit], par[hit][:, None]
    e = (b - a)[i]
    bar = a[i] + t * e
    nrm = torch.stack([e[:, 1], -e[:, 0]], 1) / e.norm(dim=1, keepdim=True)
    nrm = torch.where(((bar - xe[hit]) * nrm).sum(1, keepdim=True) < 0, -nrm, nrm)
    h = float(np.float32(sc.h))
    off = bar - h * nrm
    u_off = sum(_phase64(s, geo, off, wid[hit], p)[0] for p in range(1, sc.K + 1)) / sc.K
    c = -((geo[3] - geo[2])[i] / (e * e).sum(1))[:, None] * e - ((u[hit] - u_off) / h)[:, None] * nrm
    for w, v in ((1 - t, ev[i, 0]), (t, ev[i, 1])):
        ud[hit] += w * torch.einsum("mk,mkp->mp", c, jac[v])
        if sc.dg_vert is not None:
            ud[hit] += w * f64(sc.dg_vert)[v]
    return sc, u.reshape(n, W), ud.reshape(n, W, -1)


def _mlp64(case, seed):
    """The first training step of the network: loss and parameters after one Adam step."""
    st = prepare(case, seed)
    p = torch.as_tensor(dwos.init_mlp_params(seed).astype(np.float64)).cuda().requires_grad_(True)
    x, t, m = (st[k].double() for k in ("x", "t", "m"))
    f = torch.cat([x, torch.sin(math.pi * x), torch.sin(math.pi * x.sum(1, keepdim=True)),
                   torch.zeros(len(x), 11, dtype=torch.float64, device=x.device)], 1)
    at = 0
    for o, i in ((64, 16), (64, 64), (64, 64), (64, 64), (8, 64)):
        f = f @ p[at:at + o * i].reshape(o, i).T + p[at + o * i:at + o * i + o]
        f = torch.tanh(f) if o == 64 else f
        at += o * i + o
    loss = (m * (f[:, :2] - t)).square().sum() / len(x)
    loss.backward()
    new = p.detach() - 2e-3 * p.grad / (p.grad.abs() + 1e-8)
    return {"loss": loss.detach().reshape(1), "params": new}


def exact(case, seed):
    kind = case["kind"]
    if kind == "cvtrain":
        return _mlp64(case, seed)
    if kind not in ("opt", "disk") or case["points"] * case["walks"] * case["n_seg"] > 3e7:
        return None                                # walks in 3D, on stars, or too many for brute force
    sc, u, ud = _walks64(case, seed)
    n, W = u.shape
    mean = u.mean(1)
    if kind == "disk":
        sd = lambda v: v.std(1, correction=1) / math.sqrt(W)  # noqa: E731
        return {"u": mean, "u_se": sd(u), "du": ud.mean(1), "du_se": sd(ud)}
    ur = torch.as_tensor(np.asarray(sc.u_ref, np.float32).astype(np.float64)).cuda()
    loss = 0.5 * ((mean - ur) ** 2).sum().reshape(1)
    ub = u.reshape(n, W // sc.B, sc.B)             # U-statistic: u and du/dtheta from different walks
    wt = (ub.sum(2, keepdim=True) - ub) / (sc.B * (sc.B - 1)) - ur[:, None, None] / sc.B
    wt = (wt / (W // sc.B)).reshape(n, W)
    return loss, torch.einsum("pw,pwj->j", wt, ud)
