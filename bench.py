"""Benchmark: differential walk on spheres, reverse-mode gradient of an L2 loss.

One step = one dwos_grad_l2 call on the 2D shape-from-diffusion workload: a
box [-1,1]^2 (g = 0) around a 4096-segment star emitter (g = 1, 64 Fourier
shape parameters), sigma = 10, 256 observation points x 4096 differential
walks, K = 2 nested forward walks per differential walk, U-statistic batches
of B = 8.  Every step draws fresh walks (a new Philox walk-id range).

Printed JSON line (rank 0): walk-steps/s (distance queries of differential and
nested walks per second, whole job), ms per step, gradient estimates/s,
gradient RMSE x seconds, the walk kernel's roofline entry, the oracle's CPU
baseline on a bounded sample, the end-to-end figure through the C ABI with
host buffers, launch count and SM clocks sampled during the timed region.
After the C2 figures, and outside their timed region, the same line carries
the other configurations' headline figures (about a minute and a half in
all; skip with --no-extras): "c3" walk-steps/s of the 200k-triangle 3D
workload, "c4" the 64-problem batch against the same problems as separate
calls, "c5" the learned control variate against the plain estimator
(equal-time final losses over ten seeds, gradient RMSE x seconds per
estimate), "wost" walks on stars on the 2D thermal design and a 3D cube, and
"functional" the volume-integrated shape functional, each with the oracle's
rate on a bounded sample.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]
  python bench.py --workload {c3,c4,c5,ablation,sgd,wost} ...
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "walk-steps/s and dU/dtheta gradient-RMSE x seconds vs plain GPU WoS at 1 GB300"
UNIT = "walk-steps/s"
WORKLOADS = {
    "c2": ("2D shape-from-diffusion: box [-1,1]^2 (g=0) + 4096-segment star emitter (g=1), "
           "sigma=10, 64 Fourier shape params, 256 points x 4096 differential walks, K=2 nested, "
           "L2-loss gradient with U-statistics (B=8)"),
    "c3": ("3D thermal design: 200k-triangle SH-perturbed icosphere (81 SH coefficients, g=1) in box "
           "[-2,2]^3 (g=0), sigma=1, source 0.5, 4096 points x 2048 differential walks, K=2 nested, "
           "gradient of 1/2 sum u^2 with U-statistics (B=8)"),
    "c5": ("learned control variate on the 2D shape-from-diffusion geometry: 200 Adam steps (lr 1e-3) "
           "on 64 Fourier coefficients from a circle toward the star, walks/point annealed 256->1024, MLP "
           "5->64x4->2 (tcgen05 BF16 products, FP32 accumulation in TMEM) trained online on the walks' "
           "estimates (4 Adam iterations on every second step's walks), 10 seeds; value = gradient RMSE x "
           "seconds of one estimate at "
           "1024 walks/point, the network's inference inside the timed region"),
    "ablation": "estimator ablation (product estimators, du/dn estimators, K, h) on the 2D workload",
    "wost": ("walks on stars (Sec. 3.4, 4.2): differential gradient step (U-statistic L2 gradient, K = 2) on the "
             "2D thermal design (32 points on the insulating slab x 16384 walks) and on the 3D cube with four "
             "Neumann faces (64 points x 4096 walks)"),
    "sgd": ("noisy-gradient optimisation (Sec. 5.2) on the 2D workload's geometry: the star's position "
            "(2-vector, Vector Adam, lr 1e-3) from (0.1, -0.06) back to the target's, 256 and 16384 "
            "observation points on |x|_inf = 0.6, 600 iterations, "
            "2 / 16 / 128 walks per point and annealed 2 -> 128 (Eq. update_rule), 3 seeds each"),
    "c4": ("batched: 64 independent problems (32 2D star-in-box, 32 3D SH-sphere-in-box), elements "
           "log-uniform 1e3-5e5, 16-4096 points, sigma log-uniform 0.01-100, 256-4096 walks/point, "
           "16 shape params each; L2-loss gradients in one captured CUDA graph, autotuned walk pool"),
}
WORKLOAD = WORKLOADS["c2"]


def make_scene(name: str, walks: int = 0):
    from paper_2405_12964_gb300 import scenes
    import numpy as np
    if name == "c3":
        sc = scenes.sh_sphere_scene()
        sc.u_ref = np.zeros(sc.query.shape[0])
    else:
        sc = scenes.star_box_scene()
    if walks:
        sc.walks = walks
    return sc


TRAFFIC_SOURCES = ["walk.cu", "dwos_device.cuh", "dwos_internal.h", "bvh.cu"]


def kernel_source_hash() -> str:
    """SHA-256 over the walk kernel's sources (the build's inputs for it)."""
    import hashlib
    h = hashlib.sha256()
    for f in TRAFFIC_SOURCES:
        with open(os.path.join(ROOT, "paper_2405_12964_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()


def measured_traffic(kernel: str, workload: str, tag: str = "traffic", key: str = "dram_bytes"):
    """Bytes per walk-step of `kernel` on `workload` from a committed ncu
    summary (a line '<tag>: kernel=... workload=... <key>=... walk_steps=...
    source_sha256=...' under profiles/; tag 'traffic' for DRAM bytes, 'l2l1'
    for L2 -> L1 bytes), or None if there is none or the kernel's sources
    changed since it was captured."""
    d = os.path.join(ROOT, "profiles")
    if not os.path.isdir(d):
        return None
    want = kernel_source_hash()
    for name in sorted(os.listdir(d)):
        if not name.endswith((".md", ".txt")):
            continue
        with open(os.path.join(d, name)) as fh:
            for line in fh:
                line = line.strip().strip("`")
                if not line.startswith(tag + ":"):
                    continue
                kv = dict(t.split("=", 1) for t in line[len(tag) + 1:].split() if "=" in t)
                if kv.get("kernel") == kernel and kv.get("workload") == workload and kv.get("source_sha256") == want:
                    return float(kv[key]) / float(kv["walk_steps"])
    return None


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            p = json.load(fh)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 200 ms."""
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu: int):
        self.gpu = gpu
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        with open(self.path) as fh:
            for line in fh:
                f = [x.strip() for x in line.split(",")]
                if len(f) < 9:
                    continue
                try:
                    sm.append(float(f[1]))
                    smax.append(float(f[2]))
                except ValueError:
                    continue
                for n, v in zip(names, f[5:9]):
                    if v.lower() == "active":
                        reasons.add(n)
        os.unlink(self.path)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def aggregate_ranks(t_local: float, steps_local: float, dist=None, device=None):
    """Whole-job figures over ranks: the slowest rank's time and the sum of
    walk-steps (weak scaling: every rank runs its own walk-id range)."""
    if dist is None or not dist.is_initialized() or dist.get_world_size() == 1:
        return t_local, steps_local
    import torch
    tt = torch.tensor([t_local], device=device, dtype=torch.float64)
    dist.all_reduce(tt, op=dist.ReduceOp.MAX)
    ss = torch.tensor([float(steps_local)], device=device, dtype=torch.float64)
    dist.all_reduce(ss)
    return float(tt.item()), float(ss.item())


def cpu_baseline(sc, budget_s: float = 15.0):
    """The FP64 oracle (brute-force closest point) on a bounded sample of the
    same workload: a subset of the points (every point if affordable), as many
    differential walks each as fit the time budget on all host cores."""
    import numpy as np
    import oracle
    pr = oracle.Problem(vert=sc.vert, elem=sc.elem, jac=sc.jac, data_kind="mapped", g_vert=sc.g_vert,
                        sigma=sc.sigma, f=sc.f, eps=sc.eps, h=sc.h, K=sc.K, seed=sc.seed)
    n_cal = min(sc.query.shape[0], 2 * oracle.num_threads())
    t0 = time.perf_counter()
    oracle.run_walks(pr, sc.query[:n_cal], 1, differential=True, walk_id_base=1 << 42)
    per_walk = (time.perf_counter() - t0) / n_cal
    total = max(n_cal, int(budget_s / max(per_walk, 1e-9)))
    n_pts = min(sc.query.shape[0], total)
    W = max(1, min(4096, total // n_pts))
    t0 = time.perf_counter()
    o = oracle.run_walks(pr, sc.query[:n_pts], W, differential=True, walk_id_base=1 << 41)
    dt = time.perf_counter() - t0
    if dt < 0.5 * budget_s and W < 4096:   # the calibration overestimated the cost: one larger sample
        W = int(min(4096, max(W + 8, W * budget_s / max(dt, 1e-3))))
        t0 = time.perf_counter()
        o = oracle.run_walks(pr, sc.query[:n_pts], W, differential=True, walk_id_base=1 << 41)
        dt = time.perf_counter() - t0
    steps = int(np.clip(o["steps"], 0, None).sum())
    return {"value": steps / dt, "unit": UNIT, "cores": oracle.num_threads(), "kind": "oracle",
            "sample": f"{n_pts} points x {W} differential walks (K={sc.K}) of the same workload, "
                      f"FP64 brute-force closest point, {dt:.1f} s, {steps} walk-steps"}


def wost_summary(steps: int = 5, warmup: int = 2, oracle_budget_s: float = 3.0):
    """Walks on stars (Sec. 3.4, 4.2) on the GPU and in the oracle: walk-steps/s
    of the differential gradient step (U-statistic L2 gradient, K = 2) on the
    2D thermal scene (32 points on the insulating slab x 16384 walks), on the
    same scene with Neumann data du/dn = 0.5 on the slab (a heat flux through
    its surface) and on the 3D cube with four Neumann faces (64 interior
    points x 4096 walks), inputs resident, L2 flushed between timed steps; and
    the FP64 oracle
    (brute force over every element and silhouette) on a bounded sample of
    the same walks on the host cores."""
    import numpy as np
    import torch
    from paper_2405_12964_gb300 import build, scenes
    build.build()
    if oracle_budget_s > 0:
        import oracle
        oracle.build()
    from paper_2405_12964_gb300.dwos import Solver
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    out = {}
    data = scenes.thermal_scene(n_query=32, walks=16384)
    data.neumann_h = np.where(data.neumann == 1, 0.5, 0.0)
    for name, sc in (("thermal_2d", scenes.thermal_scene(n_query=32, walks=16384)),
                     ("thermal_2d_neumann_data", data),
                     ("cube_3d", scenes.cube_neumann_scene(n_query=64, walks=4096, K=2))):
        s = Solver(0)
        s.load_scene(sc)
        xq = torch.tensor(sc.query, dtype=torch.float32, device="cuda")
        uref = torch.zeros(sc.query.shape[0], dtype=torch.float32, device="cuda")
        total = sc.query.shape[0] * sc.walks
        for i in range(warmup):
            s.grad_l2(xq, uref, sc.walks, walk_id_base=(i + 1) * total)
        torch.cuda.synchronize()
        t, walk_steps, capped = [], 0, 0
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        for i in range(steps):
            flush.fill_(float(i))
            e0.record()
            s.grad_l2(xq, uref, sc.walks, walk_id_base=(warmup + i + 1) * total)
            e1.record()
            st = s.stats()
            t.append(e0.elapsed_time(e1))
            walk_steps += st["steps_main"] + st["steps_nested"]
            capped += st["capped"]
        device_error = None
        try:
            s.sync()   # raises on a walk that left the domain or a search out of budget
        except Exception as ex:
            device_error = str(ex)
        out[name] = {"points": int(sc.query.shape[0]), "walks_per_point": int(sc.walks), "elements": int(len(sc.elem)),
                     "neumann_elements": int(sc.neumann.sum()), "value": walk_steps / (sum(t) / 1e3), "unit": UNIT,
                     "ms_per_step": float(np.mean(t)), "walk_steps_per_step": walk_steps / steps,
                     "capped_walks": int(capped), "device_error": device_error}
        if oracle_budget_s <= 0:
            continue
        pr = oracle.Problem(vert=sc.vert, elem=sc.elem, jac=sc.jac, data_kind="mapped", g_vert=sc.g_vert,
                            sigma=sc.sigma, f=sc.f, eps=sc.eps, h=sc.h, K=sc.K, seed=sc.seed, neumann=sc.neumann,
                            neumann_h=sc.neumann_h)
        n_pts = min(8, sc.query.shape[0])
        t0 = time.perf_counter()
        o = oracle.run_walks(pr, sc.query[:n_pts], 8, differential=True, walk_id_base=1 << 41)
        per = (time.perf_counter() - t0) / (8 * n_pts)
        W = int(max(8, min(4096, oracle_budget_s / max(per, 1e-9) / n_pts)))
        t0 = time.perf_counter()
        o = oracle.run_walks(pr, sc.query[:n_pts], W, differential=True, walk_id_base=1 << 41)
        dt = time.perf_counter() - t0
        o_steps = int(np.clip(o["steps"], 0, None).sum())
        out[name]["oracle"] = {"value": o_steps / dt, "unit": UNIT, "cores": oracle.num_threads(),
                                "sample": f"{n_pts} points x {W} differential walks, {dt:.1f} s"}
    return out


def functional_summary(reps: int = 5, n_try: int = 65536, walks: int = 64, oracle_budget_s: float = 3.0):
    """The volume-integrated functional (Eq. functional, functional_deriv) on
    the 2D shape-from-diffusion geometry: J = int_M 1/2 (u - uref)^2 over the
    box M = [-0.9, 0.9]^2 with uref = 0, n_try uniform candidates in M (those in
    Omega kept), `walks` differential walks per kept point, plus the exact
    boundary term.  Seconds per gradient (synchronised, the host's uref
    evaluation included) and walk-steps/s of its walks; the FP64 oracle's walk
    rate on a bounded sample of the same points on the host cores."""
    import numpy as np
    import torch
    from paper_2405_12964_gb300 import build, scenes
    build.build()
    import oracle
    oracle.build()
    from paper_2405_12964_gb300.dwos import Solver
    sc = scenes.star_box_scene()
    s = Solver(0)
    s.load_scene(sc)
    lo, hi = [-0.9, -0.9], [0.9, 0.9]
    zero = lambda p: np.zeros(len(p))
    s.functional_gradient(lo, hi, zero, walks, n_try, seed=99)
    secs, walk_steps = [], 0
    for r in range(reps):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        s.functional_gradient(lo, hi, zero, walks, n_try, seed=r, walk_id_base=(r + 1) << 34)
        torch.cuda.synchronize()
        secs.append(time.perf_counter() - t0)
        st = s.stats()
        walk_steps += st["steps_main"] + st["steps_nested"]
    pts, _ = s.sample_domain(n_try, lo, hi, 0)
    p = pts.cpu().numpy().astype(np.float64)
    pr = oracle.Problem(vert=sc.vert, elem=sc.elem, jac=sc.jac, data_kind="mapped", g_vert=sc.g_vert,
                        sigma=sc.sigma, f=sc.f, eps=sc.eps, h=sc.h, K=sc.K, seed=sc.seed)
    n_pts = 256
    t0 = time.perf_counter()
    oracle.run_walks(pr, p[:n_pts], 2, differential=True, walk_id_base=1 << 41)
    per = (time.perf_counter() - t0) / (2 * n_pts)
    W = int(max(2, min(walks, oracle_budget_s / max(per, 1e-9) / n_pts)))
    t0 = time.perf_counter()
    o = oracle.run_walks(pr, p[:n_pts], W, differential=True, walk_id_base=1 << 41)
    dt = time.perf_counter() - t0
    o_steps = int(np.clip(o["steps"], 0, None).sum())
    return {"kept_points": int(len(p)), "candidates": n_try, "walks_per_point": walks,
            "seconds_per_gradient": float(np.median(secs)), "value": walk_steps / sum(secs), "unit": UNIT,
            "oracle": {"value": o_steps / dt, "unit": UNIT, "cores": oracle.num_threads(),
                       "sample": f"{n_pts} kept points x {W} differential walks, {dt:.1f} s"}}


def run_reference(args):
    import torch
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    from paper_2405_12964_gb300 import scenes
    import oracle
    oracle.build()
    sc = make_scene(args.workload)
    times, steps_total = [], 0
    for i in range(args.warmup + args.steps):
        cb = cpu_baseline(sc, budget_s=6.0)
        if i >= args.warmup:
            times.append(cb)
    v = statistics.mean(c["value"] for c in times)
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOADS[args.workload], "note": "oracle on host cores, bounded sample per step"},
            "cpu_baseline": {"value": v, "unit": UNIT, "cores": times[0]["cores"], "kind": "oracle",
                             "sample": times[0]["sample"]},
            "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def batched_summary(steps: int, warmup: int):
    """Config 4: the 64 problems as separate dwos_grad_l2 calls (the plain GPU
    path) and as one batched, autotuned, graph-captured pass (walk-steps/s of
    each, the speed-up, the autotuned launch shapes, clocks)."""
    import numpy as np
    import torch
    from paper_2405_12964_gb300 import build, scenes
    build.build()
    from paper_2405_12964_gb300.dwos import Batch, Solver
    probs = scenes.batched_problems(64)
    solvers = []
    for sc in probs:
        s = Solver(0)
        s.load_scene(sc)           # automatic search order: warp-wide for the 3D problems
        solvers.append(s)
    xs = [torch.tensor(sc.query, dtype=torch.float32, device="cuda") for sc in probs]
    us = [torch.tensor(sc.u_ref, dtype=torch.float32, device="cuda") for sc in probs]

    def plain(i):
        for k, (sc, s) in enumerate(zip(probs, solvers)):
            s.grad_l2(xs[k], us[k], sc.walks, walk_id_base=(i + 1) << 32)

    for i in range(warmup):
        plain(i)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t_plain = []
    for i in range(steps):
        e0.record()
        plain(100 + i)
        e1.record()
        torch.cuda.synchronize()
        t_plain.append(e0.elapsed_time(e1))
    b = Batch([(s, xs[k], sc.walks, us[k], 7 << 32) for k, (sc, s) in enumerate(zip(probs, solvers))])
    b.autotune(reps=1)
    b.capture()
    for _ in range(warmup):
        b.launch()
    b.synchronize()
    clocks = ClockSampler(0)
    clocks.start()
    time.sleep(0.3)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    for i in range(steps):
        ev[i][0].record(b.stream)
        b.launch()
        ev[i][1].record(b.stream)
    b.synchronize()
    clk = clocks.stop()
    t_b = [a.elapsed_time(c) for a, c in ev]
    st = b.stats()
    walk_steps = st["steps_main"] + st["steps_nested"]
    return {"workload": WORKLOADS["c4"], "problems": len(probs),
            "walks": int(sum(sc.query.shape[0] * sc.walks for sc in probs)),
            "value": walk_steps / (np.mean(t_b) / 1e3), "unit": UNIT, "ms_per_pass": float(np.mean(t_b)),
            "plain": {"value": walk_steps / (np.mean(t_plain) / 1e3), "ms_per_pass": float(np.mean(t_plain)),
                      "note": "the same 64 problems as separate dwos_grad_l2 calls"},
            "speedup_vs_plain": float(np.mean(t_plain) / np.mean(t_b)), "walk_steps_per_pass": walk_steps,
            "autotuned": {"2d": b.config(2), "3d": b.config(3)}, "steps": steps, "warmup": warmup, "clocks": clk}


def run_batched(args):
    r = batched_summary(args.steps, args.warmup)
    line = {"metric": METRIC, "value": r["value"], "unit": UNIT, "n_gpus": 1, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": r["ms_per_pass"], "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": WORKLOADS["c4"], "problems": r["problems"], "walks": r["walks"],
                       "autotuned": r["autotuned"]},
            "plain": r["plain"], "speedup_vs_plain": r["speedup_vs_plain"],
            "walk_steps_per_step": r["walk_steps_per_pass"], "clocks": r["clocks"]}
    print(json.dumps(line), flush=True)


def control_variate_summary(seeds=tuple(range(3, 13)), steps: int = 200, train_every: int = 2, tail: int = 10):
    """Config 5: the optimisation of the 2D shape-from-diffusion workload with
    and without the learned control variate, per seed: final losses of the CV
    run (the network trained on every train_every-th step's walks), of a plain
    run of the same number of steps and of a plain run given the CV run's wall
    time (training included), each as the loss of the final iterate and as
    the mean loss of the last `tail` iterates (the noisy optimiser's iterate
    wanders about the optimum: the plain equal-time run's final loss moved 2x
    with a change of its step count by 4); and the gradient RMSE x seconds of
    one estimate (network inference timed) at the start shape and midway.
    The plain equal-time run's step count is the CV run's time over the plain
    run's per-step time, rounded up to a multiple of 10."""
    import numpy as np
    import torch
    from paper_2405_12964_gb300 import build, scenes
    build.build()
    from paper_2405_12964_gb300 import optimize
    from paper_2405_12964_gb300.dwos import Solver
    sc = scenes.star_box_scene()
    target = sc.theta0.copy()
    start = np.zeros_like(target)
    # warm-up (module loading and first-use costs of both paths stay out of the timed runs)
    optimize.run(sc, target, start, steps=3, use_cv=False, seed=99)
    optimize.run(sc, target, start, steps=3, use_cv=True, whole_walk=True, seed=99)
    s = Solver(0)
    s.load_scene(sc)
    s.set_boundary(sc.reference_vertices(), sc.elem, sc.jac)
    s.set_dirichlet_mapped(sc.g_vert)
    s.set_params(target)
    xq = torch.tensor(sc.query, dtype=torch.float32, device="cuda")
    s_uref = s.eval(xq, 16384)["u"].cpu().numpy()

    def true_loss(theta):          # the loss of a final shape, from 16384 walks per point
        s.set_params(theta)
        u = s.eval(xq, 16384)["u"].cpu().numpy()
        s.set_params(target)
        return float(0.5 * np.sum((u - s_uref) ** 2))

    clocks = ClockSampler(0)
    clocks.start()
    runs, trainer = [], None
    for seed in seeds:
        th_p, hp, _ = optimize.run(sc, target, start, steps=steps, use_cv=False, seed=seed)
        th_c, hc, trainer = optimize.run(sc, target, start, steps=steps, use_cv=True, whole_walk=True, seed=seed,
                                         train_every=train_every)
        # equal wall time: the plain optimiser gets the seconds the CV run took (training included),
        # rounded up to a multiple of 10 steps (at least equal time; the walks-per-point schedule
        # anneals over the run, so the step count fixes the trajectory, and rounding keeps it the
        # same from one measurement to the next)
        steps_eq = max(steps, 10 * int(np.ceil(steps * hc.seconds[-1] / max(hp.seconds[-1], 1e-9) / 10)))
        th_e, he, _ = optimize.run(sc, target, start, steps=steps_eq, use_cv=False, seed=seed)
        lc, lp, le = true_loss(th_c), true_loss(th_p), true_loss(th_e)
        tail_loss = lambda h: float(np.mean([true_loss(t) for t in h.thetas[-tail:]]))
        mc, mp, me = tail_loss(hc), tail_loss(hp), tail_loss(he)
        runs.append({"seed": seed, "cv": {"final_loss": lc, "tail_mean_loss": mc, "seconds": hc.seconds[-1],
                                          "median_var_ratio_last20": float(np.median(hc.var_ratio[-20:]))},
                     "plain": {"final_loss": lp, "tail_mean_loss": mp, "seconds": hp.seconds[-1]},
                     "plain_equal_time": {"final_loss": le, "tail_mean_loss": me, "seconds": he.seconds[-1],
                                          "steps": steps_eq},
                     "ratio_cv_over_plain_equal_time": mc / me,
                     "ratio_cv_over_plain_equal_time_final_iterate": lc / le})
    clk = clocks.stop()
    ratios = np.array([r["ratio_cv_over_plain_equal_time"] for r in runs])
    ratios_f = np.array([r["ratio_cv_over_plain_equal_time_final_iterate"] for r in runs])
    mid = 0.5 * (start + target)
    rows = {}
    for name, th in [("start", start), ("midway", mid)]:
        plain = optimize.gradient_rmse_x_time(sc, th, s_uref, 1024)
        cv = optimize.gradient_rmse_x_time(sc, th, s_uref, 1024, net=trainer.net, whole_walk=True)
        rows[name] = {"plain": plain, "cv": cv, "rmse_x_seconds_ratio": cv["rmse_x_seconds"] / plain["rmse_x_seconds"]}
    return {"workload": WORKLOADS["c5"], "steps": steps, "train_every": train_every, "runs": runs,
            "equal_time_final_loss_ratio": {"geometric_mean": float(np.exp(np.mean(np.log(ratios)))),
                                            "min": float(ratios.min()), "max": float(ratios.max()),
                                            "seeds": list(seeds), "loss": f"mean over the last {tail} iterates"},
            "equal_time_final_iterate_loss_ratio": {"geometric_mean": float(np.exp(np.mean(np.log(ratios_f)))),
                                                    "min": float(ratios_f.min()), "max": float(ratios_f.max())},
            "final_loss_note": "1/2 sum (u - u_target)^2 of a shape, u from 16384 walks per point",
            "gradient_rmse_x_seconds": rows, "clocks": clk}


def run_wost(args):
    """--workload wost: the walk-on-stars summary alone (the oracle leg unless --no-cpu)."""
    r = wost_summary(steps=args.steps, warmup=args.warmup, oracle_budget_s=0.0 if args.no_cpu else 3.0)
    line = {"metric": METRIC, "value": r["thermal_2d"]["value"], "unit": UNIT, "n_gpus": 1, "steps": args.steps,
            "warmup": args.warmup, "higher_is_better": True, "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": WORKLOADS["wost"], "l2": "flushed between timed steps (256 MB write)"}}
    line.update(r)
    print(json.dumps(line), flush=True)


def run_control_variate(args):
    r = control_variate_summary()
    line = {"metric": METRIC, "value": r["gradient_rmse_x_seconds"]["start"]["cv"]["rmse_x_seconds"],
            "unit": "gradient RMSE x s", "higher_is_better": False, "n_gpus": 1, "steps": r["steps"], "warmup": 0,
            "vs_baseline": None, "dtype": "f32 walks, bf16 MLP", "data": "synthetic",
            "config": {"workload": WORKLOADS["c5"]}}
    line.update({k: v for k, v in r.items() if k != "workload"})
    print(json.dumps(line), flush=True)


def thermal_summary(steps: int, warmup: int):
    """Config 3 at its stated size: walk-steps/s of the U-statistic gradient of
    1/2 sum u^2 over 4096 points x 2048 differential walks on the 200k-triangle
    SH sphere (inputs resident, L2 flushed between timed steps)."""
    import numpy as np
    import torch
    from paper_2405_12964_gb300 import build
    build.build()
    from paper_2405_12964_gb300.dwos import Solver
    sc = make_scene("c3")
    s = Solver(0)
    s.load_scene(sc, traversal=3)
    xq = torch.tensor(sc.query, dtype=torch.float32, device="cuda")
    uref = torch.tensor(sc.u_ref, dtype=torch.float32, device="cuda")
    total = sc.query.shape[0] * sc.walks
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    for i in range(warmup):
        s.grad_l2(xq, uref, sc.walks, walk_id_base=(i + 1) * total)
    torch.cuda.synchronize()
    clocks = ClockSampler(0)
    clocks.start()
    time.sleep(0.3)
    t, walk_steps, kms = [], 0, []
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for i in range(steps):
        flush.fill_(float(i))
        e0.record()
        s.grad_l2(xq, uref, sc.walks, walk_id_base=(warmup + i + 1) * total)
        e1.record()
        st = s.stats()
        t.append(e0.elapsed_time(e1))
        walk_steps += st["steps_main"] + st["steps_nested"]
        kms.append(st["kernel_ms"])
    clk = clocks.stop()
    return {"workload": WORKLOADS["c3"], "value": walk_steps / (sum(t) / 1e3), "unit": UNIT,
            "ms_per_step": float(np.mean(t)), "walk_kernel_ms": float(np.mean(kms)),
            "walk_steps_per_step": walk_steps / steps, "elements": int(len(sc.elem)), "steps": steps,
            "warmup": warmup, "clocks": clk}


def run_ablation(args):
    """Estimator ablation on the 2D shape-from-diffusion workload at the star
    (Sec. 5.3, Fig. ablation): gradient RMSE against a 64x-walk reference,
    bias (the mean of the repeats against it) and seconds per estimate for
    the product estimators (U-statistic, correlated, uncorrelated), the two
    du/dn estimators (backward difference, ball gradient), K and h."""
    import numpy as np
    import torch
    from paper_2405_12964_gb300 import build, scenes
    build.build()
    from paper_2405_12964_gb300.dwos import Solver
    sc = scenes.star_box_scene()
    W, R = 1024, 16
    xq = torch.tensor(sc.query, dtype=torch.float32, device="cuda")
    uref = torch.tensor(sc.u_ref, dtype=torch.float32, device="cuda")
    s = Solver(0)
    s.load_scene(sc)
    ref = np.mean([s.grad_l2(xq, uref, 16384, walk_id_base=(3 << 44) + r * (1 << 30))[1].cpu().numpy()
                   for r in range(4)], axis=0)
    variants = [("ustat, backward difference, K=2, h=10 eps", dict(), "ustat"),
                ("ustat, backward difference, K=1", dict(K=1), "ustat"),
                ("ustat, backward difference, K=4", dict(K=4), "ustat"),
                ("ustat, backward difference, h=5 eps", dict(h=5 * sc.eps), "ustat"),
                ("ustat, backward difference, h=20 eps", dict(h=20 * sc.eps), "ustat"),
                ("ustat, ball gradient, K=2", dict(dudn_estimator=1), "ustat"),
                ("correlated product", dict(), "correlated"),
                ("uncorrelated product", dict(), "uncorrelated")]
    rows = []
    for name, opt, product in variants:
        s.load_scene(sc, **opt)
        s.grad_l2_product(xq, uref, W, product=product, walk_id_base=1 << 46)   # warm-up
        est, times = [], []
        for r in range(R):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            g = s.grad_l2_product(xq, uref, W, product=product, walk_id_base=(5 << 44) + r * (1 << 30))[1]
            g = g.cpu().numpy()
            times.append(time.perf_counter() - t0)
            est.append(g)
        E = np.array(est)
        rmse = float(np.sqrt(np.mean((E - ref[None]) ** 2)))
        bias = float(np.sqrt(np.mean((E.mean(0) - ref) ** 2)))
        sec = float(np.median(times))
        rows.append({"variant": name, "rmse": rmse, "bias_of_mean": bias,
                     "bias_se": float(np.sqrt(np.mean(E.var(0, ddof=1) / R))),
                     "seconds": sec, "rmse_x_seconds": rmse * sec})
    line = {"metric": METRIC, "value": rows[0]["rmse_x_seconds"], "unit": "gradient RMSE x s",
            "higher_is_better": False, "n_gpus": 1, "steps": R, "warmup": 1, "vs_baseline": None,
            "dtype": "f32", "data": "synthetic",
            "config": {"workload": "estimator ablation on the 2D shape-from-diffusion workload: 256 points x "
                                   "1024 walks per estimate, 16 repeats per variant, reference = U-statistic "
                                   "backward-difference gradient at 65536 walks per point"},
            "ablation": rows}
    print(json.dumps(line), flush=True)


def run_sgd(args):
    """Sec. 5.2's experiment: position error and loss against iterations and
    against wall time for fixed and annealed walks per point."""
    import numpy as np
    from paper_2405_12964_gb300 import build
    build.build()
    from paper_2405_12964_gb300 import optimize
    t0 = time.perf_counter()
    studies = {}
    # 256 points: even 128 walks per point leave most of the GPU idle; 16384 points:
    # 128 walks per point are 2 M walks, and the walk count sets the iteration's cost
    for n_query, tw, ew in ((256, 16384, 4096), (16384, 2048, 512)):
        res = optimize.noisy_gradient_study(n_query=n_query, target_walks=tw, eval_walks=ew)
        table = optimize.study_table(res)
        curves = {}
        for name, runs in res.items():    # seed-mean curves, every 10th iteration
            err = np.mean([r["err"] for r in runs], axis=0)
            sec = np.mean([r["seconds"] for r in runs], axis=0)
            curves[name] = {"iter": list(range(10, len(err) + 1, 10)), "err": [float(e) for e in err[9::10]],
                            "seconds": [float(x) for x in sec[9::10]],
                            "loss_iter": runs[0]["loss_iter"],
                            "loss": [float(v) for v in np.mean([r["loss"] for r in runs], axis=0)]}
        studies["%d points" % n_query] = {"target_walks": tw, "eval_walks": ew, "table": table, "curves": curves}
    big = studies["16384 points"]["table"]
    ann = [k for k in big if k.startswith("annealed")][0]
    last_t = list(big[ann]["err_at_time"])[-1]
    line = {"metric": "position error at equal wall time (Sec. 5.2)", "value": big[ann]["err_at_time"][last_t],
            "unit": "|theta - theta*|", "higher_is_better": False, "n_gpus": 1, "steps": 600, "warmup": 0,
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": WORKLOADS["sgd"], "equal_time_reference": "fractions of the fastest run's time",
                       "value": "annealed run, 16384 points, at the fastest run's end"},
            "studies": studies, "seconds": time.perf_counter() - t0}
    print(json.dumps(line), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="dwos")
    ap.add_argument("--walks", type=int, default=0, help="walks per point (0: the workload's)")
    ap.add_argument("--workload", default="c2", choices=sorted(WORKLOADS))
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-extras", action="store_true",
                    help="skip the C3 / C4 / C5 summaries that the default line carries after the C2 figures")
    ap.add_argument("--traversal", type=int, default=-1,
                    help="closest-point search: 0 binary per lane, 1 climb, 2 wide tree warp-wide, 3 routed "
                         "(only queries that reach inside the binary root's child boxes are searched, warp-wide; "
                         "-1: 3)")
    args = ap.parse_args()
    if args.impl == "reference":
        return run_reference(args)
    if args.workload == "c4":
        return run_batched(args)
    if args.workload == "c5":
        return run_control_variate(args)
    if args.workload == "ablation":
        return run_ablation(args)
    if args.workload == "sgd":
        return run_sgd(args)
    if args.workload == "wost":
        return run_wost(args)

    import numpy as np
    import torch

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)

    from paper_2405_12964_gb300 import build
    build.build()
    from paper_2405_12964_gb300.dwos import Solver, lib, MEM_HOST
    import ctypes

    sc = make_scene(args.workload, args.walks)
    s = Solver(local)
    trav = args.traversal if args.traversal >= 0 else 3
    s.load_scene(sc, traversal=trav)
    n_pts, W = sc.query.shape[0], sc.walks
    total = n_pts * W
    xq = torch.tensor(sc.query, dtype=torch.float32, device=dev)
    uref = torch.tensor(sc.u_ref, dtype=torch.float32, device=dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)   # > L2 (129 MB)

    # reference gradient for the RMSE figure: 16x the walks, its own walk ids
    ref_grads = []
    for r in range(4):
        _, g = s.grad_l2(xq, uref, 4 * W, walk_id_base=(1 << 44) + r * 4 * total)
        ref_grads.append(g.cpu().numpy())
    g_ref = np.mean(ref_grads, axis=0)

    stream = torch.cuda.current_stream(dev)
    launches0 = s.stats()["launches"]

    def step(i):
        return s.grad_l2(xq, uref, W, walk_id_base=(rank * 100000 + i + 1) * total)

    for i in range(args.warmup):
        step(i)
    torch.cuda.synchronize()
    launches_warm = s.stats()["launches"]

    clocks = ClockSampler(local)
    clocks.start()
    time.sleep(0.3)
    if dist:
        dist.barrier()
    torch.cuda.synchronize()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    # the timed steps are enqueued back to back (no host synchronisation inside the
    # region), each bracketed by its own events, with the L2 flush between them
    grads_dev = []
    for i in range(args.steps):
        flush.fill_(float(i))                      # evict L2 between timed steps (outside the events)
        ev[i][0].record(stream)
        loss, g = step(args.warmup + i)
        ev[i][1].record(stream)
        grads_dev.append(g)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    clk = clocks.stop()
    launches = s.stats()["launches"] - launches_warm
    step_ms = [a.elapsed_time(b) for a, b in ev]
    t_local = sum(step_ms) / 1e3
    grads = [g.cpu().numpy() for g in grads_dev]
    # walk-step counts, search counters and the walk kernel's own launch time: the
    # same steps replayed one at a time (same walk ids, hence the same walks)
    steps_done = nodes = wnodes = prims = 0
    kernel_ms = []
    for i in range(args.steps):
        flush.fill_(float(i))
        step(args.warmup + i)
        st = s.stats()                             # synchronises
        steps_done += st["steps_main"] + st["steps_nested"]
        nodes += st["nodes_visited"]
        wnodes += st["wide_nodes_visited"]
        prims += st["prims_tested"]
        kernel_ms.append(st["kernel_ms"])
    t, steps_all = aggregate_ranks(t_local, steps_done, dist, dev)
    value = steps_all / t
    ms_per_step = 1e3 * t / args.steps

    # gradient quality: RMSE of one step's gradient against the 16x-walk reference
    G = np.array(grads)
    rmse = float(np.sqrt(np.mean((G - g_ref[None]) ** 2)))
    rel = rmse / float(np.sqrt(np.mean(g_ref ** 2)))

    # roofline of the walk kernel: algorithmic bytes = binary node fetches x 48 / 64 B
    # + wide-node visits in units of 32 child slots x 640 B (2D: a float4 and a code per
    # slot, leaf segments included) / 2048 B (3D: four nodes of 8 oriented boxes)
    # + element fetches outside the nodes (the previous step's element, outsized
    # elements; all element tests of the binary search) x 16 / 48 B
    # + one 32 B record per walk + 8 B query load per walk
    node_b = 48 if sc.dim == 2 else 64
    wide_b = 640 if sc.dim == 2 else 2048
    prim_b = 16 if sc.dim == 2 else 48
    alg_bytes = nodes * node_b + wnodes * wide_b + prims * prim_b + args.steps * total * (32 + 8)
    walk_s = sum(kernel_ms) / 1e3
    achieved = alg_bytes / walk_s / 1e9 / args.steps * args.steps
    hbm, src = peaks()
    from paper_2405_12964_gb300.dwos import probe_l2_read
    l2 = probe_l2_read(local)
    kname = f"walk_kernel<{sc.dim},{'true' if trav in (2, 3) else 'false'}>"
    traffic_per_step = measured_traffic(kname, args.workload)
    l2l1_per_step = measured_traffic(kname, args.workload, tag="l2l1", key="bytes")

    e2e = None
    if rank == 0:
        # end to end through the C ABI with pinned host buffers: copies in the timed region
        xh = torch.tensor(sc.query, dtype=torch.float32).pin_memory()
        uh = torch.tensor(sc.u_ref, dtype=torch.float32).pin_memory()
        gh = torch.empty(sc.n_param, dtype=torch.float64).pin_memory()
        lh = torch.empty(1, dtype=torch.float64).pin_memory()
        L = lib()
        s._stream()
        e2e_t, e2e_steps = [], 0
        for i in range(args.warmup + max(3, args.steps // 2)):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            stt = L.dwos_grad_l2(s._h, n_pts, ctypes.c_void_p(xh.data_ptr()), ctypes.c_void_p(uh.data_ptr()), W,
                                 (1 << 45) + i * total, ctypes.c_void_p(lh.data_ptr()),
                                 ctypes.c_void_p(gh.data_ptr()), None, MEM_HOST)
            t1 = time.perf_counter()
            if stt:
                raise RuntimeError(L.dwos_last_error(s._h).decode())
            if i >= args.warmup:
                e2e_t.append(t1 - t0)
                st = s.stats()
                e2e_steps += st["steps_main"] + st["steps_nested"]
        e2e = {"value": e2e_steps / sum(e2e_t), "unit": UNIT,
               "h2d_bytes_per_step": int(xh.numel() * 4 + uh.numel() * 4),
               "d2h_bytes_per_step": int(gh.numel() * 8 + lh.numel() * 8)}

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu:
        cpu = cpu_baseline(sc)

    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": WORKLOADS[args.workload], "points": n_pts, "walks_per_point": W, "K": sc.K, "B": sc.B,
                       "n_param": sc.n_param, "eps": sc.eps, "h": sc.h,
                       "closest_point_search": {0: "binary LBVH, per lane", 1: "binary LBVH climbing from the hint",
                                                2: "wide BVH (2D 32, 3D 8 children), warp-wide",
                                                3: "routed: binary-root test per query, then the wide BVH "
                                                   "warp-wide for the queries that need the tree"}[trav],
                       "l2": "flushed between timed steps (256 MB write outside the events)",
                       "timing": ("timed steps enqueued back to back, each between its own CUDA events; "
                                  "walk-step counts and the walk kernel's launch time from a replay of the "
                                  "same walk ids"),
                       "parallelism": f"replicas x{world} (independent walk ranges, no collective)"},
            "gradient_estimates_per_s": world * total * args.steps / t,
            "grad_rmse": rmse, "grad_rel_rmse": rel, "grad_rmse_x_seconds": rmse * (ms_per_step / 1e3),
            "walk_steps_per_step": steps_done / args.steps,
            "closest_point_search": {"nodes_per_query": nodes / max(steps_done, 1),
                                     "wide_nodes_per_query": wnodes / max(steps_done, 1),
                                     "element_fetches_per_query": prims / max(steps_done, 1)},
            "roofline": {"bound": "latency", "achieved": achieved, "peak": hbm, "unit": "GB/s",
                         "frac": achieved / hbm,
                         "bound_note": ("ncu: dependent-instruction and L1/L2 latency (fixed-latency and "
                                        "long-scoreboard stalls, about a third of the warp slots active); the "
                                        "tree bytes come from L1/L2, DRAM sees under 0.01 % of them, so the frac "
                                        "against the HBM copy peak is a bandwidth-equivalent figure, not a "
                                        "binding roof"),
                         "traffic": (None if traffic_per_step is None
                                     else traffic_per_step * steps_done / args.steps),
                         "traffic_source": ("ncu dram__bytes_read.sum + dram__bytes_write.sum of one launch, "
                                            "scaled to this launch's walk-steps" if traffic_per_step is not None
                                            else "no ncu capture of the current kernel sources"),
                         "kernel": kname, "peak_source": src,
                         "bytes_per_walk_step": alg_bytes / max(steps_done, 1),
                         "l2_to_l1_bytes_per_walk_step": l2l1_per_step,
                         "l2_to_l1_source": ("ncu lts__t_sectors_srcunit_tex_op_read.sum x 32 B of one launch "
                                             "(full section set on 1024 walks per point)"
                                             if l2l1_per_step is not None
                                             else "no ncu capture of the current kernel sources"),
                         "walk_kernel_ms": walk_s * 1e3 / args.steps,
                         "l2": {"peak": l2, "unit": "GB/s", "frac": achieved / l2,
                                "peak_source": "measured in this run: 32 MB L2-resident buffer read 50 times "
                                               "(dwos_probe_l2_read)"}},
            "cpu_baseline": cpu, "e2e": e2e,
            "gpu_launches": int(launches),
            "clocks": clk,
        }
        if world == 1 and not args.no_extras and args.workload == "c2":
            # the other configurations' headline figures, measured after the C2 timed region
            t_x = time.perf_counter()
            line["c3"] = thermal_summary(steps=5, warmup=2)
            line["c4"] = batched_summary(steps=3, warmup=2)
            line["c5"] = control_variate_summary()
            line["wost"] = wost_summary()
            line["functional"] = functional_summary()
            line["extras_seconds"] = time.perf_counter() - t_x
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
