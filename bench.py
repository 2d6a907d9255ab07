"""Benchmark: Diffusing Winding Gradients orientation on one GB300.

Workload (default): union-15m, the largest single-GPU configuration: 15,000,000
samples of the boundary of a union of 20 random tori and 20 random
ellipsoids, Gaussian noise 0.25 % of the bounding-box diagonal, a_i = 1,
screened kernel lambda = 100 (Eq. 5), octree depth 10, k = 10, Barnes-Hut far
field with the opening angle, leaf size and test form picked by the library's
autotuner (2.5 % w budget), random initial normals (seed 1), stopping when
the mean normal change of Fig. 6 is at most the chord of 0.1 deg or after 40
iterations.  Beside it (untimed): the learned warm start and the paper's PCA
and Gauss-map starts to the same rule, and the time to equal accuracy.

One step = one full orientation (dwg_orient): every iteration evaluates w and
grad w at all N points and w at all Q octree-leaf corners, extracts the
w_bar level set, scatters face gradients to the 10 nearest points, updates
the normals and tests convergence, all inside one CUDA graph launch.

Metric: GWN+grad interactions per second (kernel evaluations performed,
counted on the device), whole job over all ranks; also seconds to converged
normals.  Multi-GPU: batch-64 shards its independent clouds over the ranks;
the single-cloud workloads run independent replicas (weak scaling): the
method's per-cloud loop has an exchange step only when one cloud is split,
which this benchmark does not do.

Other workloads (--workload): torus-100k (100,000 noisy torus points, exact
all-pairs, plain or --kernel 1 screened), metaballs-1m (Barnes-Hut path),
batch-64 (64 clouds in one handle).

--impl reference times the FP64 CPU oracle on a bounded sample of the same
workload on the host cores.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import synth  # noqa: E402

# FP32 operations per interaction in the minimal formulation of each kernel
# (sub x3, fma x3 for rho^2, mul+fma x2 for <m,d>, then the kernel's own):
#   w only, plain 12 | w and grad, plain 20 | w only, screened 16 | w and grad, screened 27
# (screened: F / rho^3 = e inv^2 (inv + s)); each interaction also takes one
# MUFU rsqrt and, screened, one MUFU ex2
# The exact path's leaf corners lie on a lattice: eight corners share the terms'
# x and y parts, 66 / 8 and 98 / 8 operations an interaction.
FP32_OPS = {("w", 0): 12, ("wg", 0): 20, ("w", 1): 16, ("wg", 1): 27,
            ("lattice", 0): 8.25, ("lattice", 1): 12.25}
FP32_LANES_PER_SM = 128


def alu_peaks(what, kind, sm_count, fmax_hz, ffma=None, rsq=None, ex2=None):
    """Interactions per second of an evaluator.  what: "w", "wg" or "lattice" (w
    at the leaf corners on the exact path); kind: 0 plain, 1 screened.  derived: SMs x 128 FP32 lanes x clock / FP32
    operations per interaction.  With the microbenchmarks' rates (packed-FMA
    lane operations, MUFU rsqrt and ex2 per second): the FMA-pipe bound, the
    MUFU bound (one rsqrt, and for the screened kernel one ex2, per
    interaction) and the lower of the two."""
    ops = FP32_OPS[(what, kind)]
    out = {"ops": ops, "derived": sm_count * FP32_LANES_PER_SM * fmax_hz / ops}
    if ffma is not None:
        mufu = 1.0 / (1.0 / rsq + (1.0 / ex2 if kind else 0.0))
        out.update(fma_bound=ffma / ops, mufu_bound=mufu, measured=min(ffma / ops, mufu))
    return out


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--kernel", type=int, default=0, help="0 plain, 1 screened (lambda 10)")
    ap.add_argument("--depth", type=int, default=None)
    ap.add_argument("--workload", default="union-15m",
                    choices=["torus-100k", "metaballs-1m", "union-15m", "batch-64"])
    ap.add_argument("--no-tune", action="store_true", help="keep the default evaluator shapes")
    ap.add_argument("--tuning", default=None,
                    help="apply these settings instead of tuning, e.g. "
                         "'corners_pairs=2,corners_threads=128' (profiler captures)")
    ap.add_argument("--no-warm", action="store_true",
                    help="skip the comparison of initial normals (random, learned, PCA, Gauss map)")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true", help="skip the CPU oracle baseline")
    ap.add_argument("--one-step", action="store_true",
                    help="run one iteration of the workload and exit (for profiler captures)")
    ap.add_argument("--init", default="random", choices=["random", "learned", "pca", "gauss"],
                    help="initial normals of --one-step (learned: the warm-start network runs)")
    ap.add_argument("--reg", default="soften", choices=["soften", "clamp"],
                    help="near-field regularisation of --one-step (clamp: the modified kernel of "
                         "Sec. 5.2 with the paper's radii)")
    return ap.parse_args()


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def workload(args):
    """The named workload with its method parameters.  The torus follows the
    benchmark's plain-kernel configuration; the Barnes-Hut workloads use the
    paper's recommended screening (lambda in [10, 100], Sec. 5.1) and octree
    depth, and the convergence measure of Fig. 6 (DWG_CONV_MEAN), since their
    outliers and noise keep the top-1 % statistic above 0.1 degrees."""
    if args.workload == "metaballs-1m":
        W = synth.workload_metaballs1m()
        W.update(path=2, depth=9, kernel=1, lam=100.0, rule=1, max_iters=80)
    elif args.workload == "union-15m":
        W = synth.workload_union15m()
        W.update(path=2, depth=10, kernel=1, lam=100.0, rule=1, max_iters=40)
    else:
        W = synth.workload_torus100k()
        W.update(path=1, theta=0.5, kernel=args.kernel, lam=10.0 if args.kernel == 1 else 0.0,
                 rule=1, max_iters=60)
    if args.depth:
        W["depth"] = args.depth
    return W


def profiled_bytes_per_interaction(which):
    """DRAM bytes per interaction of the list evaluator from the committed
    ncu summary (None when absent)."""
    key = f"dram_bytes_per_interaction_{which}:"
    try:
        for line in open(os.path.join(ROOT, "profiles", "tree_lists_metaballs1m.md")):
            if line.startswith(key):
                return float(line.split(":")[1])
    except OSError:
        return None
    return None


def profiled_lattice_bytes(corners):
    """DRAM bytes of one corner launch of the exact path from the committed ncu
    summary (None when absent or of another cloud)."""
    got = {}
    try:
        for line in open(os.path.join(ROOT, "profiles", "gwn_lattice_torus100k.md")):
            for key in ("corners:", "dram_bytes_per_launch:"):
                if line.startswith(key):
                    got[key] = int(line.split(":")[1])
    except OSError:
        return None
    return got.get("dram_bytes_per_launch:") if got.get("corners:") == corners else None


def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f)
    except Exception:
        return {}


class Clocks:
    """nvidia-smi sampling during the timed region."""

    def __init__(self, gpu_index):
        self.proc = None
        out_dir = os.environ.get("DWG_BENCH_CLOCKS_DIR", tempfile.gettempdir())
        self.path = os.path.join(out_dir, f"clocks_bench_{os.getpid()}.csv")
        q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(gpu_index), f"--query-gpu={q}", "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if not self.proc:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.f.close()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def flush_l2(torch, buf):
    buf.add_(1.0)  # writes 256 MiB, larger than the 129 MB L2


def agreement(out, nt, labels=None):
    """Share of points whose normal agrees in sign with the analytic one,
    after aligning the global sign (points without an analytic normal, the
    outliers, are left out).  With labels (the primitive of each sample of a
    union of shapes), the sign is aligned per label: each connected part of
    the surface is oriented on its own."""
    m = np.linalg.norm(nt, axis=1) > 0
    d = np.sum(np.asarray(out, np.float64)[m] * nt[m], axis=1)
    if labels is None:
        s = 1.0 if d.sum() >= 0 else -1.0
        return float(np.mean(s * d > 0))
    lab = np.asarray(labels)[m]
    sums = np.bincount(lab, weights=d)
    s = np.where(sums >= 0, 1.0, -1.0)[lab]
    return float(np.mean(s * d > 0))


def configure(dwg, h, W, weights):
    dwg.dwg_set_weights(h, weights)
    dwg.dwg_set_params(h, W["kernel"], W["eps"], W["lam"], W["max_iters"], W["tol"])
    dwg.dwg_set_update(h, W["depth"], 10, dwg.DWG_UPDATE_LEVELSET)
    dwg.dwg_set_tree(h, W["path"], W.get("theta", 0.5))
    dwg.dwg_set_convergence(h, W["rule"])


def tune(dwg, h, W, args):
    """The library's autotuner: evaluator shapes on the exact path; leaf size,
    test form and opening angle on the Barnes-Hut path, with an error budget
    of 2.5 % of the winding number's inside value (a first-order far field
    at theta 0.5 is at 2-3.5 %, and orients the metaballs to 100 %),
    measured with the analytic normals (the regime of a converged
    orientation)."""
    if args.tuning:
        kv = dict(item.split("=") for item in args.tuning.split(","))
        dwg.dwg_set_tuning(h, **{k: (float(v) if k == "theta" else int(v)) for k, v in kv.items()})
        return dwg.dwg_get_tuning(h)
    if args.no_tune:
        return dwg.dwg_get_tuning(h)
    if W["path"] == dwg.DWG_PATH_ALLPAIRS:
        return dwg.dwg_autotune(h, dwg.DWG_TUNE_SHAPES, 1e-3, None)
    n = len(W["points"])
    nt = np.asarray(W["normals_true"], np.float32).copy()
    bad = ~(np.linalg.norm(nt, axis=1) > 0)   # outliers: no analytic normal
    nt[bad] = synth.random_unit_normals(int(bad.sum()), seed=3).astype(np.float32)
    dwg.dwg_set_normals(h, nt)
    sel = (synth.uniform(4, 5, 2048) * n).astype(np.int64)
    q = np.ascontiguousarray(W["points"][sel])
    w = np.zeros(len(q), np.float32)
    dwg.dwg_eval_gwn(h, q, w)
    scale = 2.0 * float(np.median(np.abs(w)))   # w at the surface is half the inside value
    t = dwg.dwg_autotune(h, dwg.DWG_TUNE_TREE, 0.025 * scale, None)
    t["w_budget"] = 0.025 * scale
    return t


def _agreement_fn(torch, dev, W):
    """Agreement with the analytic normals computed on the device (same
    definition as agreement())."""
    nt = np.nan_to_num(np.asarray(W["normals_true"], np.float32))
    ntd = torch.from_numpy(nt).to(dev)
    lab = W.get("labels")
    if lab is None:
        labd, K = torch.zeros(len(nt), dtype=torch.int64, device=dev), 1
    else:
        labd, K = torch.from_numpy(np.asarray(lab, np.int64)).to(dev), int(np.max(lab)) + 1
    valid = (ntd.abs().sum(1) > 0)
    nv = float(valid.sum())

    def fn(out):
        d = (out * ntd).sum(1).double()
        sums = torch.bincount(labd, weights=d, minlength=K)
        sgn = torch.where(sums >= 0, 1.0, -1.0).double()[labd]
        return float((((sgn * d) > 0) & valid).double().sum()) / nv
    return fn


def warm_start_compare(dwg, torch, dev, W, tuning, weights, max_iters):
    """Seconds to converged normals from each initialisation: random, the
    learned warm start, and the paper's PCA and Gauss-map options (Sec. 5.1),
    all to the same rule (the Fig. 6 mean change <= the chord of 0.1 deg,
    checked after every iteration as dwg_orient does) and cap.  Each run is
    one iteration per dwg_step call, timed with the device synchronised on
    both sides, with the agreement with the analytic normals recorded after
    every iteration; the learned start's time includes its kNN features and
    network.  At equal accuracy: the target is the lower of the random and
    learned final agreements, and each side's time is its time to the first
    iteration at or above it."""
    from paper_2405_13839_gb300 import train_init
    params = np.load(train_init.DEFAULT_WEIGHTS).astype(np.float32)
    agree = _agreement_fn(torch, dev, W)
    chord = 2 * math.sin(math.radians(W["tol"]) / 2)
    n = len(W["points"])
    modes = {"random": dwg.DWG_INIT_RANDOM, "pca": dwg.DWG_INIT_PCA, "gauss": dwg.DWG_INIT_GAUSS,
             "learned": dwg.DWG_INIT_LEARNED}
    out = {}
    pts = torch.from_numpy(W["points"]).to(dev)
    for init in ("random", "learned", "pca", "gauss"):
        h = dwg.dwg_create(pts)
        try:
            configure(dwg, h, W, weights)
            dwg.dwg_set_params(h, W["kernel"], W["eps"], W["lam"], max_iters, W["tol"])
            dwg.dwg_set_convergence(h, dwg.DWG_CONV_MEAN)
            dwg.dwg_set_tuning(h, **{k: tuning[k] for k in TUNING_KEYS})
            res = torch.empty((n, 3), dtype=torch.float32, device=dev)
            dwg.dwg_step(h)   # builds the buffers, lists and kNN candidates once
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            dwg.dwg_set_init(h, modes[init], 1, params if init == "learned" else None)
            torch.cuda.synchronize()
            t_init = time.perf_counter() - t0
            dwg.dwg_get_normals(h, res)
            prev = res.clone()
            trace = [(0, t_init, agree(res))]
            t_sum, it, conv, stat = t_init, 0, False, float("nan")
            while it < max_iters:
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                _, stat = dwg.dwg_step(h)
                torch.cuda.synchronize()
                t_sum += time.perf_counter() - t0
                it += 1
                dwg.dwg_get_normals(h, res)
                trace.append((it, t_sum, agree(res)))
                mean_dn = float((res - prev).double().norm(dim=1).mean())
                prev.copy_(res)
                if mean_dn <= chord:
                    conv = True
                    break
            out[init] = {"s": t_sum, "init_s": t_init, "iterations": it, "converged": conv,
                         "agreement": trace[-1][2], "agreement_at_start": trace[0][2],
                         "top1_stat_deg_last": stat,
                         "trace": [(i, round(t, 4), round(a, 5)) for i, t, a in trace]}
        finally:
            dwg.dwg_destroy(h)
    out["rule"] = ("mean |n_new - n_old| <= chord of 0.1 deg (Fig. 6 measure), every init, "
                   f"cap {max_iters} iterations")
    for k in ("learned", "pca", "gauss"):
        out["speedup" if k == "learned" else f"speedup_{k}"] = out["random"]["s"] / out[k]["s"]
    target = min(out["learned"]["agreement"], out["random"]["agreement"])

    def first_at(tr):
        for i, t, a in tr:
            if a >= target:
                return i, t
        return tr[-1][0], tr[-1][1]
    ir, sr = first_at(out["random"]["trace"])
    il, sl = first_at(out["learned"]["trace"])
    out["equal_accuracy"] = {"agreement": target, "random_iterations": ir, "random_s": sr,
                             "learned_iterations": il, "learned_s": sl, "speedup": sr / sl}
    for k in ("random", "learned", "pca", "gauss"):   # keep the line short
        tr = out[k].pop("trace")
        out[k]["agreement_every_10"] = [a for i, t, a in tr if i % 10 == 0]
    return out


def setup_and_variants(dwg, torch, dev, W, reps=3):
    """Device time of the one-time per-cloud steps the paper adds around the
    iteration (Sec. 5.1 area weights and initialisations, Sec. 5.2 clamp
    radii) on this workload, and the w + grad w throughput at the points of
    the modified kernel (Sec. 5.2) beside the softened one, both all-pairs."""
    n = len(W["points"])
    pts = torch.from_numpy(W["points"]).to(dev)
    out = {}
    h = dwg.dwg_create(pts)
    try:
        nrm = torch.empty((n, 3), dtype=torch.float32, device=dev)

        def timed(fn):
            ts = []
            for _ in range(reps):
                torch.cuda.synchronize()
                t0 = time.perf_counter()
                fn()
                torch.cuda.synchronize()
                ts.append(1e3 * (time.perf_counter() - t0))
            return round(statistics.median(ts), 3)

        out["voronoi_weights_ms"] = timed(lambda: dwg.dwg_voronoi_weights(h, 15))
        from paper_2405_13839_gb300 import train_init
        params = np.load(train_init.DEFAULT_WEIGHTS).astype(np.float32)
        for name, mode in (("random", dwg.DWG_INIT_RANDOM), ("pca", dwg.DWG_INIT_PCA),
                           ("gauss", dwg.DWG_INIT_GAUSS), ("learned", dwg.DWG_INIT_LEARNED)):
            def init(mode=mode):
                dwg.dwg_set_init(h, mode, 1, params if mode == dwg.DWG_INIT_LEARNED else None)
                dwg.dwg_get_normals(h, nrm)
            # learned: kNN-16 features and the tcgen05 network included
            out[f"init_{name}_ms"] = timed(init)
        out["clamp_radii_ms"] = timed(lambda: dwg.dwg_set_regularization(
            h, dwg.DWG_REG_CLAMP, 10, 0.0, 0.0))
        dwg.dwg_set_regularization(h, dwg.DWG_REG_SOFTEN)
        # the level set of the analytic normals as triangles, into device memory
        dwg.dwg_set_weights(h, torch.from_numpy(W["weights"]).to(dev))
        dwg.dwg_set_params(h, W["kernel"], W["eps"], W["lam"], 30, 0.1)
        dwg.dwg_set_update(h, W["depth"], 10, dwg.DWG_UPDATE_LEVELSET)
        nt_ok = np.nan_to_num(W["normals_true"]).astype(np.float32)
        nt_ok[np.linalg.norm(nt_ok, axis=1) == 0] = [0.0, 0.0, 1.0]
        dwg.dwg_set_init(h, dwg.DWG_INIT_GIVEN, 0, nt_ok)
        ntri, _ = dwg.dwg_extract_level_set(h)
        tri = torch.empty((max(ntri, 1), 9), dtype=torch.float32, device=dev)
        out["level_set_triangles"] = int(ntri)
        out["level_set_extract_ms"] = timed(lambda: dwg.dwg_extract_level_set(h, tri))
        if n <= 200_000:
            dwg.dwg_set_weights(h, torch.from_numpy(W["weights"]).to(dev))
            dwg.dwg_set_params(h, W["kernel"], W["eps"], W["lam"], 30, 0.1)
            dwg.dwg_set_tree(h, dwg.DWG_PATH_ALLPAIRS, 0.5)
            w = torch.empty(n, dtype=torch.float32, device=dev)
            g = torch.empty((n, 3), dtype=torch.float32, device=dev)
            for reg in (dwg.DWG_REG_SOFTEN, dwg.DWG_REG_CLAMP):
                dwg.dwg_set_regularization(h, reg, 10, 0.0, 0.0)
                dwg.dwg_eval_gwn(h, pts, w, g)  # warm-up
                ms = timed(lambda: dwg.dwg_eval_gwn(h, pts, w, g))
                key = "softened" if reg == dwg.DWG_REG_SOFTEN else "modified_kernel"
                out[f"eval_points_{key}"] = {"ms": ms, "interactions_per_s": n * n / (ms / 1e3)}
            out["eval_points_basis"] = ("dwg_eval_gwn at the n points, w and grad w, all-pairs, "
                                        "call wall time incl. the reduce (median of 3)")
        else:
            # the Barnes-Hut path: one whole iteration (group lists, MC, kNN) each way
            dwg.dwg_set_weights(h, torch.from_numpy(W["weights"]).to(dev))
            dwg.dwg_set_params(h, W["kernel"], W["eps"], W["lam"], 30, 0.1)
            dwg.dwg_set_update(h, W["depth"], 10, dwg.DWG_UPDATE_LEVELSET)
            dwg.dwg_set_tree(h, dwg.DWG_PATH_TREE, 0.5)
            for reg in (dwg.DWG_REG_SOFTEN, dwg.DWG_REG_CLAMP):
                dwg.dwg_set_regularization(h, reg, 10, 0.0, 0.0)
                dwg.dwg_set_init(h, dwg.DWG_INIT_RANDOM, 1)
                dwg.dwg_step(h)  # builds the lists for this kernel
                ms = timed(lambda: dwg.dwg_step(h))
                key = "softened" if reg == dwg.DWG_REG_SOFTEN else "modified_kernel"
                out[f"tree_step_{key}_ms"] = ms
            out["tree_step_basis"] = ("dwg_step on the Barnes-Hut path (theta 0.5, leaf 16, group "
                                      "lists), one iteration, median of 3")
    finally:
        dwg.dwg_destroy(h)
    out["basis"] = "median of 3 calls, host wall time around synchronous C-ABI calls"
    return out


TUNING_KEYS = ("path", "points_pairs", "points_threads", "corners_pairs", "corners_threads",
               "tree_leaf", "theta", "tree_group")


def run_ours(args, rank, world, local):
    import torch
    from paper_2405_13839_gb300 import dwg

    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    W = workload(args)
    p_host = W["points"]
    n = len(p_host)
    stream = torch.cuda.current_stream(dev)
    p_dev = torch.from_numpy(p_host).to(dev)
    a_dev = torch.from_numpy(W["weights"]).to(dev)
    h = dwg.dwg_create(p_dev)
    dwg.dwg_set_stream(h, stream.cuda_stream)
    configure(dwg, h, W, a_dev)
    tuning = tune(dwg, h, W, args)
    dwg.dwg_set_init(h, dwg.DWG_INIT_RANDOM, 1)
    out = torch.empty((n, 3), dtype=torch.float32, device=dev)
    flush = torch.zeros(64 * 1024 * 1024, dtype=torch.float32, device=dev)

    for _ in range(args.warmup):
        dwg.dwg_orient(h, out)
    torch.cuda.synchronize()

    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
          for _ in range(args.steps)]
    clocks = Clocks(local)
    if world > 1:
        import torch.distributed as dist
        dist.barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    inter = 0.0
    it_list, rc_list = [], []
    for k in range(args.steps):
        flush_l2(torch, flush)
        ev[k][0].record(stream)
        rc, it = dwg.dwg_orient(h, out)
        ev[k][1].record(stream)
        s = dwg.dwg_get_stats(h)
        inter += s["interactions"]
        it_list.append(it)
        rc_list.append(rc)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()  # the timed region is bracketed by barriers on both sides
    wall = time.perf_counter() - t0
    ck = clocks.stop()
    ms = [a.elapsed_time(b) for a, b in ev]
    dev_s = sum(ms) / 1e3
    st_orient = dwg.dwg_get_stats(h)
    agree = agreement(out.cpu().numpy(), W["normals_true"], W.get("labels"))
    if world > 1:
        import torch.distributed as dist
        t = torch.tensor([dev_s, inter], dtype=torch.float64, device=dev)  # NCCL: device tensors
        tt = t.clone()
        dist.all_reduce(tt, op=dist.ReduceOp.SUM)
        tmax = t.clone()
        dist.all_reduce(tmax, op=dist.ReduceOp.MAX)
        dev_s = float(tmax[0])
        inter = float(tt[1])
    value = inter / dev_s

    # per-kernel device times of one iteration (same kernels and launch shapes)
    dwg.dwg_set_init(h, dwg.DWG_INIT_RANDOM, 1)
    prof = []
    for _ in range(3):
        prof.append(dwg.dwg_profile_step(h))
    kms = {k: statistics.median(p[k] for p in prof) for k in prof[0]}
    st = dwg.dwg_get_stats(h)
    nc = st["n_corners"]
    peaks = measured_peaks()
    sm_count = torch.cuda.get_device_properties(dev).multi_processor_count
    fmax = (peaks.get("sm_max_mhz") or 2070.0) * 1e6
    lanes = sm_count * FP32_LANES_PER_SM * fmax
    kind = W["kernel"]
    iter_ms = sum(kms.values())
    if W["path"] == dwg.DWG_PATH_ALLPAIRS:
        # dominant kernel: w at the leaf corners
        dom = "eval_corners" if kms.get("eval_corners", 0) >= kms["eval_points"] else "eval_points"
        if dom == "eval_corners":
            work = float(nc) * n
            what = "lattice"
        else:
            work = float(n) * n
            what = "wg"
        achieved = work / (kms[dom] / 1e3)
        # DRAM bytes of the launch as captured by ncu (the torus cloud's corners)
        traffic = profiled_lattice_bytes(nc) if dom == "eval_corners" else None
        traffic_basis = ("ncu dram bytes of k_gwn_lattice (profiles/gwn_lattice_torus100k.md)"
                         if traffic is not None else "not captured for this launch")
    else:
        # Barnes-Hut: the dominant of the two tree launches (w and grad at the
        # points, w at the corners), its evaluations performed (counted on the
        # device during the profiled step) per second of its launch
        if kms.get("eval_corners", 0) >= kms["eval_points"]:
            dom, work, what = "eval_corners", st["interactions_corners_step"], "w"
        else:
            dom, work, what = "eval_points", st["interactions_points_step"], "wg"
        dom += " (Barnes-Hut lists)"
        achieved = work / (kms[dom.split()[0]] / 1e3)
        # DRAM bytes of the same list kernel captured by ncu on metaballs-1m,
        # per interaction, times this launch's interactions (the lists, item
        # partials and record misses grow with the records per group)
        bpi = profiled_bytes_per_interaction(
            "corners" if dom.startswith("eval_corners") else "points")
        traffic = bpi * work if (bpi is not None and tuning.get("tree_group")) else None
        traffic_basis = ("ncu dram bytes of k_tree_eval_lists on metaballs-1m per interaction "
                         "(profiles/tree_lists_metaballs1m.md) x this launch's interactions")
    pk = alu_peaks(what, kind, sm_count, fmax)
    ops, peak = pk["ops"], pk["derived"]
    roof = {"bound": "alu", "kernel": dom, "achieved": achieved / 1e9, "peak": peak / 1e9,
            "unit": "Ginteractions/s", "frac": achieved / peak, "traffic": traffic,
            "traffic_basis": traffic_basis,
            "peak_basis": f"{sm_count} SMs x {FP32_LANES_PER_SM} FP32 lanes x {fmax/1e6:.0f} MHz"
                          f" / {ops} FP32 ops per interaction (the MUFU bound, from the measured "
                          f"rsqrt and ex2 rates, is in fp32_measured)",
            "kernel_ms": {k: round(v, 4) for k, v in kms.items()},
            "share": {k: round(v / iter_ms, 4) for k, v in kms.items()}}
    # the same denominator measured: packed-FMA, MUFU rsqrt and ex2 microbenchmarks
    try:
        ffma, rsq, ex2 = dwg.dwg_measure_fp32_peaks(local)
        pm = alu_peaks(what, kind, sm_count, fmax, ffma, rsq, ex2)
        roof["fp32_measured"] = {
            "ffma_lane_ops_per_s": ffma, "rsqrt_per_s": rsq, "ex2_per_s": ex2,
            "derived_lane_ops_per_s": lanes, "ffma_over_derived": ffma / lanes,
            "mufu_bound_interactions_per_s": pm["mufu_bound"],
            "peak_from_measured": pm["measured"] / 1e9,
            "frac_of_measured": achieved / pm["measured"]}
    except Exception as e:  # reported beside the derived peak, never instead of it
        roof["fp32_measured"] = {"error": str(e)}

    # the library's w and grad w at the oracle leg's sampled points, with the
    # oracle leg's normals (its precision is reported beside the oracle's time)
    gpu_sample = None
    if world == 1 and not args.no_cpu:
        n0 = sample_normals(W).astype(np.float32)
        dwg.dwg_set_normals(h, torch.from_numpy(n0).to(dev))
        qs = torch.from_numpy(np.ascontiguousarray(p_host[sample_points(W)])).to(dev)
        ws = torch.empty(len(qs), dtype=torch.float32, device=dev)
        gs = torch.empty((len(qs), 3), dtype=torch.float32, device=dev)
        dwg.dwg_eval_gwn(h, qs, ws, gs)
        gpu_sample = (ws.cpu().numpy(), gs.cpu().numpy())

    # end to end through the C ABI with host buffers
    e2e = None
    if not args.no_e2e:
        ph = torch.from_numpy(p_host).pin_memory()
        ah = torch.from_numpy(W["weights"]).pin_memory()
        oh = torch.empty((n, 3), dtype=torch.float32).pin_memory()
        e2e_t = []
        e2e_inter = 0.0
        reps = 1 if n > 5_000_000 else max(1, min(args.steps, 3))
        for k in range(reps):
            torch.cuda.synchronize()
            t1 = time.perf_counter()
            h2 = dwg.dwg_create(ph)
            configure(dwg, h2, W, ah)
            dwg.dwg_set_tuning(h2, **{k: tuning[k] for k in TUNING_KEYS})
            dwg.dwg_set_init(h2, dwg.DWG_INIT_RANDOM, 1)
            dwg.dwg_orient(h2, oh)
            e2e_inter += dwg.dwg_get_stats(h2)["interactions"]
            dwg.dwg_destroy(h2)
            e2e_t.append(time.perf_counter() - t1)
        e2e = {"value": e2e_inter / sum(e2e_t), "unit": "interactions/s",
               "s_per_orient": statistics.median(e2e_t),
               "h2d_bytes_per_step": int(ph.numel() * 4 + ah.numel() * 4),
               "d2h_bytes_per_step": int(oh.numel() * 4 + 4)}
    dwg.dwg_destroy(h)
    warm = None
    if not args.no_warm and world == 1:
        cap = W["max_iters"] if n > 5_000_000 else max(100, W["max_iters"])
        warm = warm_start_compare(dwg, torch, dev, W, tuning, a_dev, cap)
    extras = None
    if not args.no_warm and world == 1:
        extras = setup_and_variants(dwg, torch, dev, W)
    # reset, random init, pack, then the graph's kernels once per iteration
    launches_per_step = 3 + st_orient["kernels_per_iteration"] * statistics.mean(it_list)
    return dict(value=value, dev_s=dev_s, ms=ms, iters=it_list, rcs=rc_list, st=st_orient,
                roof=roof, clocks=ck, e2e=e2e, wall=wall, agree=agree, tuning=tuning, warm=warm,
                extras=extras, launches=int(round(launches_per_step * args.steps)), W=W, nc=nc,
                gpu_sample=gpu_sample)


SAMPLE = 4096   # sampled points (and corners) of the oracle leg, at most


def sample_points(W):
    """Indices of the points the oracle leg evaluates (seeded)."""
    return (synth.uniform(5, 1, SAMPLE) * len(W["points"])).astype(np.int64)


def oracle_setup(W):
    """The oracle's octree-leaf corners of the workload and the sampled
    corners, computed once (FP64 oracle)."""
    import oracle
    oracle.build()
    p = W["points"]
    L = oracle.octree_leaves(p, W["depth"])
    K = oracle.corner_keys(L, W["depth"])
    C = oracle.corner_positions(K, W["depth"], oracle.cube(p, W["depth"]))
    rng_cor = (synth.uniform(5, 2, SAMPLE) * len(C)).astype(np.int64)
    # the sources in the oracle's FP64 layout once, so that the timed calls
    # measure the sums and not the conversion of the arrays
    return {"corners": C[rng_cor], "n_corners": int(len(C)),
            "p64": np.ascontiguousarray(p, dtype=np.float64),
            "a64": np.ascontiguousarray(W["weights"], dtype=np.float64),
            "n64": np.ascontiguousarray(sample_normals(W), dtype=np.float64)}


def sample_normals(W):
    """Normals of the oracle leg: the analytic ones (the regime of an
    oriented cloud, where w is about 1 inside), random unit normals (seed 1)
    where a point has none (outliers)."""
    nt = np.array(W["normals_true"], dtype=np.float64)
    bad = ~np.all(np.isfinite(nt), axis=1) | ~(np.linalg.norm(nt, axis=1) > 0)
    if bad.any():
        nt[bad] = synth.random_unit_normals(len(nt), seed=1)[bad]
    return nt


def cpu_baseline(W, setup, budget_s=12.0, single_thread=True, gpu_sample=None):
    """The oracle timed on a bounded sample: w and grad w at sampled points and
    w at sampled octree corners, against all N sources (FP64, all host cores),
    sized to about budget_s seconds.  With gpu_sample (the library's w and
    grad w at the same sampled points, same normals), also the library's
    error against these FP64 values."""
    import oracle
    p, a, n0 = setup["p64"], setup["a64"], setup["n64"]
    n = len(p)
    rng_pts = sample_points(W)
    Cs = setup["corners"]
    kern, lam, eps = W["kernel"], W["lam"], W["eps"]
    # probe, then size the sample to about budget_s seconds
    t = time.perf_counter()
    oracle.gwn(p, n0, a, p[rng_pts[:16]], kernel=kern, eps=eps, lam=lam)
    probe = time.perf_counter() - t
    m = int(max(16, min(SAMPLE, 16 * budget_s / 2 / max(probe, 1e-6))))
    t = time.perf_counter()
    wo, go = oracle.gwn(p, n0, a, p[rng_pts[:m]], kernel=kern, eps=eps, lam=lam)
    tg = time.perf_counter() - t
    t = time.perf_counter()
    oracle.gwn(p, n0, a, Cs[:m], kernel=kern, eps=eps, lam=lam, grad=False)
    tw = time.perf_counter() - t
    per_q_g = tg / m
    per_q_w = tw / m
    rate = (2 * m * n) / (tg + tw)
    cores = oracle.set_threads(0)
    rate1, m1 = None, 0
    if single_thread:  # one thread on a sample an eighth of the size
        m1 = max(4, m // 8)
        oracle.set_threads(1)
        try:
            t = time.perf_counter()
            oracle.gwn(p, n0, a, p[rng_pts[:m1]], kernel=kern, eps=eps, lam=lam)
            oracle.gwn(p, n0, a, Cs[:m1], kernel=kern, eps=eps, lam=lam, grad=False)
            rate1 = (2 * m1 * n) / (time.perf_counter() - t)
        finally:
            oracle.set_threads(cores)
    # extrapolated time of one iteration of the full workload
    it_s = n * per_q_g + setup["n_corners"] * per_q_w
    out = {"value": rate, "unit": "interactions/s", "cores": cores, "kind": "oracle",
           "sample": f"w+grad at {m} sampled points and w at {m} sampled octree corners, "
                     f"each against all {n} sources (FP64, OpenMP); per-iteration time "
                     f"extrapolated to all points and corners",
           "single_thread": ({"value": rate1, "sample": f"{m1} points and {m1} corners"}
                             if single_thread else None),
           "extrapolated_s_per_iteration": it_s, "corners": setup["n_corners"]}
    if gpu_sample is not None:
        wg, gg = gpu_sample
        dw = np.abs(wg[:m].astype(np.float64) - wo)
        dg = np.linalg.norm(gg[:m].astype(np.float64) - go, axis=1)
        gn = np.linalg.norm(go, axis=1)
        scale = float(np.median(np.abs(wo)))

        def st(x):
            return {"max": float(x.max()), "p99": float(np.percentile(x, 99)),
                    "median": float(np.median(x))}
        out["precision"] = {
            "what": f"library (the bench's path and settings) vs FP64 at the {m} sampled "
                    "points, analytic normals (random where a point has none)",
            "w_abs": st(dw), "w_rel_to_median_abs_w": st(dw / max(scale, 1e-300)),
            "grad_abs": st(dg), "grad_rel": st(dg / np.maximum(gn, 1e-300))}
    return out


def one_step(args):
    """One iteration of the workload: the launch shapes of a bench step (the
    tuner's settings, the defaults with --no-tune, or --tuning's)."""
    import torch
    from paper_2405_13839_gb300 import dwg
    W = workload(args)
    h = dwg.dwg_create(W["points"])
    configure(dwg, h, W, W["weights"])
    tune(dwg, h, W, args)
    if args.reg == "clamp":
        dwg.dwg_set_regularization(h, dwg.DWG_REG_CLAMP, 10, 0.0, 0.0)
    if args.init == "learned":
        from paper_2405_13839_gb300 import train_init
        params = np.load(train_init.DEFAULT_WEIGHTS).astype(np.float32)
        dwg.dwg_set_init(h, dwg.DWG_INIT_LEARNED, 1, params)
    else:
        dwg.dwg_set_init(h, {"random": dwg.DWG_INIT_RANDOM, "pca": dwg.DWG_INIT_PCA,
                             "gauss": dwg.DWG_INIT_GAUSS}[args.init], 1)
    iso, stat = dwg.dwg_step(h)
    torch.cuda.synchronize()
    t = dwg.dwg_get_tuning(h)
    dwg.dwg_destroy(h)
    print(json.dumps({"one_step": W["name"], "iso": iso, "stat": stat, "tuning": t}))


def run_batch(args, rank=0, world=1, local=0):
    """64 clouds in one handle: one CUDA graph launch orients all of them.
    With several ranks the clouds are independent problems: each rank
    orients its share (balanced by estimated work) in its own batch handle,
    with no exchange on the data path; the job time is the slowest rank's."""
    import torch
    from paper_2405_13839_gb300 import dwg, shard
    W = synth.workload_batch64()
    P_all, off_all = W["points"], W["offsets"]
    mine = shard.assign(W["sizes"], world)[rank]
    P, off = shard.sub_batch(P_all, off_all, mine)
    nt_all = W["normals_true"]
    nt = np.vstack([nt_all[off_all[c]:off_all[c + 1]] for c in mine])
    nc = len(off) - 1
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    hb = dwg.dwg_create_batch(torch.from_numpy(P).to(dev), off)
    dwg.dwg_set_params(hb, 1, 0.0, 10.0, 80, 0.1)   # eps 0: each cloud's default softening
    dwg.dwg_set_convergence(hb, dwg.DWG_CONV_MEAN)
    # every cloud tuned on its own: path, leaf size, test form and opening
    # angle within 2.5 % of its winding-number scale
    t0 = time.perf_counter()
    tuned = None
    if not args.no_tune:
        tuned = dwg.dwg_autotune(hb, dwg.DWG_TUNE_SHAPES | dwg.DWG_TUNE_TREE | dwg.DWG_TUNE_RELATIVE,
                                 0.025, None)
    tune_s = time.perf_counter() - t0
    out = torch.empty_like(torch.from_numpy(P), device=dev)
    for _ in range(args.warmup):
        dwg.dwg_set_init(hb, dwg.DWG_INIT_RANDOM, 1)
        dwg.dwg_orient_batch(hb, out, nc)
    clocks = Clocks(local)
    ms, inter, iters = [], 0.0, None
    if world > 1:
        import torch.distributed as dist
        dist.barrier()
    for _ in range(args.steps):
        dwg.dwg_set_init(hb, dwg.DWG_INIT_RANDOM, 1)
        torch.cuda.synchronize()
        rc, iters = dwg.dwg_orient_batch(hb, out, nc)
        st = dwg.dwg_get_stats(hb)
        ms.append(st["ms_orient"])
        inter += st["interactions"]
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    ck = clocks.stop()
    o = out.cpu().numpy()
    ags = [agreement(o[off[c]:off[c + 1]], nt[off[c]:off[c + 1]]) for c in range(nc)]
    # the same orientation in the other batch modes (untimed by the line; the
    # same results): batched phases on 4 and 8 lanes, and each cloud's chain
    # as a graph branch
    modes = {"phases_1_lane": (dwg.dwg_get_stats(hb)["kernels_per_iteration"], sum(ms) / 1e3 / args.steps)}
    for name, lanes in (("phases_4_lanes", 4), ("phases_8_lanes", 8), ("branches", 0)):
        dwg.dwg_set_batch_mode(hb, lanes)
        dwg.dwg_set_init(hb, dwg.DWG_INIT_RANDOM, 1)
        dwg.dwg_orient_batch(hb, out, nc)   # captures the mode's graph
        dwg.dwg_set_init(hb, dwg.DWG_INIT_RANDOM, 1)
        dwg.dwg_orient_batch(hb, out, nc)
        st = dwg.dwg_get_stats(hb)
        modes[name] = (st["kernels_per_iteration"], st["ms_orient"] / 1e3)
    dwg.dwg_set_batch_mode(hb, 1)
    # the other initialisations on every cloud (one run each): the learned
    # warm start and the paper's PCA and Gauss-map options
    from paper_2405_13839_gb300 import train_init
    params = np.load(train_init.DEFAULT_WEIGHTS).astype(np.float32)
    inits = {}
    for name, mode in (("learned", dwg.DWG_INIT_LEARNED), ("pca", dwg.DWG_INIT_PCA),
                       ("gauss", dwg.DWG_INIT_GAUSS)):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        dwg.dwg_set_init(hb, mode, 1, params if name == "learned" else None)
        _, its_i = dwg.dwg_orient_batch(hb, out, nc)
        torch.cuda.synchronize()
        s_i = time.perf_counter() - t0
        o = out.cpu().numpy()
        inits[name] = (s_i, list(its_i),
                       [agreement(o[off[c]:off[c + 1]], nt[off[c]:off[c + 1]]) for c in range(nc)])
    dwg.dwg_destroy(hb)
    dev_s = sum(ms) / 1e3
    its = list(iters)
    if world > 1:
        import torch.distributed as dist
        t = torch.tensor([dev_s, inter] + [inits[k][0] for k in inits], dtype=torch.float64,
                         device=dev)
        tmax = t.clone()
        dist.all_reduce(tmax, op=dist.ReduceOp.MAX)
        tsum = t.clone()
        dist.all_reduce(tsum, op=dist.ReduceOp.SUM)
        dev_s, inter = float(tmax[0]), float(tsum[1])
        gathered = [None] * world
        dist.all_gather_object(gathered, (ags, its, {k: v[1:] for k, v in inits.items()}))
        ags = [a for g in gathered for a in g[0]]
        its = [i for g in gathered for i in g[1]]
        inits = {k: (float(tmax[2 + j]), [i for g in gathered for i in g[2][k][0]],
                     [a for g in gathered for a in g[2][k][1]])
                 for j, k in enumerate(inits)}
        if rank != 0:
            return
    iters = its
    nc = len(ags)
    warm = {k: {"s": s_i, "iterations_mean": float(np.mean(it_i)), "iterations_max": int(max(it_i)),
                "agreement_mean": float(np.mean(ag_i)), "agreement_min": min(ag_i),
                "clouds_at_least_99pct": int(sum(a >= 0.99 for a in ag_i))}
            for k, (s_i, it_i, ag_i) in inits.items()}
    line = {"metric": "GWN+grad interactions/s", "value": inter / dev_s, "unit": "interactions/s",
            "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * dev_s / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": "batch-64", "clouds": nc, "points": int(off_all[-1]),
                       "parallelism": f"clouds sharded over {world} rank(s), no data-path exchange",
                       "kernel": "screened lambda=10", "eps": "per cloud 0.5 L / sqrt(n)",
                       "rule": "mean change <= chord of 0.1 deg", "max_iters": 80,
                       "tuning": ("per cloud, relative w budget 2.5 % (largest cloud: " +
                                  json.dumps({k: tuned[k] for k in TUNING_KEYS}) + ")")
                                 if tuned else "defaults",
                       "tuning_s": round(tune_s, 1)},
            "s_to_converged_normals": dev_s / args.steps,
            "iterations": {"min": int(min(iters)), "max": int(max(iters)),
                           "mean": float(np.mean(iters))},
            "agreement": {"min": min(ags), "mean": float(np.mean(ags)),
                          "clouds_at_least_99pct": int(sum(a >= 0.99 for a in ags))},
            "warm_start": warm,
            "batch_modes": {k: {"s": s_m, "kernels_per_iteration": k_m}
                            for k, (k_m, s_m) in modes.items()},
            "clocks": ck}
    print(json.dumps(line))


def common_config(W, world):
    """The workload's configuration, shared by both arms' JSON lines."""
    return {"workload": W["name"], "points": len(W["points"]),
            "kernel": "plain" if W["kernel"] == 0 else f"screened lambda={W['lam']:g}",
            "depth": W["depth"], "knn": 10, "tol_deg": W["tol"],
            "rule": "top-1% mean change (Sec. 5.1)" if W["rule"] == 0 else
                    "mean change (Fig. 6 measure)",
            "max_iters": W["max_iters"], "init": "random seed 1",
            "parallelism": f"replicas x{world}",
            "l2": "flushed (256 MiB write) before every step"}


def main():
    args = parse()
    rank, world, local = dist_env()
    if args.one_step:
        one_step(args)
        return
    if world > 1:
        import torch
        import torch.distributed as dist
        backend = "nccl" if args.impl == "ours" else "gloo"
        if backend == "nccl":
            torch.cuda.set_device(local)
        dist.init_process_group(backend=backend)
    if args.impl == "reference":
        if rank != 0:
            return
        W = workload(args)
        n = len(W["points"])
        setup = oracle_setup(W)
        for _ in range(args.warmup):
            cpu_baseline(W, setup, budget_s=1.0, single_thread=False)
        vals = []
        t0 = time.perf_counter()
        last = None
        for _ in range(args.steps):
            last = cpu_baseline(W, setup, budget_s=8.0, single_thread=False)
            vals.append(last["value"])
        wall = time.perf_counter() - t0
        v = statistics.median(vals)
        line = {"impl": "reference", "metric": "GWN+grad interactions/s", "value": v,
                "unit": "interactions/s", "n_gpus": args.gpus, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": 1e3 * wall / args.steps,
                "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
                "data": "synthetic",
                "config": common_config(W, args.gpus) | {"path": "FP64 all-pairs (oracle)"},
                "cpu_baseline": {k: last[k] for k in ("kind", "cores", "sample")} | {"value": v, "unit": "interactions/s"},
                "e2e": {"value": v, "unit": "interactions/s", "h2d_bytes_per_step": 0,
                        "d2h_bytes_per_step": 0}}
        print(json.dumps(line))
        return

    if args.workload == "batch-64":
        run_batch(args, rank, world, local)
        return
    r = run_ours(args, rank, world, local)
    if rank != 0:
        return
    W = r["W"]
    n = len(W["points"])
    cpu = None
    if world == 1 and not args.no_cpu:
        try:
            cpu = cpu_baseline(W, oracle_setup(W), gpu_sample=r["gpu_sample"])
        except Exception as e:  # the oracle is a reported baseline only
            cpu = {"error": str(e)}
    ms_per_step = 1e3 * r["dev_s"] / args.steps
    t = r["tuning"]
    path = ("all-pairs exact, compensated FP32" if t["path"] == 1 else
            f"Barnes-Hut theta {t['theta']:.2f}, leaf {t['tree_leaf']}, "
            f"{'group' if t['tree_group'] else 'per-query'} opening test")
    line = {
        "metric": "GWN+grad interactions/s", "value": r["value"], "unit": "interactions/s",
        "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": common_config(W, world) | {
            "corners": r["nc"], "path": path, "tuning": {k: t[k] for k in TUNING_KEYS}},
        "s_to_converged_normals": ms_per_step / 1e3,
        "iterations": r["iters"][0],
        "converged": r["rcs"][0] == 0,
        "top1_stat_deg_last": r["st"]["stat_last"],
        "agreement_with_analytic_normals": r["agree"],
        "agreement_basis": ("sign aligned per primitive of the union (each connected part is "
                            "oriented on its own)" if W.get("labels") is not None else
                            "one global sign"),
        "warm_start": r["warm"],
        "setup_and_variants": r["extras"],
        "interactions_per_step": r["value"] * r["dev_s"] / args.steps / world,
        "roofline": r["roof"], "cpu_baseline": cpu, "clocks": r["clocks"], "e2e": r["e2e"],
        "gpu_launches": r["launches"],
    }
    if isinstance(cpu, dict) and "precision" in cpu:
        line["precision"] = cpu.pop("precision")   # measured in the oracle leg
    print(json.dumps(line))


if __name__ == "__main__":
    main()
