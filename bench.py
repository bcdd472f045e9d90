#!/usr/bin/env python
"""Benchmark: LM bundle-adjustment iterations per second on one synthetic
scene of 4,000 cameras, 1.2M points and ~8.04M observations (the ba4000
workload: views per point 2+Geom0(1/5.7), 1 px noise), block-Jacobi PCG
capped at 50 iterations, and the time to reach (1 + 1e-6) F_ref, F_ref the
converged FP64 cost.  The headline is the FP64 path (the paper's
arithmetic); the FP32 variant (FP32 per-observation arithmetic, FP64
reductions and cost) is reported in the same line.

A step is one LM trial: linearisation (when theta changed), block assembly,
Schur reduction, PCG on the reduced camera system, back-substitution, trial
cost and accept/reject -- all through the library's C ABI.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                    [--precision both|f64|f32] [--mode partition|replicas]

Prints one JSON line (rank 0).  Under torchrun (N > 1) the ranks by default
solve ONE problem partitioned by points (every camera on every rank, NCCL
all-reduce at the exchanges of a trial: strong scaling, value = the whole
problem's trials over the slowest rank's time); --mode replicas gives each
rank its own replica instead (weak scaling).
"""
from __future__ import annotations

import os

for _v in ("OPENBLAS_NUM_THREADS", "OMP_NUM_THREADS", "MKL_NUM_THREADS"):
    os.environ.setdefault(_v, "1")

import argparse
import csv
import hashlib
import io
import json
import math
import signal
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

import scenegen  # noqa: E402

METRIC = "LM iters/s and time-to-cost (1e-6 rel) vs plain GPU and oracle; HBM GB/s vs peak"
UNIT = "LM iters/s"
WORKLOAD = "ba4000"
PCG_MAXITER = 50
PCG_TOL = 1e-4


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=60)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--backend", choices=["nccl", "gloo"], default="nccl",
                    help="torch.distributed backend of the exchanges under torchrun (gloo: ranks may share a GPU)")
    ap.add_argument("--e2e-steps", type=int, default=0,
                    help="trials of the end-to-end leg (default: --steps, the timed trials)")
    ap.add_argument("--profile-trials", type=int, default=4)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--jacobian", choices=["auto", "recompute", "store"], default="auto")
    ap.add_argument("--precision", choices=["both", "f64", "f32"], default="both",
                    help="both: the FP64 line (the paper's arithmetic) with the FP32 variant inside it")
    ap.add_argument("--mode", choices=["partition", "replicas"], default="partition",
                    help="N > 1: one problem partitioned by points over the GPUs (strong scaling), or one "
                         "replica of the problem per GPU (weak scaling)")
    ap.add_argument("--no-time-to-cost", action="store_true",
                    help="skip F_ref and the time-to-cost runs (profiling only)")
    ap.add_argument("--points", type=int, default=0,
                    help="profiling only: same recipe with fewer points")
    ap.add_argument("--workload", choices=["ba4000", "batch512", "learned", "adjoint", "pgo", "direct"],
                    default="ba4000",
                    help="batch512: 512 sliding-window problems solved by one persistent launch; "
                         "learned: time to 1e-6 relative cost with the learned block-Jacobi correction")
    ap.add_argument("--train-scenes", type=int, default=200, help="learned: training scenes")
    ap.add_argument("--seeds", type=int, default=3, help="learned: training seeds (initialisation and shuffle)")
    ap.add_argument("--batch-problems", type=int, default=512,
                    help="batch512: problems per rank (profiling only: a smaller batch of the same recipe)")
    ap.add_argument("--no-sequential", action="store_true",
                    help="batch512: skip the 512 sequential single-problem solves")
    return ap.parse_args()


def dist_env():
    return (int(os.environ.get("RANK", "0")), int(os.environ.get("WORLD_SIZE", "1")),
            int(os.environ.get("LOCAL_RANK", "0")))


def rank_max(value, device, world):
    """The largest value over all ranks (the slowest rank's time); the value
    itself on one rank.  No data-path collective: timing only."""
    if world <= 1:
        return float(value)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def batch_seed(rank):
    """Seed of a rank's own batch of problems (weak scaling: every rank
    solves BATCH_N problems of its own, no data-path collective)."""
    return 4 + 1000 * rank


# --------------------------------------------------------------------------
# the CPU oracle on a bounded sample (cpu_baseline and --impl reference)
# --------------------------------------------------------------------------

def oracle_sample_rate(scene, n_obs_target, trials=1, warmup=0):
    """LM trials/s of the oracle on a sample of the scene, scaled to the full
    scene by its observation count (per-trial work is linear in O)."""
    import oracle as orc
    n_pts = max(50, int(round(n_obs_target * scene.P / scene.O)))
    sub = scenegen.subsample_points(scene, n_pts, seed=123)
    pix = orc.pixels_from_scene(sub)
    opts = orc.LMOptions(solver="pcg", pcg_tol=0.0, pcg_maxiter=PCG_MAXITER,
                         huber_delta=sub.huber_delta)
    if warmup:
        orc.lm(sub.cams_init, sub.points_init, sub.cam_idx, sub.pt_idx, pix, warmup, opts)
    t0 = time.perf_counter()
    _, _, tr = orc.lm(sub.cams_init, sub.points_init, sub.cam_idx, sub.pt_idx, pix, trials, opts)
    dt = time.perf_counter() - t0
    rate_sample = trials / dt
    return dict(rate_full=rate_sample * sub.O / scene.O, seconds=dt, O=sub.O, P=sub.P,
                trials=trials, pcg=[t["pcg_iters"] for t in tr])


def run_reference(args):
    rank, world, _ = dist_env()
    if rank != 0:
        return
    scene = scenegen.config_scene(WORKLOAD)
    # per-step sample sized so (K + W) steps take about two minutes
    per_step_s = 120.0 / max(1, args.steps + args.warmup)
    n_obs = int(min(1_000_000, max(3000, per_step_s / 45e-6)))
    r = oracle_sample_rate(scene, n_obs, trials=args.steps, warmup=args.warmup)
    v = r["rate_full"]
    sample = (f"{r['P']} of {scene.P} points with their {r['O']} of {scene.O} observations, "
              f"all {scene.C} cameras; {args.steps} LM trials per run, PCG fixed at "
              f"{PCG_MAXITER} iterations; rate scaled by O_full/O_sample")
    line = {"metric": METRIC, "value": v, "unit": UNIT, "impl": "reference", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000.0 / v,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic",
            "config": {"workload": WORKLOAD, "cameras": scene.C, "points": scene.P,
                       "observations": scene.O, "pcg_maxiter": PCG_MAXITER},
            "cpu_baseline": {"value": v, "unit": UNIT, "cores": 1, "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# --------------------------------------------------------------------------
# GPU arm
# --------------------------------------------------------------------------

class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.f = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        self.proc = None
        self.gpu = gpu_index
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(gpu_index), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.f, stderr=subprocess.DEVNULL)
        except (FileNotFoundError, OSError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.send_signal(signal.SIGTERM)
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.f.seek(0)
        text = self.f.read()
        os.unlink(self.f.name)
        return parse_clock_samples(text)


def parse_clock_samples(text):
    """Summary of nvidia-smi samples in the ClockSampler.Q column order
    (csv, no header, no units): median SM clock, the highest maximum clock,
    the throttle reasons seen Active in any sample, and the sample count;
    None without samples."""
    rows = [r for r in csv.reader(io.StringIO(text)) if len(r) >= 9]
    if not rows:
        return None
    sm = [float(r[1]) for r in rows if r[1].strip().replace(".", "").isdigit()]
    mx = [float(r[2]) for r in rows if r[2].strip().replace(".", "").isdigit()]
    names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
    reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i].strip() == "Active"})
    return {"sm_mhz": statistics.median(sm) if sm else None,
            "sm_max_mhz": max(mx) if mx else None, "reasons": reasons, "samples": len(rows)}


def algorithmic_bytes(kind, C, P, O, npieces, tsize, mf, huber=False, pairs=0):
    """Compulsory HBM bytes of one launch: every array element the kernel
    must read or write, each counted once (per-observation planes, indices
    and weights; per-point / per-camera vectors once)."""
    # stored planes (the passes of the Schur product and the linearisation
    # also read or write the 6 planes of Jp) or sqrt(w)
    ob = (24 if kind in ("pass_b", "pass_a1", "pass_fa", "schur_cam", "lin_cam") else 18) * tsize if not mf else \
        (tsize if huber else 0)
    sw = tsize if huber else 0
    if kind == "pass_b":   # cm_pt; point record (X, t) per point; camera table; partials
        return O * (4 + ob) + P * 8 * tsize + npieces * 9 * 8 + C * 16 * tsize
    if kind == "pass_a1":  # cm_pt (+ sqrt(w)) or planes in, one 4-vector out per obs; points once
        return O * (4 + ob + 4 * tsize) + (P * 4 * tsize if mf else 0) + C * (16 + 12) * tsize
    if kind == "pass_a2":  # order map + one 4-vector per obs; rowptr, V*^-1, t out per point
        return O * (4 + 4 * tsize) + P * (4 + 6 * tsize + 4 * tsize)
    if kind == "pass_fa":
        if not mf:  # stored: the point-major planes + camera position per obs; rowptr, V*^-1 in, t out per point
            return O * (ob + 2) + P * (4 + 6 * tsize + 4 * tsize) + C * 9 * tsize
        # recompute: point index + chunk camera position (+ sqrt(w)) per obs; X in, V*^-1, t out per point
        return O * (4 + 2 + sw) + P * (4 + 4 * tsize + 6 * tsize + 4 * tsize)
    if kind == "lin_cam":  # pixels + point index in; planes / weights out; points once; partials
        return O * (2 * tsize + 4 + ob) + P * 3 * tsize + npieces * 54 * 8
    if kind == "lin_pt":
        return O * (2 * tsize + 8 + ob) + P * (4 + 3 * tsize + 9 * 8) + C * 32 * tsize
    if kind == "schur_cam":
        return O * (4 + ob) + P * ((3 * tsize if mf else 0) + 9 * tsize) + npieces * 54 * 8
    if kind == "form":     # per pair its two slots (FP32 also its point); the lean planes, or points and V*^-1
        return pairs * 12 + P * (8 + 6) * tsize + C * 32 * tsize if mf else pairs * 8 + O * 20 * tsize
    if kind == "cost":     # pixels, point index, (model) planes; trial + current points, dp
        return O * (2 * tsize + 4 + ob) + P * 9 * tsize + npieces * 2 * 8
    if kind == "backsub":  # A1 + A2 of the back-substitution (two launches per trial)
        return (O * (4 + ob + 4 * tsize) + (P * 4 * tsize if mf else 0)
                + O * (4 + 4 * tsize) + P * (4 + 6 * tsize + 3 * tsize + 3 * 8 + 9 * tsize)) // 2
    return 0


# Floating-point operations per observation of the PCG passes (an FMA counts
# two), read off the kernels' arithmetic.  Recompute mode (FP32 default): the
# factored Jacobian (58) plus the pass's products (the fused pass A adds the
# 3 additions of its per-point sums).  Stored mode (FP64 default): products
# with the stored planes only (pass A1: e = Jc x, 18 FMA, and z = Jp^T e;
# pass B: h = Jp t and the sum of Jc^T h, 18 FMA).
FLOPS_PER_OBS = {"pass_b": 116, "pass_a1": 113, "pass_fa": 116}
FLOPS_PER_OBS_STORED = {"pass_a1": 45, "pass_a2": 3, "pass_fa": 48, "pass_b": 46}
# per point: V*^-1 times the summed 3-vector (9 FMA)
FLOPS_PER_POINT = {"pass_a2": 18, "pass_fa": 18}


def pass_flops(kind, O, P, mf):
    per_obs = (FLOPS_PER_OBS if mf else FLOPS_PER_OBS_STORED).get(kind)
    if per_obs is None:
        return None
    return per_obs * O + FLOPS_PER_POINT.get(kind, 0) * P


def fp32_peak_tflops(sm_mhz):
    """152 SMs x 128 FP32 lanes x 2 flops per FMA x clock."""
    return 152 * 128 * 2 * sm_mhz * 1e6 / 1e12


def kernel_source_hash():
    h = hashlib.sha256()
    for f in ("ba_kernels.cuh", "ba_schur.cuh", "ba_vec.cuh", "ba_api.cu"):
        with open(os.path.join(ROOT, "paper_2409_12190_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def measured_traffic(kernel, src_hash, prec):
    """dram bytes per launch of the kernel class at this precision from a
    committed ncu summary, only if it was taken on the current kernel
    source."""
    path = os.path.join(ROOT, "profiles", "ncu_traffic.json")
    try:
        with open(path) as fh:
            d = json.load(fh)
    except (OSError, ValueError):
        return None
    e = d.get(f"{kernel}_{prec}")
    if not e or e.get("source_hash") != src_hash:
        return None
    return e.get("dram_bytes_per_launch")


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            d = json.load(fh)
        return float(d["hbm_gbs"]), "measured"
    except (OSError, ValueError, KeyError):
        return 6800.0, "fallback"


# F_ref (the converged FP64 cost of the ba4000 workload): the benchmark's FP32
# run until it stalls, then FP64 trials with a tight PCG from its parameters
# until an accepted trial lowers the cost by less than F_REF_STOP (relative).
F_REF_F32_TRIALS = 150
F_REF_PCG = (1500, 1e-12)
F_REF_MAX_TRIALS = 12
F_REF_STOP = 1e-9
TTC_REL = 1e-6          # time to (1 + 1e-6) F_ref
TTC_MAX_TRIALS = {"f64": 150, "f32": 250}


def converged_cost(trace, F0):
    """Lowest cost of an LM trace: the starting cost or an accepted trial's."""
    acc = [t["cost_trial"] for t in trace if t["accepted"]]
    return min([F0] + acc)


def f_ref_stop(trace, rel=F_REF_STOP):
    """True once the last accepted trial of a polishing run lowered the cost
    by less than rel (relative)."""
    acc = [t for t in trace if t["accepted"]]
    return bool(acc) and (acc[-1]["cost"] - acc[-1]["cost_trial"]) <= rel * acc[-1]["cost"]


def first_at_or_below(costs, target):
    """Index of the first cost at or below target, else None."""
    return next((i for i, c in enumerate(costs) if c <= target), None)


def _scene_inputs(scene, dev):
    """The scene's indices and its pixels (projection of the ground truth by
    the library in FP64, plus the scene's noise), on the device."""
    import torch
    import paper_2409_12190_gb300 as ba
    ci = torch.from_numpy(scene.cam_idx).to(dev)
    pi = torch.from_numpy(scene.pt_idx).to(dev)
    cams_gt = torch.tensor(scene.cams_gt, dtype=torch.float64, device=dev)
    pts_gt = torch.tensor(scene.points_gt, dtype=torch.float64, device=dev)
    pix = ba.project(cams_gt, pts_gt, ci, pi) + torch.tensor(scene.noise, dtype=torch.float64, device=dev)
    return ci, pi, pix


def _problem(scene, ci, pi, pix, prec, dev, jacobian="auto", maxiter=PCG_MAXITER, tol=PCG_TOL, part=None):
    """The benchmark's problem in precision prec; with part = (bounds, rank,
    allreduce) this rank's part of the point-partitioned problem."""
    import torch
    import paper_2409_12190_gb300 as ba
    opts = ba.Options(precision=prec, pcg_maxiter=maxiter, pcg_tol=tol, use_graph=True, jacobian=jacobian)
    dt = torch.float32 if prec == "f32" else torch.float64
    if part is None:
        return ba.Problem(scene.cams_init, scene.points_init, ci, pi, pix.to(dt), opts, device=dev)
    from paper_2409_12190_gb300.partition import PartProblem
    bounds, rank, allreduce = part
    lo, hi = int(bounds[rank]), int(bounds[rank + 1])
    obs = torch.nonzero((pi >= lo) & (pi < hi)).flatten()
    prob = PartProblem(scene.cams_init, scene.points_init[lo:hi], ci[obs], pi[obs] - lo, pix[obs].to(dt),
                       allreduce, opts, device=dev)
    prob.pix_part = pix[obs]
    return prob


def compute_f_ref(scene, ci, pi, pix, dev, want_params=False, part=None):
    """F_ref and how it was reached (see F_REF_*); with want_params also the
    FP64 parameters (cams, points) at which it was evaluated (this part's
    points for a partitioned problem)."""
    import torch
    t0 = time.perf_counter()
    with _problem(scene, ci, pi, pix, "f32", dev, part=part) as p32:
        p32.solve(F_REF_F32_TRIALS)
        cams, pts = p32.params()
        F32, _ = p32.scalars()
    with _problem(scene, ci, pi, pix, "f64", dev, maxiter=F_REF_PCG[0], tol=F_REF_PCG[1], part=part) as p64:
        p64.set_params(cams.double(), pts.double())
        p64.set_lambda(1e-6)
        n = 0
        while n < F_REF_MAX_TRIALS:
            p64.solve(1)
            n += 1
            if f_ref_stop(p64.stats(cap=n)):
                break
        trace = p64.stats(cap=n)
        F, _ = p64.scalars()
        params = p64.params() if want_params else None
    torch.cuda.synchronize()
    last = [t for t in trace if t["accepted"]]
    return F, {"f_ref": F, "rule": (f"FP32 benchmark run for {F_REF_F32_TRIALS} trials (cost {F32:.9g}), then FP64 "
                                    f"trials with PCG maxiter {F_REF_PCG[0]} / tol {F_REF_PCG[1]:g} until an accepted "
                                    f"trial lowers the cost by less than {F_REF_STOP:g} relative"),
               "fp64_trials": n, "last_accepted_decrease_rel": ((last[-1]["cost"] - last[-1]["cost_trial"])
                                                                / last[-1]["cost"]) if last else None,
               "seconds": time.perf_counter() - t0}, *((params,) if want_params else ())


def time_to_f_ref(prob, state0, f_ref, max_trials, stream):
    """From the starting state: LM trials one by one (graph replay) with an
    event after each, until the cost is within TTC_REL of f_ref."""
    import torch
    prob.set_state(state0)
    torch.cuda.synchronize()
    prob.stats()
    target = (1.0 + TTC_REL) * f_ref
    e0 = torch.cuda.Event(enable_timing=True)
    evs = []
    costs = []
    e0.record(stream)
    chunk = 10
    while len(costs) < max_trials:
        for _ in range(min(chunk, max_trials - len(costs))):
            prob.solve(1)
            ev = torch.cuda.Event(enable_timing=True)
            ev.record(stream)
            evs.append(ev)
        torch.cuda.synchronize()
        st = prob.stats(cap=len(evs) - len(costs))
        costs += [t["cost_trial"] if t["accepted"] else t["cost"] for t in st]
        if first_at_or_below(costs, target) is not None:
            break
    hit = first_at_or_below(costs, target)
    return {"time_to_cost_s": e0.elapsed_time(evs[hit]) / 1000.0 if hit is not None else None,
            "trials_to_cost": None if hit is None else hit + 1, "target": target, "trials_run": len(costs),
            "final_cost": costs[-1], "rel_gap_at_end": costs[-1] / f_ref - 1.0}


# operations per pair of observations of one point, where the reduced system
# is formed: 157 FP64 multiply-adds from the lean form; FP32 the 9 x 3 by 3 x 9
# product of the two couplings
FORM_FLOPS_PER_PAIR = {"f64": 314, "f32": 486}


def observation_pairs(pt_idx):
    n = np.bincount(pt_idx).astype(np.int64)
    return int((n * (n - 1) // 2).sum())


def kernel_table(per, C, P, O, lay, tsize, mf, huber, alu_peak, pairs=0, flops_per_pair=0):
    """Per kernel class: launches, mean CUDA-event time, share, algorithmic
    GB/s and (PCG passes, forming S) TFLOP/s with their fractions."""
    total = sum(v[0] for v in per.values())
    out = {}
    for name, (kms, n) in per.items():
        if n == 0:
            continue
        pieces = lay["product_pieces" if name.startswith("pass_") else "pieces"]
        b = algorithmic_bytes(name, C, P, O, pieces, tsize, mf, huber, pairs)
        avg = kms / n
        row = {"launches": n, "avg_us": 1000.0 * avg, "share": kms / total,
               "gbs": (b / (avg / 1000.0) / 1e9) if b else None, "bytes_per_launch": b or None}
        fl = flops_per_pair * pairs if name == "form" else pass_flops(name, O, P, mf)
        if fl:
            row["tflops"] = fl / (avg / 1000.0) / 1e12
            row["flops_per_launch"] = fl
            row["alu_frac"] = row["tflops"] / alu_peak
        out[name] = row
    return out


def roofline_of(kernels, per, hbm_peak, hbm_kind, alu_peak, alu_source, src_hash, prof_ms, it_bytes, prec):
    """Roofline block of the dominant kernel (largest share of the profiled
    time among the kernels with an algorithmic byte count): its HBM and ALU
    fractions; "bound" is the larger of the two."""
    dom = max((k for k in kernels if kernels[k]["gbs"]), key=lambda k: per[k][0])
    kr = kernels[dom]
    hbm = {"achieved": kr["gbs"], "peak": hbm_peak, "unit": "GB/s", "frac": kr["gbs"] / hbm_peak,
           "peak_source": hbm_kind}
    roof = {"bound": "hbm", "kernel": dom, **hbm, "bytes_per_launch": kr["bytes_per_launch"],
            "traffic": measured_traffic(dom, src_hash, prec), "kernel_source": src_hash, "hbm": hbm}
    if "tflops" in kr:
        alu = {"achieved": kr["tflops"], "peak": alu_peak, "unit": "TFLOP/s", "frac": kr["alu_frac"],
               "flops_per_launch": kr["flops_per_launch"], "peak_source": alu_source}
        roof["alu"] = alu
        if alu["frac"] > hbm["frac"]:
            roof.update({"bound": "alu", "achieved": alu["achieved"], "peak": alu_peak, "unit": "TFLOP/s",
                         "frac": alu["frac"], "peak_source": alu_source})
    roof["iteration_gbs"] = it_bytes / (prof_ms / 1000.0) / 1e9
    roof["iteration_frac"] = roof["iteration_gbs"] / hbm_peak
    return roof


def run_precision(args, prec, scene, ci, pi, pix, dev, world, f_ref, peaks_d, barrier, clocks_for_rank, part=None):
    """One precision of the benchmark: timed trials, per-kernel profile and
    roofline, time to F_ref, and the end-to-end leg through the public API.
    With part, every rank solves its part of one point-partitioned problem
    (strong scaling: the value counts the whole problem's trials once)."""
    import torch
    import paper_2409_12190_gb300 as ba
    prob = _problem(scene, ci, pi, pix, prec, dev, jacobian=args.jacobian, part=part)
    C, P, O = prob.C, prob.P, prob.O       # this rank's share of the work
    tsize = 4 if prec == "f32" else 8
    torch.cuda.synchronize()
    lay = prob.layout()
    mf = not lay["stored"]
    state_init = prob.get_state()
    prob.solve(args.warmup)   # captures the trial graph on first use
    torch.cuda.synchronize()
    prob.stats()
    state0 = prob.get_state()  # the end-to-end leg replays the timed trials from here
    stream = torch.cuda.current_stream()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    clocks = clocks_for_rank()
    time.sleep(0.3 if clocks else 0)
    barrier()
    torch.cuda.synchronize()
    n0 = ba.kernel_launch_count()
    e0.record(stream)
    prob.solve(args.steps)
    e1.record(stream)
    torch.cuda.synchronize()
    barrier()
    launches = ba.kernel_launch_count() - n0
    clk = clocks.stop() if clocks else None
    ms = rank_max(e0.elapsed_time(e1), dev, world)
    trials = prob.stats(cap=args.steps)
    copies = 1 if part is not None else world   # replicas: every rank solves a whole problem
    value = copies * args.steps / (ms / 1000.0)

    # per-kernel CUDA-event timing of real trials (direct launches)
    per, prof_ms = prob.profile_trials(args.profile_trials)
    sm_mhz = (clk or {}).get("sm_max_mhz") or 2070.0
    if prec == "f32":
        alu_peak, alu_source = fp32_peak_tflops(sm_mhz), f"152 SMs x 128 FP32 lanes x 2 x {sm_mhz:.0f} MHz"
    else:
        alu_peak = peaks_d["fp64_fma_tflops"]
        alu_source = "measured (ba_measure_fma_peak: FP64 FMA chains on every SM, best of 3)"
    huber = scene.huber_delta > 0
    formed = lay["formed"] == 1
    pairs = observation_pairs(scene.pt_idx) if formed else 0
    kernels = kernel_table(per, C, P, O, lay, tsize, mf, huber, alu_peak, pairs, FORM_FLOPS_PER_PAIR[prec])
    it_bytes = sum((k["bytes_per_launch"] or 0) * k["launches"] for k in kernels.values())
    roof = roofline_of(kernels, per, peaks_d["hbm_gbs"], peaks_d["hbm_kind"], alu_peak, alu_source,
                       kernel_source_hash(), prof_ms, it_bytes, prec)

    # end to end through the public API: the same trials as the timed region
    # (restarted from its starting state), each step uploading parameters and
    # pixels from pinned host memory and reading parameters and cost back
    e2e_steps = args.e2e_steps if args.e2e_steps > 0 else args.steps
    dt = torch.float32 if prec == "f32" else torch.float64
    prob.set_state(state0)
    hc = torch.empty((C, 9), dtype=dt).pin_memory()
    hp = torch.empty((P, 3), dtype=dt).pin_memory()
    hx = getattr(prob, "pix_part", pix).to(dt).cpu().pin_memory()
    prob.get_params_into(hc, hp)
    torch.cuda.synchronize()
    barrier()
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        prob.set_params(hc, hp)
        prob.set_pixels(hx)
        prob.lm_step()
        prob.get_params_into(hc, hp)
        prob.scalars()
    torch.cuda.synchronize()
    e2e_s = rank_max(time.perf_counter() - t0, dev, world)
    e2e_trials = prob.stats(cap=e2e_steps)
    same = ([t["pcg_iters"] for t in e2e_trials] == [t["pcg_iters"] for t in trials[:e2e_steps]]
            and [t["accepted"] for t in e2e_trials] == [t["accepted"] for t in trials[:e2e_steps]])
    e2e = {"value": copies * e2e_steps / e2e_s, "unit": UNIT,
           "h2d_bytes_per_step": (9 * C + 3 * P + 2 * O) * tsize,
           "d2h_bytes_per_step": (9 * C + 3 * P) * tsize + 8, "steps": e2e_steps,
           "same_trials_as_timed": same}

    # time to (1 + 1e-6) F_ref from the scene's initial parameters
    ttc = time_to_f_ref(prob, state_init, f_ref, TTC_MAX_TRIALS[prec], stream) if f_ref else None
    prob.close()
    pcg = [t["pcg_iters"] for t in trials]
    cfg = {"workload": scene.name, "cameras": C, "points": P, "observations": O,
           "precision": ("f32 per-observation, f64 reductions" if prec == "f32" else "f64 throughout"),
           "loss": "squared", "pcg": f"block-Jacobi, maxiter {PCG_MAXITER}, tol {PCG_TOL}",
           "pcg_iters_mean": statistics.mean(pcg) if pcg else None, "pcg_iters_total": sum(pcg),
           "accepted": sum(t["accepted"] for t in trials),
           "l2": "inputs larger than L2 (each pass streams >0.1 GB of per-observation data; L2 129 MB)",
           "parallelism": (f"points partitioned over {world} GPUs (cameras replicated, NCCL all-reduce at the "
                           f"six exchanges of a trial)" if part is not None else
                           ("replicas" if world > 1 else "single GPU")),
           "graph": "direct launches (exchanges)" if part is not None else "one CUDA graph per LM trial",
           "jacobian": "recomputed in every pass" if mf else "stored planes",
           "schur_product": ("formed S, its PCG in one launch" if formed else
                             "fused point-major pass A + pass B" if lay["fused_a"] else "passes A1, A2, B")}
    return {"value": value, "ms_per_step": ms / args.steps, "dtype": prec, "config": cfg, "gpu_launches": launches,
            "clocks": clk, "roofline": roof, "kernels": kernels, "e2e": e2e, "time_to_cost": ttc}


def _oracle_sample_job(job):
    """One bounded oracle run (a spawned worker): LM trials/s of the oracle on
    a sample of the scene, scaled to the full scene by its observation count.
    The sample is drawn by the parent, so only it crosses the process
    boundary."""
    sub, O_full, trials = job
    import oracle as orc
    pix = orc.pixels_from_scene(sub)
    opts = orc.LMOptions(solver="pcg", pcg_tol=0.0, pcg_maxiter=PCG_MAXITER, huber_delta=sub.huber_delta)
    t0 = time.perf_counter()
    orc.lm(sub.cams_init, sub.points_init, sub.cam_idx, sub.pt_idx, pix, trials, opts)
    dt = time.perf_counter() - t0
    return {"rate_full": trials / dt * sub.O / O_full, "seconds": dt, "O": sub.O, "P": sub.P}


def _sample(scene, n_obs, seed):
    n_pts = max(50, int(round(n_obs * scene.P / scene.O)))
    return scenegen.subsample_points(scene, n_pts, seed=seed)


def cpu_baseline(scene, n_obs_single=500_000, n_obs_each=250_000):
    """The oracle on the host cores: one thread on one sample, then one
    single-threaded process per core (spawned), each on its own sample, run
    together (the host's throughput); plus one full ba250 trial, unscaled."""
    import multiprocessing as mp
    import oracle as orc
    ncores = os.cpu_count() or 1
    single = _oracle_sample_job((_sample(scene, n_obs_single, 123), scene.O, 1))
    jobs = [(_sample(scene, n_obs_each, 1000 + i), scene.O, 1) for i in range(ncores)]
    with mp.get_context("spawn").Pool(ncores) as pool:
        t0 = time.perf_counter()
        many = pool.map(_oracle_sample_job, jobs)
        wall = time.perf_counter() - t0
    del jobs
    total_rate = sum(r["O"] for r in many) / scene.O / wall   # full-scene trials/s of all processes together
    b250 = scenegen.config_scene("ba250")
    pix = orc.pixels_from_scene(b250)
    t0 = time.perf_counter()
    orc.lm(b250.cams_init, b250.points_init, b250.cam_idx, b250.pt_idx, pix, 1,
           orc.LMOptions(solver="pcg", pcg_tol=1e-4, pcg_maxiter=PCG_MAXITER, huber_delta=b250.huber_delta))
    t250 = time.perf_counter() - t0
    return {"value": total_rate, "unit": UNIT, "cores": ncores, "kind": "oracle",
            "sample": (f"{ncores} single-threaded oracle processes (one per host core, spawned), each one LM "
                       f"trial (PCG fixed at {PCG_MAXITER} iterations) on its own sample of ~{n_obs_each} of "
                       f"{scene.O} observations with all {scene.C} cameras, run together in {wall:.1f} s "
                       f"(spawn and imports included); throughput scaled by O_full/O_sample"),
            "nproc": ncores,
            "single_thread": {"value": single["rate_full"], "cores": 1,
                              "sample": f"1 trial on {single['O']} observations, {single['seconds']:.1f} s, "
                                        f"scaled by O_full/O_sample"},
            "ba250_full_trial_s": t250}


def run_ours(args):
    import torch
    import paper_2409_12190_gb300 as ba
    from paper_2409_12190_gb300 import build as bbuild

    rank, world, local = dist_env()
    local = local % max(1, torch.cuda.device_count())  # ranks share the GPUs when there are fewer
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        import torch.distributed as dist
        if args.backend == "nccl":
            dist.init_process_group("nccl", device_id=dev)
        else:
            dist.init_process_group("gloo")
    bbuild.build()

    def barrier():
        if world > 1:
            import torch.distributed as dist
            dist.barrier()

    if args.points:
        scene = scenegen.ring_scene(4000, args.points, seed=3, view_p=1.0 / 5.7, name="ba4000-small")
    else:
        scene = scenegen.config_scene(WORKLOAD)
    ci, pi, pix = _scene_inputs(scene, dev)
    part = None
    if world > 1 and args.mode == "partition":
        from paper_2409_12190_gb300.partition import dist_allreduce, partition_points
        bounds, _ = partition_points(scene.pt_idx, scene.P, world)
        part = (bounds, rank, dist_allreduce())
    hbm, hbm_kind = peaks()
    peaks_d = {"hbm_gbs": hbm, "hbm_kind": hbm_kind, "fp64_fma_tflops": ba.measure_fma_peak("f64"),
               "fp32_fma_tflops": ba.measure_fma_peak("f32")}
    f_ref, f_ref_info = (None, None) if args.no_time_to_cost else compute_f_ref(scene, ci, pi, pix, dev, part=part)
    precs = ["f64", "f32"] if args.precision == "both" else [args.precision]
    res = {}
    for p in precs:
        res[p] = run_precision(args, p, scene, ci, pi, pix, dev, world, f_ref, peaks_d, barrier,
                               lambda: ClockSampler(local) if rank == 0 else None, part=part)
    if rank != 0:
        return
    cpu = None
    if world == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline(scene)
    head = res[precs[0]]
    line = {"metric": METRIC, "value": head["value"], "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": head["ms_per_step"], "higher_is_better": True,
            "scaling": "strong" if part is not None else "weak", "vs_baseline": None, "dtype": head["dtype"],
            "data": "synthetic",
            "config": dict(head["config"], f_ref=f_ref_info),
            "gpu_launches": head["gpu_launches"], "clocks": head["clocks"], "roofline": head["roofline"],
            "kernels": head["kernels"], "cpu_baseline": cpu, "e2e": head["e2e"],
            "time_to_cost": head["time_to_cost"],
            "measured_peaks": {k: v for k, v in peaks_d.items()}}
    if len(precs) > 1:
        line["variants"] = {p: res[p] for p in precs[1:]}
    print(json.dumps(line), flush=True)


# --------------------------------------------------------------------------
# batch512: many small problems, one persistent launch per solve
# --------------------------------------------------------------------------

BATCH_N = 512
BATCH_ITERS = 10
# operations of a 9 x 9 block of the formed system in a product
BATCH_FLOPS_PER_BLOCK = 162


def run_batch(args):
    import torch
    import paper_2409_12190_gb300 as ba
    from paper_2409_12190_gb300 import build as bbuild

    rank, world, local = dist_env()
    local = local % max(1, torch.cuda.device_count())
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        import torch.distributed as dist
        if args.backend == "nccl":
            dist.init_process_group("nccl", device_id=dev)
        else:
            dist.init_process_group("gloo")
    bbuild.build()
    n_prob = args.batch_problems
    scenes = scenegen.batch_scenes(n_prob, seed=batch_seed(rank))
    O = sum(s.O for s in scenes)
    inputs = []
    for s in scenes:
        ci = torch.from_numpy(s.cam_idx).to(dev)
        pi = torch.from_numpy(s.pt_idx).to(dev)
        px = ba.project(torch.tensor(s.cams_gt, dtype=torch.float32, device=dev),
                        torch.tensor(s.points_gt, dtype=torch.float32, device=dev), ci, pi)
        px = px + torch.tensor(s.noise, dtype=torch.float32, device=dev)
        inputs.append((s.cams_init, s.points_init, ci, pi, px))
    opts = ba.Options(precision="f32", pcg_maxiter=PCG_MAXITER, pcg_tol=PCG_TOL)
    bt = ba.Batch(inputs, opts, device=dev)
    cache = os.path.join(ROOT, "paper_2409_12190_gb300", ".autotune.jsonl")
    cfg, tune_ms = bt.autotune(BATCH_ITERS, cache)
    for _ in range(args.warmup):
        bt.reset()
        bt.solve(BATCH_ITERS)
    torch.cuda.synchronize()

    stream = torch.cuda.current_stream()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    clocks = ClockSampler(local) if rank == 0 else None
    time.sleep(0.3 if clocks else 0)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    n0 = ba.kernel_launch_count()
    e0.record(stream)
    for _ in range(args.steps):
        bt.reset()
        bt.solve(BATCH_ITERS)
    e1.record(stream)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    launches = ba.kernel_launch_count() - n0
    clk = clocks.stop() if clocks else None
    ms = e0.elapsed_time(e1)
    ms = rank_max(ms, dev, world)
    stats = bt.stats()
    pcg_total = sum(t["pcg_iters"] for st in stats for t in st)
    costs, _ = bt.scalars()
    # problem-iterations per second over all ranks
    value = world * n_prob * BATCH_ITERS * args.steps / (ms / 1000.0)

    # the solve alone (one persistent launch, no reset) for the roofline
    bt.reset()
    torch.cuda.synchronize()
    e0.record(stream)
    bt.solve(BATCH_ITERS)
    e1.record(stream)
    torch.cuda.synchronize()
    solve_ms = e0.elapsed_time(e1)
    st2 = bt.stats()
    # the windows' systems are formed once a trial (FP32, recomputed Jacobians)
    flops = sum(len(st) * FORM_FLOPS_PER_PAIR["f32"] * observation_pairs(s.pt_idx)
                + BATCH_FLOPS_PER_BLOCK * s.C * s.C * sum(t["pcg_iters"] for t in st) for st, s in zip(st2, scenes))
    sm_mhz = (clk or {}).get("sm_max_mhz") or 2070.0
    alu_peak = fp32_peak_tflops(sm_mhz)
    ach = flops / (solve_ms / 1000.0) / 1e12
    roofline = {"bound": "alu", "kernel": "k_batch_lm", "achieved": ach, "peak": alu_peak, "unit": "TFLOP/s",
                "frac": ach / alu_peak, "flops_per_launch": flops,
                "peak_source": f"152 SMs x 128 FP32 lanes x 2 x {sm_mhz:.0f} MHz",
                "note": "forming (486 FP32 flops per pair of observations of a point) and the formed products "
                        "(162 per camera pair and PCG iteration); each problem's arrays stay in L2", "traffic": None}

    # end to end: pinned host parameters in, solve, parameters out
    C, P = bt.C, bt.P
    hc = torch.from_numpy(np.concatenate([s.cams_init for s in scenes]).astype(np.float32)).pin_memory()
    hp = torch.from_numpy(np.concatenate([s.points_init for s in scenes]).astype(np.float32)).pin_memory()
    oc = torch.empty((C, 9), dtype=torch.float32).pin_memory()
    op = torch.empty((P, 3), dtype=torch.float32).pin_memory()
    torch.cuda.synchronize()
    e2e_steps = args.e2e_steps if args.e2e_steps > 0 else args.steps
    t0 = time.perf_counter()
    for _ in range(e2e_steps):
        bt.reset(hc, hp)
        bt.solve(BATCH_ITERS)
        cams_d, pts_d = bt.params(split=False)
        oc.copy_(cams_d, non_blocking=True)
        op.copy_(pts_d, non_blocking=True)
        torch.cuda.synchronize()
    e2e_s = time.perf_counter() - t0
    e2e = {"value": world * n_prob * BATCH_ITERS * e2e_steps / e2e_s, "unit": "problem LM iters/s",
           "h2d_bytes_per_step": (9 * C + 3 * P) * 4, "d2h_bytes_per_step": (9 * C + 3 * P) * 4,
           "steps": e2e_steps}

    if rank != 0:
        return
    seq = None
    if world == 1 and not args.no_sequential:
        # the same problems solved one after another by the single-problem path
        ev0 = torch.cuda.Event(enable_timing=True)
        ev1 = torch.cuda.Event(enable_timing=True)
        tot = 0.0
        worst = 0.0
        for b, inp in enumerate(inputs):
            pr = ba.Problem(*inp, options=opts, device=dev)
            torch.cuda.synchronize()
            ev0.record(stream)
            pr.solve(BATCH_ITERS)
            ev1.record(stream)
            torch.cuda.synchronize()
            tot += ev0.elapsed_time(ev1)
            F, _ = pr.scalars()
            worst = max(worst, abs(costs[b] - F) / F)
            pr.close()
        seq = {"ms": tot, "problem_iters_per_s": n_prob * BATCH_ITERS / (tot / 1000.0),
               "speedup_of_batch": tot / solve_ms, "max_rel_final_cost_diff": worst}
    cpu = None
    if world == 1 and not args.no_cpu_baseline:
        import oracle as orc
        t0 = time.perf_counter()
        n_done, obs_done = 0, 0
        for s in scenes[:3]:
            pix = orc.pixels_from_scene(s)
            orc.lm(s.cams_init, s.points_init, s.cam_idx, s.pt_idx, pix, BATCH_ITERS,
                   orc.LMOptions(solver="pcg", pcg_tol=PCG_TOL, pcg_maxiter=PCG_MAXITER))
            n_done += 1
            obs_done += s.O
        dt = time.perf_counter() - t0
        rate = n_done * BATCH_ITERS / dt * (obs_done / n_done) / (O / n_prob)
        cpu = {"value": rate, "unit": "problem LM iters/s", "cores": 1, "kind": "oracle",
               "sample": f"{n_done} of {n_prob} problems ({obs_done} observations), {BATCH_ITERS} LM trials "
                         f"each, {dt:.1f} s; rate scaled to the mean problem size"}
    line = {"metric": METRIC, "value": value, "unit": "problem LM iters/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": "batch512" if n_prob == BATCH_N else f"batch{n_prob}", "problems": n_prob,
                       "lm_iters_per_problem": BATCH_ITERS,
                       "cameras": bt.C, "points": bt.P, "observations": O,
                       "pcg": f"block-Jacobi, maxiter {PCG_MAXITER}, tol {PCG_TOL}",
                       "pcg_iters_mean": pcg_total / max(1, n_prob * BATCH_ITERS),
                       "step": "reset + one persistent launch solving every problem for 10 LM trials",
                       "launch": cfg, "l2": "per-problem arrays L2-resident by design; no flush"},
            "gpu_launches": launches, "clocks": clk, "roofline": roofline, "solve_ms": solve_ms,
            "sequential_single_problem": seq, "cpu_baseline": cpu, "e2e": e2e}
    print(json.dumps(line), flush=True)
    bt.close()


# --------------------------------------------------------------------------
# learned: the learned block-Jacobi correction against block-Jacobi
# --------------------------------------------------------------------------

LEARN_PCG_TOL = 1e-5
LEARN_PCG_MAXITER = 500
LEARN_TRIALS = 20


def _timed_trials(prob, trials, stream):
    """Run `trials` LM trials one by one with an event after each; returns
    (seconds after each trial, cost after each trial, PCG iterations)."""
    import torch
    evs = [torch.cuda.Event(enable_timing=True) for _ in range(trials + 1)]
    evs[0].record(stream)
    for i in range(trials):
        prob.solve(1)
        evs[i + 1].record(stream)
    torch.cuda.synchronize()
    st = prob.stats(cap=trials, raise_nonfinite=False)
    t = [evs[0].elapsed_time(e) / 1000.0 for e in evs[1:]]
    cost = [s["cost_trial"] if s["accepted"] else s["cost"] for s in st]
    bad = sum(1 for s in st if not math.isfinite(s["cost_trial"]))
    return t, cost, [s["pcg_iters"] for s in st], bad


def time_to_cost(runs, f_ref, rel=1e-6):
    """Time to a fixed cost: runs maps a name to (cumulative seconds after
    each trial, cost after each trial, PCG iterations per trial, non-finite
    trials).  A run reaches the target at its first trial whose cost is at or
    below (1 + rel) f_ref; a run that never gets there has no time (None),
    however close it ends."""
    out = {}
    for name, (t, cost, pcg, bad) in runs.items():
        hit = next((i for i, c in enumerate(cost) if c <= (1 + rel) * f_ref), None)
        out[name] = {"time_to_cost_s": t[hit] if hit is not None else None,
                     "trials_to_cost": None if hit is None else hit + 1,
                     "pcg_iters_to_cost": None if hit is None else sum(pcg[:hit + 1]), "final_cost": cost[-1],
                     "lowest_cost": min(cost), "ms_per_pcg_iter": 1000.0 * t[-1] / max(1, sum(pcg)),
                     "pcg_iters_per_trial": pcg, "cost_per_trial": cost, "nonfinite_trials": bad}
    return out


def speedup(out, base, other):
    """Ratio of the base run's time to cost to the other's; None unless both
    reached the target."""
    a, b = out[base]["time_to_cost_s"], out[other]["time_to_cost_s"]
    return a / b if a is not None and b is not None and b > 0 else None


def run_learned(args):
    import torch
    import paper_2409_12190_gb300 as ba
    from paper_2409_12190_gb300 import build as bbuild, learned
    rank, world, local = dist_env()
    if rank != 0:
        return
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    bbuild.build()

    def make(scene, prec="f32", tol=1e-4, maxiter=50):
        ci = torch.from_numpy(scene.cam_idx).to(dev)
        pi = torch.from_numpy(scene.pt_idx).to(dev)
        dt = torch.float32 if prec == "f32" else torch.float64
        px = ba.project(torch.tensor(scene.cams_gt, dtype=dt, device=dev), torch.tensor(scene.points_gt, dtype=dt, device=dev),
                        ci, pi) + torch.tensor(scene.noise, dtype=dt, device=dev)
        return ba.Problem(scene.cams_init, scene.points_init, ci, pi, px,
                          ba.Options(precision=prec, pcg_maxiter=maxiter, pcg_tol=tol), device=dev)

    # training set: ring scenes of 500-2,000 cameras (seeds 1000..)
    t0 = time.perf_counter()
    rng = np.random.default_rng(1000)
    samples = []
    for i in range(args.train_scenes):
        C = int(rng.integers(500, 2001))
        sc = scenegen.ring_scene(C, 30 * C, seed=1000 + i, view_p=1.0 / 5.7, name=f"train{i}")
        with make(sc) as pr:
            samples.append(learned.collect(pr, seed=i))
    t_collect = time.perf_counter() - t0
    n_samples = sum(s[0].shape[0] for s in samples)
    trained = []
    for seed in range(args.seeds):
        t0 = time.perf_counter()
        params, hist = learned.train(samples, epochs=100, lr=2e-3, seed=seed)
        torch.cuda.synchronize()
        trained.append((seed, params, hist, time.perf_counter() - t0))
    del samples

    # evaluation on the bench scene: block-Jacobi, then each trained network
    scene = scenegen.config_scene(WORKLOAD)
    stream = torch.cuda.current_stream()

    def evaluate(par):
        with make(scene, tol=LEARN_PCG_TOL, maxiter=LEARN_PCG_MAXITER) as pr:
            pr.set_preconditioner(par)
            pr.solve(1)  # warm-up: captures the trial graph
            pr.set_params(torch.tensor(scene.cams_init, dtype=torch.float32, device=dev),
                          torch.tensor(scene.points_init, dtype=torch.float32, device=dev))
            pr.set_lambda(1e-4)
            pr.stats()
            return _timed_trials(pr, LEARN_TRIALS, stream)

    runs = {"block_jacobi": evaluate(None)}
    for seed, params, _, _ in trained:
        runs[f"learned_seed{seed}"] = evaluate(params)
    # the target is the plain method's own best cost: a learned run must
    # reach what block-Jacobi reaches, to 1e-6 relative
    f_ref = min(runs["block_jacobi"][1])
    out = time_to_cost(runs, f_ref)
    names = [f"learned_seed{sd}" for sd, _, _, _ in trained]
    times = [out[n]["time_to_cost_s"] for n in names]
    reached = [t for t in times if t is not None]
    value = statistics.mean(reached) if reached and len(reached) == len(times) else None
    # the preconditioners' own measure: PCG iterations over the leading
    # trials in which block-Jacobi stays below the iteration cap (later
    # trials all run to the cap, and their steps drift apart by truncation)
    pcg_bj = out["block_jacobi"]["pcg_iters_per_trial"]
    lead = next((i for i, n in enumerate(pcg_bj) if n >= LEARN_PCG_MAXITER), len(pcg_bj))
    lead_iters = {n: sum(out[n]["pcg_iters_per_trial"][:lead]) for n in ["block_jacobi"] + names}
    line = {"metric": METRIC, "value": value, "unit": "s to 1e-6 relative cost", "n_gpus": 1,
            "steps": LEARN_TRIALS, "warmup": 1, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic",
            "config": {"workload": scene.name, "cameras": scene.C, "points": scene.P, "observations": scene.O,
                       "pcg": f"tol {LEARN_PCG_TOL}, maxiter {LEARN_PCG_MAXITER}",
                       "f_ref": f_ref,
                       "f_ref_rule": "block-Jacobi's lowest cost; a learned run has no time if it never reaches it",
                       "training": {"scenes": args.train_scenes, "cameras": "500-2000", "points_per_camera": 30,
                                    "samples": n_samples, "epochs": 100, "collect_s": t_collect,
                                    "seeds": [{"seed": sd, "train_s": ts, "loss_first_last": [h[0], h[-1]]}
                                              for sd, _, h, ts in trained]}},
            "block_jacobi": out["block_jacobi"],
            "learned": {n: out[n] for n in names},
            "time_to_cost_by_seed": dict(zip(names, times)),
            "spread_s": (max(reached) - min(reached)) if reached else None,
            "speedup_by_seed": {n: speedup(out, "block_jacobi", n) for n in names},
            "uncapped_trials": lead,
            "pcg_iters_uncapped": lead_iters,
            "pcg_iters_change_by_seed": {n: lead_iters[n] / max(1, lead_iters["block_jacobi"]) - 1.0
                                         for n in names}}
    print(json.dumps(line), flush=True)


# --------------------------------------------------------------------------
# adjoint: the implicit-function adjoint (ba_backward) on the ba64 scene
# --------------------------------------------------------------------------

def run_adjoint(args):
    import torch
    import paper_2409_12190_gb300 as ba
    from paper_2409_12190_gb300 import build as bbuild
    import oracle as orc
    rank, world, local = dist_env()
    if rank != 0:
        return
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    bbuild.build()
    scene = scenegen.config_scene("ba64")
    ci = torch.from_numpy(scene.cam_idx).to(dev)
    pi = torch.from_numpy(scene.pt_idx).to(dev)
    px = ba.project(torch.tensor(scene.cams_gt, device=dev), torch.tensor(scene.points_gt, device=dev), ci, pi) + \
        torch.tensor(scene.noise, device=dev)
    fixed = np.zeros((scene.C, 9), dtype=bool)
    fixed[0, :] = True
    fixed[1, 3] = True
    prob = ba.Problem(scene.cams_init, scene.points_init, ci, pi, px,
                      ba.Options(precision="f64", pcg_maxiter=600, pcg_tol=1e-12, lambda0=1e-6), device=dev)
    prob.set_fixed(torch.from_numpy(fixed))
    stream = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    prob.solve(30)
    e1.record(stream)
    torch.cuda.synchronize()
    fwd_ms = e0.elapsed_time(e1)
    cams, pts = prob.params()
    tgt = torch.tensor(scene.cams_gt[:, 3:6], device=dev)
    g = torch.zeros_like(cams)
    g[:, 3:6] = 2.0 * (cams[:, 3:6] - tgt)
    lam, maxiter, tol = 1e-8, 2000, 1e-12
    for _ in range(args.warmup):
        prob.backward(g, None, lam=lam, maxiter=maxiter, tol=tol)
    torch.cuda.synchronize()
    e0.record(stream)
    for _ in range(args.steps):
        dpix, dc0, _, its, rel = prob.backward(g, None, lam=lam, maxiter=maxiter, tol=tol)
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / args.steps
    # the oracle's adjoint at the GPU's converged parameters, timed on the host
    t0 = time.perf_counter()
    ref_pix, ref_c0, _, _ = orc.adjoint_schur(cams.cpu().numpy(), pts.cpu().numpy(), scene.cam_idx, scene.pt_idx,
                                              px.cpu().numpy(), g.cpu().numpy(), np.zeros((scene.P, 3)), fixed,
                                              0.0, lam)
    t_orc = time.perf_counter() - t0
    err = float(np.max(np.abs(dpix.cpu().numpy() - ref_pix)) / np.max(np.abs(ref_pix)))
    line = {"metric": METRIC, "value": 1000.0 / ms, "unit": "adjoint solves/s", "n_gpus": 1, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": "ba64", "cameras": scene.C, "points": scene.P, "observations": scene.O,
                       "loss": "sum over cameras of |t - t_gt|^2", "gauge": "camera 0 and t_x of camera 1 frozen",
                       "forward": "30 LM trials, FP64, PCG tol 1e-12", "adjoint_pcg": f"tol {tol}, maxiter {maxiter}",
                       "step": "one ba_backward: linearisation, Schur/PCG solve of H v = dL/dtheta, dL/dpixels"},
            "forward_ms_30_trials": fwd_ms, "adjoint_pcg_iters": its, "adjoint_rel_res": rel,
            "max_rel_err_vs_oracle_dense_adjoint": err,
            "cpu_baseline": {"value": 1.0 / t_orc, "unit": "adjoint solves/s", "cores": 1, "kind": "oracle",
                             "sample": f"the whole ba64 adjoint (explicit Schur, dense Cholesky), {t_orc:.1f} s"}}
    print(json.dumps(line), flush=True)


# --------------------------------------------------------------------------
# direct: the direct solver of the reduced camera system (Sec. IV-C) on ba250
# --------------------------------------------------------------------------

DIRECT_STOP = 1e-9            # converged: an accepted trial gains less than this (relative)
DIRECT_MAX_TRIALS = 400


def _ba_solve_to_convergence(prob, stream, target=None):
    """LM trials one at a time until an accepted trial gains less than
    DIRECT_STOP (relative), or, with a target, until the cost reaches it;
    at most DIRECT_MAX_TRIALS.  Returns (seconds, trials, final cost)."""
    import torch
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    trials = 0
    while trials < DIRECT_MAX_TRIALS:
        prob.solve(1)
        trials += 1
        st = prob.stats(cap=1)[-1]
        F = st["cost_trial"] if st["accepted"] else st["cost"]
        if target is not None:
            if F <= target:
                break
        elif st["accepted"] and st["cost"] - st["cost_trial"] <= DIRECT_STOP * st["cost"]:
            break
    e1.record(stream)
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / 1000.0, trials, prob.scalars()[0]


def run_direct(args):
    """ba250 (250 cameras, 60,000 points, ~480k observations, Huber) in FP64
    with the direct solver: S = U* - W V*^-1 W^T formed explicitly (9C =
    2,250 unknowns), a tiled Cholesky and both triangular solves in one
    task-graph launch.  F_ref is the
    direct solver's converged cost; the line times LM to (1 + 1e-6) F_ref
    with the direct solver and, beside it, with the PCG of the headline
    settings (block-Jacobi, tol 1e-4, maxiter 50)."""
    import torch
    import paper_2409_12190_gb300 as ba
    from paper_2409_12190_gb300 import build as bbuild
    rank, world, local = dist_env()
    if rank != 0:
        return
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    bbuild.build()
    scene = scenegen.config_scene("ba250")
    ci = torch.from_numpy(scene.cam_idx).to(dev)
    pi = torch.from_numpy(scene.pt_idx).to(dev)
    px = ba.project(torch.tensor(scene.cams_gt, device=dev), torch.tensor(scene.points_gt, device=dev), ci, pi) + \
        torch.tensor(scene.noise, device=dev)
    stream = torch.cuda.current_stream()
    opts = {sv: ba.Options(precision="f64", solver=sv, huber_delta=scene.huber_delta, pcg_maxiter=PCG_MAXITER,
                           pcg_tol=PCG_TOL) for sv in ("cholesky", "pcg")}
    if args.no_time_to_cost:
        # per-trial time only: W warm-up trials, then K timed (a short run,
        # e.g. for a profiler's launch list)
        per_trial = {}
        for solver in ("cholesky", "pcg"):
            with ba.Problem(scene.cams_init, scene.points_init, ci, pi, px, opts[solver], device=dev) as prob:
                prob.solve(args.warmup)
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                prob.solve(args.steps)
                e1.record(stream)
                torch.cuda.synchronize()
                per_trial[solver] = e0.elapsed_time(e1) / args.steps
        print(json.dumps({"metric": "direct solver: ms per LM trial, ba250 FP64", "value": per_trial["cholesky"],
                          "unit": "ms", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
                          "ms_per_step": per_trial["cholesky"], "higher_is_better": False, "scaling": "weak",
                          "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                          "config": {"workload": "ba250", "cameras": scene.C, "points": scene.P,
                                     "observations": scene.O},
                          "pcg_ms_per_trial": per_trial["pcg"]}), flush=True)
        return
    # F_ref: the direct solver run until an accepted trial gains less than
    # DIRECT_STOP (this run also warms up)
    with ba.Problem(scene.cams_init, scene.points_init, ci, pi, px, opts["cholesky"], device=dev) as prob:
        ref_secs, ref_trials, f_ref = _ba_solve_to_convergence(prob, stream)
    target = f_ref * (1.0 + 1e-6)
    out = {}
    for solver in ("cholesky", "pcg"):
        for rep in range(2):  # the first run warms up
            with ba.Problem(scene.cams_init, scene.points_init, ci, pi, px, opts[solver], device=dev) as prob:
                F0 = prob.scalars()[0]
                secs, trials, F = _ba_solve_to_convergence(prob, stream, target)
                per = prob.stats(cap=DIRECT_MAX_TRIALS)
        out[solver] = {"time_to_cost_s": secs, "trials": trials, "ms_per_trial": 1000.0 * secs / trials,
                       "initial_cost": F0, "final_cost": F, "accepted": sum(1 for t in per if t["accepted"]),
                       "pcg_iters_total": sum(t["pcg_iters"] for t in per)}
    ch = out["cholesky"]
    line = {"metric": "direct solver: time to (1 + 1e-6) F_ref (s), ba250 FP64", "value": ch["time_to_cost_s"],
            "unit": "s",
            "n_gpus": 1, "steps": ch["trials"], "warmup": 1, "ms_per_step": ch["ms_per_trial"],
            "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": "ba250", "cameras": scene.C, "points": scene.P, "observations": scene.O,
                       "loss": f"Huber, delta {scene.huber_delta} px",
                       "solver": "explicit S (9C = %d), tiled Cholesky and triangular solves in one launch"
                                 % (9 * scene.C),
                       "f_ref": {"f_ref": f_ref, "trials": ref_trials, "seconds": ref_secs,
                                 "rule": f"the direct solver until an accepted trial gains < {DIRECT_STOP} relative "
                                         f"(at most {DIRECT_MAX_TRIALS} trials)"},
                       "l2": "S (41 MB) stays in L2; the per-observation passes stream more than L2"},
            "solvers": out,
            "pcg_time_to_same_cost_s": out["pcg"]["time_to_cost_s"]}
    if not args.no_cpu_baseline:
        # one LM trial of the oracle with its direct solve (explicit Schur,
        # dense Cholesky), one host thread's BLAS as it stands
        import oracle as orc
        pix = px.cpu().numpy()
        t0 = time.perf_counter()
        orc.lm(scene.cams_init, scene.points_init, scene.cam_idx, scene.pt_idx, pix, 1,
               orc.LMOptions(solver="cholesky", huber_delta=scene.huber_delta))
        t_orc = time.perf_counter() - t0
        line["cpu_baseline"] = {"value": 1.0 / t_orc, "unit": "LM trials/s", "cores": 1, "kind": "oracle",
                                "sample": f"one whole ba250 LM trial with the oracle's direct solve, {t_orc:.1f} s",
                                "gpu_trials_per_s": 1000.0 / ch["ms_per_trial"]}
    print(json.dumps(line), flush=True)


# --------------------------------------------------------------------------
# pgo: pose-graph optimisation (Sec. IV-D) on the paper's PGO graph sizes
# --------------------------------------------------------------------------

PGO_GRAPHS = ("sphere2500", "garage1661")
PGO_PCG = (2000, 1e-6)        # PCG maxiter, tol per LM trial
PGO_STOP = 1e-9               # converged: an accepted trial gains less than this (relative)
PGO_MAX_TRIALS = 100


def pgo_flops_per_iteration(N, E):
    """FP64 flops of one PCG iteration on the pose graph: the product (each
    edge's B (x_i - x_j) at both ends: 2 x (36 FMA + 6 subtractions)), the
    damping term, the 6 x 6 block-Jacobi product per node, and the vector
    updates and three dot products."""
    return 156 * E + N * (6 + 72 + 4 * 6 + 2 * 6 + 3 * 2 * 6)


def _pgo_solve_to_convergence(pg, stream):
    """LM trials one at a time until an accepted trial gains less than
    PGO_STOP (relative) or PGO_MAX_TRIALS; returns (seconds, trials, stats)."""
    import torch
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    trials = 0
    while trials < PGO_MAX_TRIALS:
        pg.solve(1)
        trials += 1
        st = pg.stats(cap=1)[-1]
        if st["accepted"] and st["cost"] - st["cost_trial"] <= PGO_STOP * st["cost"]:
            break
    e1.record(stream)
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / 1000.0, trials, pg.stats(cap=PGO_MAX_TRIALS)


def _pgo_oracle_trial(which):
    """One LM trial of the oracle (PCG with the bench's settings) on the graph,
    seconds; spawned so that its BLAS threads are its own."""
    import oracle as orc
    from oracle import pgo as opgo
    g = scenegen.pose_graph_config(which)
    Ts, Tms, infos, _ = opgo.graph_inputs(g)
    fixed = np.zeros(g.N, bool)
    fixed[0] = True
    t0 = time.perf_counter()
    opgo.lm(Ts, g.ei, g.ej, Tms, infos, 1, orc.LMOptions(solver="pcg", pcg_maxiter=PGO_PCG[0], pcg_tol=PGO_PCG[1]),
            fixed)
    return time.perf_counter() - t0


def run_pgo(args):
    import torch
    import paper_2409_12190_gb300 as ba
    from paper_2409_12190_gb300 import build as bbuild
    from paper_2409_12190_gb300.pgo import PoseGraph, synthesize
    rank, world, local = dist_env()
    if rank != 0:
        return
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    bbuild.build()
    stream = torch.cuda.current_stream()
    graphs = {}
    clocks = ClockSampler(local)
    time.sleep(0.3)
    n0 = ba.kernel_launch_count()
    for which in PGO_GRAPHS:
        g = scenegen.pose_graph_config(which)
        meas, init = synthesize(g.poses_gt, g.ei, g.ej, g.noise, g.drift, device=dev)
        out = {"nodes": g.N, "edges": g.E}
        for solver in ("pcg", "cholesky"):
            opts = ba.Options(precision="f64", solver=solver, pcg_maxiter=PGO_PCG[0], pcg_tol=PGO_PCG[1])
            with PoseGraph(init, g.ei, g.ej, meas, g.info, options=opts, device=dev) as warm:
                warm.solve(2)
            with PoseGraph(init, g.ei, g.ej, meas, g.info, options=opts, device=dev) as pg:
                F0, _ = pg.scalars()
                secs, trials, st = _pgo_solve_to_convergence(pg, stream)
                F, _ = pg.scalars()
                rec = {"time_s": secs, "trials": trials, "ms_per_trial": 1000.0 * secs / trials,
                       "initial_cost": F0, "final_cost": F, "chi2": 2.0 * F,
                       "pcg_iters_total": int(sum(t["pcg_iters"] for t in st)),
                       "accepted": int(sum(t["accepted"] for t in st))}
                if solver == "pcg":
                    # PCG iteration time: K iterations of the damped solve at the
                    # converged poses, less the same call with no iteration
                    pg.damped_solve(1e-6, 0, 0.0)
                    times = {}
                    for K in (0, 500):
                        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                        e0.record(stream)
                        for _ in range(3):
                            pg.damped_solve(1e-6, K, 0.0)
                        e1.record(stream)
                        torch.cuda.synchronize()
                        times[K] = e0.elapsed_time(e1) / 3.0
                    it_us = 1000.0 * (times[500] - times[0]) / 500.0
                    fl = pgo_flops_per_iteration(g.N, g.E)
                    rec["pcg_iteration_us"] = it_us
                    rec["pcg_iteration_tflops"] = fl / (it_us * 1e-6) / 1e12
            out[solver] = rec
        # the same graph with its poses renumbered at random: the Cholesky
        # solver then factors in its reverse Cuthill-McKee order
        gr = scenegen.relabel(g, seed=7)
        meas_r, init_r = synthesize(gr.poses_gt, gr.ei, gr.ej, gr.noise, gr.drift, device=dev)
        opts = ba.Options(precision="f64", solver="cholesky", pcg_maxiter=PGO_PCG[0], pcg_tol=PGO_PCG[1])
        gauge = int(scenegen.relabel_perm(g.N, seed=7)[0])  # the renumbered pose 0
        with PoseGraph(init_r, gr.ei, gr.ej, meas_r, gr.info, fixed=(gauge,), options=opts, device=dev) as pg:
            secs, trials, st = _pgo_solve_to_convergence(pg, stream)
            F, _ = pg.scalars()
            out["cholesky_relabelled"] = {"time_s": secs, "trials": trials, "ms_per_trial": 1000.0 * secs / trials,
                                          "final_cost": F, "chi2": 2.0 * F}
        out["final_cost_rel_diff_pcg_vs_cholesky"] = abs(out["pcg"]["final_cost"] - out["cholesky"]["final_cost"]) / \
            out["cholesky"]["final_cost"]
        graphs[which] = out
    launches = ba.kernel_launch_count() - n0
    clk = clocks.stop()
    peaks_d = measured_peaks_fp64(dev)
    head = graphs[PGO_GRAPHS[0]]
    fl = pgo_flops_per_iteration(head["nodes"], head["edges"])
    roof = {"bound": "alu", "kernel": "k_pgo_pcg (one PCG iteration)", "achieved": head["pcg"]["pcg_iteration_tflops"],
            "peak": peaks_d, "unit": "TFLOP/s", "frac": head["pcg"]["pcg_iteration_tflops"] / peaks_d,
            "flops_per_iteration": fl, "peak_source": "measured (ba_measure_fma_peak, FP64)", "traffic": None,
            "note": "the graph's arrays (B: 288 B per edge) stay in L2; the iteration is bound by FP64 issue and "
                    "its two grid exchanges"}
    cpu = None
    if not args.no_cpu_baseline:
        import multiprocessing as mp
        with mp.get_context("spawn").Pool(1) as pool:
            t_or = pool.apply(_pgo_oracle_trial, ("garage1661",))
        gpu_trial_s = graphs["garage1661"]["pcg"]["ms_per_trial"] / 1000.0
        cpu = {"value": 1.0 / t_or, "unit": "LM trials/s", "cores": 1, "kind": "oracle",
               "sample": f"one LM trial of the oracle on garage1661 (PCG maxiter {PGO_PCG[0]}, tol {PGO_PCG[1]}), "
                         f"{t_or:.1f} s", "gpu_trials_per_s_same_graph": 1.0 / gpu_trial_s}
    line = {"metric": "PGO time to converged cost (s), sphere2500 with PCG", "value": head["pcg"]["time_s"],
            "unit": "s", "n_gpus": 1, "steps": head["pcg"]["trials"], "warmup": 2,
            "ms_per_step": head["pcg"]["ms_per_trial"], "higher_is_better": False, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": "pgo", "graphs": {k: f"{v['nodes']} nodes, {v['edges']} edges"
                                                     for k, v in graphs.items()},
                       "pcg": f"block-Jacobi 6x6, maxiter {PGO_PCG[0]}, tol {PGO_PCG[1]}",
                       "stop": f"first accepted trial gaining < {PGO_STOP} relative, at most {PGO_MAX_TRIALS} trials",
                       "gauge": "pose 0 fixed", "l2": "the whole graph fits in L2 (problem sizes of the paper's PGO "
                                                     "benchmark files)"},
            "graphs": graphs, "gpu_launches": launches, "clocks": clk, "roofline": roof, "cpu_baseline": cpu}
    print(json.dumps(line), flush=True)


def measured_peaks_fp64(dev):
    import paper_2409_12190_gb300 as ba
    return ba.measure_fma_peak("f64")


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
    elif args.workload == "batch512":
        run_batch(args)
    elif args.workload == "learned":
        run_learned(args)
    elif args.workload == "adjoint":
        run_adjoint(args)
    elif args.workload == "pgo":
        run_pgo(args)
    elif args.workload == "direct":
        run_direct(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
