#!/usr/bin/env python
"""Benchmark: EM fit of a K=512 full-covariance GMM to a synthetic 640x480 depth frame.

One step = one full ``gira_gmm_fit`` (pack, k-means++ seeding, Lloyd, one-hot
M-step, up to 30 EM iterations with tol 1e-4 on the mean log-likelihood, final
log-likelihood) on a ~276k-point frame already resident in HBM.  Prints one
JSON line (rank 0).

value       EM point-component-iterations per second, whole job:
            sum over ranks of N*K*iters_done / max over ranks of summed step time
            (k-means++/Lloyd time is inside the step time, its work is not counted)
roofline    the fused E-step/statistics kernel against the FP32-pipe roofline
            (23 FP32-pipe operations per point-component-iteration)
e2e         the same metric through the C ABI with host buffers (pinned points in,
            model and log-likelihood trace out, copies inside the timed region)
cpu_baseline  the FP64 oracle on the host: EM iterations of the frame over every
            core (OpenMP), and the single-threaded oracle on one core

``--impl reference`` times the all-core oracle alone (rank 0; the baseline arm).
Multi-GPU (torchrun): every rank fits its own frame (weak scaling, no collective
on the data path; barriers only bracket the timed region).
"""
from __future__ import annotations

import argparse
import datetime
import hashlib
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "EM point-component-iters/sec and ms per 300k-pt K=512 frame; % FP32/SFU roofline"
UNIT = "point-component-iters/s"
K, ITERS, TOL, REG, SEED, LLOYD = 512, 30, 1e-4, 1e-6, 0, 10
FP32_OPS_PER_UNIT = 23          # algorithmic FP32-pipe operations per (point, component, iteration)
# the point-stationary E-step's FP32-pipe lane operations per (component pair, point) it evaluates:
# reach-listed pairs (q' of both components, exp2 argument, running total) and live pairs
# (q' again, responsibilities, 10 statistics of both components)
PT_OPS_NEAR, PT_OPS_LIVE, PT_WARP_POINTS = 26, 54, 128
FP32_LANES_PER_SM = 128
L2_FLUSH_BYTES = 256 << 20      # > 129 MB L2
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "estep_frame276k_k512.traffic.json")
EM_SOURCE = os.path.join(ROOT, "paper_2307_00071_gb300", "csrc", "em_kernels.cu")


def parse():
    p = argparse.ArgumentParser()
    p.add_argument("--gpus", type=int, default=1)
    p.add_argument("--steps", type=int, default=30)
    p.add_argument("--warmup", type=int, default=3)
    p.add_argument("--impl", choices=["gira", "reference"], default="gira")
    p.add_argument("--no-cpu-baseline", action="store_true")
    p.add_argument("--no-extras", action="store_true", help="skip the measurements of the paths beyond the fit")
    return p.parse_args()


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def aggregate(local, world):
    """Whole-job figures from per-rank (units, seconds, e2e_units, e2e_seconds).

    Units add over ranks (each rank fits its own frame); time is the slowest
    rank's.  Uses torch.distributed when world > 1 (any backend).
    """
    import torch
    vals = torch.tensor(local, dtype=torch.float64)
    if world > 1:
        import torch.distributed as dist
        if dist.get_backend() == "nccl":
            vals = vals.cuda()
        gathered = [torch.zeros_like(vals) for _ in range(world)]
        dist.all_gather(gathered, vals)
        g = torch.stack(gathered).cpu().numpy()
    else:
        g = vals.reshape(1, -1).cpu().numpy()
    return float(g[:, 0].sum()), float(g[:, 1].max()), float(g[:, 2].sum()), float(g[:, 3].max())


def workload_config(n_points):
    return {"workload": f"synthetic 640x480 depth frame (procedural scene, 5 mm noise, 10% dropout) -> "
                        f"{n_points} points; K={K} full-covariance GMM; k-means++ + {LLOYD} Lloyd + up to "
                        f"{ITERS} EM iters, tol {TOL:g}",
            "N": int(n_points), "K": K, "iters": ITERS, "tol": TOL, "reg_covar": REG,
            "l2": "flushed between steps (256 MB write); frame (4.4 MB) is L2-resident within a fit"}


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            d = json.load(f)
        return float(d.get("sm_max_mhz", 2070.0)), "MEASURED_PEAKS.json sm_max_mhz"
    return 2070.0, "fallback 2070 MHz"


def source_hash():
    with open(EM_SOURCE, "rb") as f:
        return hashlib.sha256(f.read()).hexdigest()[:16]


def traffic_per_launch():
    """DRAM bytes per E-step launch from the committed ncu capture, if the kernel is unchanged."""
    try:
        with open(TRAFFIC_FILE) as f:
            d = json.load(f)
    except (OSError, ValueError):
        return None
    if d.get("em_kernels_sha256_16") != source_hash():
        return None
    return d.get("dram_bytes_per_launch")


class ClockSampler:
    """nvidia-smi SM clock / throttle sampling; started before the warm-up (the
    tool takes a while to start), only samples inside [mark_start, mark_end]
    are summarised."""

    def __init__(self, index=0, period_ms=25):
        self.path = tempfile.mktemp(suffix=".csv")
        self.t0 = self.t1 = None
        q = ("timestamp,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(index), f"--query-gpu={q}",
                                          "--format=csv,noheader,nounits", "-lms", str(period_ms)],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def mark_start(self):
        self.t0 = time.time()

    def mark_end(self):
        self.t1 = time.time()

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        self.proc.wait()
        rows = []
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                ts = datetime.datetime.strptime(parts[0], "%Y/%m/%d %H:%M:%S.%f").timestamp()
            except ValueError:
                continue
            if self.t0 is not None and self.t1 is not None and not (self.t0 <= ts <= self.t1):
                continue
            rows.append(parts[1:])
        os.unlink(self.path)
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples inside the timed region"],
                    "samples": 0}
        mhz = [float(r[0]) for r in rows if r[0].replace(".", "").isdigit()]
        mx = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if "Active" in r[4 + i] and "Not" not in r[4 + i]})
        return {"sm_mhz": statistics.median(mhz) if mhz else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


# --------------------------------------------------------------------------- reference arm
def host_cpu():
    """(logical cores, CPU model) of this host."""
    model = None
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.split(":")[0].strip() == "Model name":
                model = line.split(":", 1)[1].strip()
                break
    except (OSError, subprocess.SubprocessError):
        pass
    if model is None:
        try:
            for line in open("/proc/cpuinfo"):
                if line.lower().startswith("model name"):
                    model = line.split(":", 1)[1].strip()
                    break
        except OSError:
            pass
    return os.cpu_count(), model or "unknown"


def oracle_start_model(frame_pts, seed=123):
    """A K-component start for the oracle's timing runs: thin discs (20 cm x 10 cm x 1 cm)
    centred on random frame points, Dirichlet weights.  The oracle's cost does not depend
    on the parameters (it evaluates every point-component pair)."""
    rng = np.random.default_rng(seed)
    m = frame_pts[rng.choice(len(frame_pts), K, replace=False)].astype(np.float64)
    c = np.empty((K, 3, 3))
    for b in range(K):
        q, _ = np.linalg.qr(rng.normal(size=(3, 3)))
        c[b] = q @ np.diag([0.2 ** 2, 0.1 ** 2, 0.01 ** 2]) @ q.T
    return rng.dirichlet(np.ones(K)), m, c


def run_reference(args):
    """The baseline arm: the FP64 oracle over every host core (OpenMP), one EM
    iteration (E-step + M-step) of the full frame per step."""
    rank, world, _ = dist_env()
    if rank != 0:
        return 0
    import oracle
    from paper_2307_00071_gb300 import synth
    frame = synth.depth_frame(seed=1)
    n = len(frame.points)
    w, mu, cov = oracle_start_model(frame.points)
    times = []
    for step in range(args.warmup + args.steps):
        t0 = time.perf_counter()
        r = oracle.em_par(frame.points, w, mu, cov, iters=1, tol=0.0, reg=REG, final=False)
        dt = time.perf_counter() - t0
        w, mu, cov = r["weights"], r["means"], r["covs"]
        if step >= args.warmup:
            times.append(dt)
    tot = sum(times)
    value = n * K * len(times) / tot
    cores, model = host_cpu()
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * tot / len(times),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": workload_config(n),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": oracle.max_threads(), "nproc": cores,
                             "cpu_model": model, "kind": "oracle",
                             "sample": f"one EM iteration (E-step + M-step, binary64, OpenMP over "
                                       f"{oracle.max_threads()} threads) of the full {n}-point frame per step, "
                                       f"K={K}, from a seeded start model"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# --------------------------------------------------------------------------- extras
GRAD_K, GRAD_SCAN = 1024, 100_000
GRAD_FP32_OPS = 32   # per unit, survey conventions: the fit's 23 + z = P'^T y (6) + sum of gamma z (3)


def bench_grad(gira, frame_pts, sms, mhz, reps=20):
    """Differentiable log-likelihood on the registration workload: a K=1024 GMM of
    the frame and a 100k-point scan of it under a rigid offset; one call returns
    L and every gradient (points, pose, twist, logits, means, Cholesky factors)."""
    import torch
    rng = np.random.default_rng(5)
    x = torch.as_tensor(frame_pts, device="cuda")
    fit = gira.gira_gmm_fit(x, GRAD_K, iters=20, tol=1e-4, seed=0, lloyd_iters=10)
    logits = torch.log(fit["weights"])
    chol = torch.linalg.cholesky(fit["covs"].double()).float()
    sub = frame_pts[rng.choice(len(frame_pts), GRAD_SCAN, replace=False)].astype(np.float64)
    th = np.radians(10.0)
    R = np.array([[np.cos(th), -np.sin(th), 0], [np.sin(th), np.cos(th), 0], [0, 0, 1]])
    scan = torch.as_tensor(((sub - 0.1) @ R).astype(np.float32), device="cuda")
    pose = torch.as_tensor(np.concatenate([R.reshape(9), [0.1, 0.1, 0.1]]).astype(np.float32), device="cuda")
    args = (scan, logits, fit["means"], chol, pose)
    for _ in range(3):
        gira.gira_gmm_loglik_grad(*args)
    gira.gira_profile_enable(True)
    gira.gira_profile_read(reset=True)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    ev0.record()
    for _ in range(reps):
        gira.gira_gmm_loglik_grad(*args)
    ev1.record()
    torch.cuda.synchronize()
    prof = gira.gira_profile_read(reset=True)
    gira.gira_profile_enable(False)
    call_s = ev0.elapsed_time(ev1) / 1e3 / reps
    kern_s = prof["estep_ms"] / max(prof["estep_launches"], 1) / 1e3
    units = GRAD_SCAN * GRAD_K
    peak = FP32_LANES_PER_SM * sms * mhz * 1e6 / GRAD_FP32_OPS
    return {"workload": f"L and all gradients: {GRAD_SCAN}-point scan, K={GRAD_K} GMM of the frame, 10 deg + 0.17 m offset",
            "unit": UNIT, "value": units / call_s, "ms_per_call": call_s * 1e3,
            "kernel": prof["estep_kernel"],
            "kernel_ms": kern_s * 1e3, "kernel_units_per_s": units / kern_s if kern_s else None,
            "frac_fp32": (units / kern_s) / peak if kern_s else None,
            "peak_basis": f"{FP32_LANES_PER_SM} lanes x {sms} SMs x {mhz:.0f} MHz / {GRAD_FP32_OPS} FP32 ops per unit"}


BATCH_B, BATCH_ITERS, BATCH_KS = 256, 25, (16, 32, 64, 128, 256, 512)


def batch_workload(seed=7):
    """256 clouds, N log-uniform in [2k, 200k], each drawn from a random K=8 GMM as in
    the small configuration; K per instance drawn from {16, ..., 512}."""
    from paper_2307_00071_gb300 import synth
    rng = np.random.default_rng(seed)
    sizes = np.exp(rng.uniform(np.log(2_000), np.log(200_000), size=BATCH_B)).astype(np.int64)
    ks = rng.choice(BATCH_KS, size=BATCH_B).astype(np.int32)
    clouds = [synth.gmm_cloud(int(n), 8, seed=1000 + i).points for i, n in enumerate(sizes)]
    offsets = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    return np.concatenate(clouds), offsets, ks


def bench_batched(gira):
    """Batched EM (one CUDA graph per call) against a loop of single fits, same
    initial parameters, 25 EM iterations per instance, tol 0."""
    import torch
    pts, offs, ks = batch_workload()
    x = torch.as_tensor(pts, device="cuda")
    init = gira.gira_gmm_fit_batched(x, offs, ks, iters=0, tol=0.0, seed=0, lloyd_iters=10, final_loglik=False)
    w0, m0, c0 = init["weights"], init["means"], init["covs"]
    cks = np.concatenate([[0], np.cumsum(ks)])
    units = float(np.sum((offs[1:] - offs[:-1]) * ks)) * BATCH_ITERS
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def batched():
        return gira.gira_gmm_fit_batched(x, offs, ks, iters=BATCH_ITERS, tol=0.0, init=(w0, m0, c0),
                                         final_loglik=False)

    def loop():
        for i in range(len(ks)):
            sl, cl = slice(int(offs[i]), int(offs[i + 1])), slice(int(cks[i]), int(cks[i + 1]))
            gira.gira_gmm_fit(x[sl], int(ks[i]), iters=BATCH_ITERS, tol=0.0,
                              init=(w0[cl].clone(), m0[cl].clone(), c0[cl].clone()), final_loglik=False)

    def batched_full():
        return gira.gira_gmm_fit_batched(x, offs, ks, iters=BATCH_ITERS, tol=0.0, seed=0, lloyd_iters=10,
                                         final_loglik=False)

    def loop_full():
        for i in range(len(ks)):
            sl = slice(int(offs[i]), int(offs[i + 1]))
            gira.gira_gmm_fit(x[sl], int(ks[i]), iters=BATCH_ITERS, tol=0.0, seed=0, lloyd_iters=10,
                              final_loglik=False)

    out = {}
    for name, fn, reps in (("batched", batched, 3), ("loop", loop, 1), ("batched_full", batched_full, 2),
                           ("loop_full", loop_full, 1)):
        fn()   # warm (first batched call also tunes points per CTA)
        torch.cuda.synchronize()
        ev0.record()
        for _ in range(reps):
            fn()
        ev1.record()
        torch.cuda.synchronize()
        out[name] = ev0.elapsed_time(ev1) / reps
    return {"workload": f"{BATCH_B} clouds, N log-uniform [2k, 200k] (sum {int(offs[-1])}), K in {list(BATCH_KS)}, "
                        f"{BATCH_ITERS} EM iterations from the same k-means init, tol 0",
            "unit": UNIT, "value": units / (out["batched"] / 1e3), "ms_batched": out["batched"],
            "ms_per_instance_loop": out["loop"], "loop_units_per_s": units / (out["loop"] / 1e3),
            "speedup_vs_loop": out["loop"] / out["batched"],
            "with_kinit": {"ms_batched": out["batched_full"], "ms_per_instance_loop": out["loop_full"],
                           "speedup_vs_loop": out["loop_full"] / out["batched_full"]}}


REG_STEPS, REG_SEEDS = 100, (3, 4, 5)


def bench_registration(gira, frame_pts):
    """The differentiable-registration configuration end to end: a K=1024 GMM fitted to
    the frame; a second scan of the same scene (own 5 mm sensor noise and dropout), 100k
    points under a random rigid offset (<= 15 deg, <= 0.5 m); 100 Adam steps on the twist,
    each one call of the fused log-likelihood / adjoint kernel.  Timed per registration."""
    import torch
    from paper_2307_00071_gb300 import autograd as ag, synth
    x = torch.as_tensor(frame_pts, device="cuda")
    fit = gira.gira_gmm_fit(x, GRAD_K, iters=ITERS, tol=TOL, seed=0, lloyd_iters=LLOYD)
    logits = torch.log(fit["weights"])
    chol = torch.linalg.cholesky(fit["covs"].double()).float()
    runs = []
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for seed in REG_SEEDS:
        scan, R_off, t_off = synth.registration_scan(seed=1, offset_seed=seed)
        s = torch.as_tensor(scan, device="cuda")
        ag.register_scan(s, logits, fit["means"], chol, steps=3)   # warm
        torch.cuda.synchronize()
        ev0.record()
        R, t, ll = ag.register_scan(s, logits, fit["means"], chol, steps=REG_STEPS)
        ev1.record()
        torch.cuda.synchronize()
        R, t = R.cpu().numpy(), t.cpu().numpy()
        dR = R @ R_off
        ang = float(np.degrees(np.arccos(np.clip((np.trace(dR) - 1) / 2, -1, 1))))
        off = float(np.degrees(np.arccos(np.clip((np.trace(R_off) - 1) / 2, -1, 1))))
        runs.append({"offset_deg": off, "offset_m": float(np.linalg.norm(t_off)), "ms": ev0.elapsed_time(ev1),
                     "rot_err_deg": ang, "trans_err_m": float(np.linalg.norm(t + R_off.T @ t_off)),
                     "mean_loglik": ll})
    ms = float(np.mean([r["ms"] for r in runs]))
    return {"workload": f"K={GRAD_K} GMM of the frame; second scan of the scene, {GRAD_SCAN} points, random rigid "
                        f"offset <= 15 deg / 0.5 m; {REG_STEPS} Adam steps on the twist (L and its gradient per step)",
            "ms_per_registration": ms, "ms_per_step": ms / REG_STEPS, "runs": runs}


REG_B, REG_N, REG_K = 64, 100_000, 1024


def bench_batched_registrations(gira, frame_pts):
    """64 registrations (100k-point scans of the frame under random poses, one K=1024 GMM of
    the frame each): one batched call (one CUDA graph) against 64 single calls, L and every
    gradient."""
    import torch
    rng = np.random.default_rng(17)
    x = torch.as_tensor(frame_pts, device="cuda")
    fit = gira.gira_gmm_fit(x, REG_K, iters=20, tol=1e-4, seed=0, lloyd_iters=10)
    logits = torch.log(fit["weights"])
    chol = torch.linalg.cholesky(fit["covs"].double()).float()
    scans, poses = [], []
    for _ in range(REG_B):
        sub = frame_pts[rng.choice(len(frame_pts), REG_N, replace=False)].astype(np.float64)
        th = np.radians(rng.uniform(-10, 10))
        R = np.array([[np.cos(th), -np.sin(th), 0], [np.sin(th), np.cos(th), 0], [0, 0, 1]])
        t = rng.uniform(-0.2, 0.2, size=3)
        scans.append(((sub - t) @ R).astype(np.float32))
        poses.append(np.concatenate([R.reshape(9), t]).astype(np.float32))
    S = torch.as_tensor(np.concatenate(scans), device="cuda")
    P = torch.as_tensor(np.stack(poses), device="cuda")
    offs = np.arange(REG_B + 1, dtype=np.int64) * REG_N
    ks = np.full(REG_B, REG_K, np.int32)
    L = logits.repeat(REG_B).contiguous()
    M = fit["means"].repeat(REG_B, 1).contiguous()
    C = chol.repeat(REG_B, 1, 1).contiguous()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def batched():
        gira.gira_gmm_loglik_grad_batched(S, offs, ks, L, M, C, P)

    def loop():
        for i in range(REG_B):
            gira.gira_gmm_loglik_grad(S[i * REG_N:(i + 1) * REG_N], logits, fit["means"], chol, P[i])

    out = {}
    for name, fn, reps in (("batched", batched, 5), ("loop", loop, 2)):
        fn()
        torch.cuda.synchronize()
        ev0.record()
        for _ in range(reps):
            fn()
        ev1.record()
        torch.cuda.synchronize()
        out[name] = ev0.elapsed_time(ev1) / reps
    units = float(REG_B) * REG_N * REG_K
    return {"workload": f"{REG_B} registrations: {REG_N}-point scans of the frame under random poses, "
                        f"K={REG_K} GMM of the frame; L and every gradient",
            "unit": UNIT, "value": units / (out["batched"] / 1e3), "ms_batched": out["batched"],
            "ms_per_instance_loop": out["loop"], "speedup_vs_loop": out["loop"] / out["batched"]}


MAP_FRAMES, MAP_N, MAP_K, MAP_ITERS = 16, 4_000_000, 8192, 20


def bench_large_map(gira):
    """16 depth frames under random poses (yaw, +-10 m), the first 4M points, K = 8192,
    20 EM iterations (the E-step above K = 1024) from means at random points."""
    import torch
    from paper_2307_00071_gb300 import synth
    rng = np.random.default_rng(11)
    parts = []
    for i in range(MAP_FRAMES):
        f = synth.depth_frame(seed=100 + i).points.astype(np.float64)
        th = rng.uniform(0, 2 * np.pi)
        R = np.array([[np.cos(th), -np.sin(th), 0], [np.sin(th), np.cos(th), 0], [0, 0, 1]])
        parts.append(f @ R.T + np.array([rng.uniform(-10, 10), rng.uniform(-10, 10), 0.0]))
    pts = np.concatenate(parts)[:MAP_N].astype(np.float32)
    x = torch.as_tensor(pts, device="cuda")
    idx = rng.choice(len(pts), MAP_K, replace=False)
    w0 = torch.full((MAP_K,), 1.0 / MAP_K, device="cuda")
    m0 = x[torch.as_tensor(idx, device="cuda")].clone()
    c0 = (torch.eye(3, device="cuda") * 0.05 ** 2).expand(MAP_K, 3, 3).contiguous()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    gira.gira_gmm_fit(x, MAP_K, iters=1, tol=0.0, init=(w0.clone(), m0.clone(), c0.clone()), final_loglik=False)
    torch.cuda.synchronize()
    ev0.record()
    r = gira.gira_gmm_fit(x, MAP_K, iters=MAP_ITERS, tol=0.0, init=(w0.clone(), m0.clone(), c0.clone()),
                          final_loglik=False)
    ev1.record()
    torch.cuda.synchronize()
    ms = ev0.elapsed_time(ev1)
    units = float(len(pts)) * MAP_K * r["iters_done"]
    return {"workload": f"{MAP_FRAMES} depth frames under random poses, N={len(pts)}, K={MAP_K}, "
                        f"{MAP_ITERS} EM iterations, tol 0",
            "unit": UNIT, "value": units / (ms / 1e3), "ms": ms, "ms_per_iteration": ms / max(r["iters_done"], 1),
            "trace_first_last": [float(r["trace"][0]), float(r["trace"][-1])]}


D4_K = 512
# per unit, the fewest FP32 operations the 4D step needs: logit P'x + b' and its squares 14,
# sum 1, statistics 20 (gamma, S0, gamma d, S1, S2); the kernel issues 8 more (d = x - mu
# in both passes) and one MUFU ex2
D4_FP32_OPS = 33     # per unit, survey conventions: y 10, q 4, l 1, LSE 2, gamma 1, S0 1, S1 4, S2 10


def bench_d4(gira, frame_pts, sms, mhz, reps=5):
    """The frame with an intensity channel (N x 4: xyz + I, the paper's SOGMM data),
    K = 512, the main fit's settings; plus intensity regression at every point of the
    frame and resampling of a frame-sized cloud from the fitted model."""
    import torch
    from paper_2307_00071_gb300 import synth
    pts4 = np.concatenate([frame_pts, synth.frame_intensity(frame_pts, 1)[:, None]], axis=1)
    x = torch.as_tensor(pts4, device="cuda")
    n = len(pts4)

    def fit():
        return gira.gira_gmm_fit4(x, D4_K, iters=ITERS, tol=TOL, reg_covar=REG, seed=SEED, lloyd_iters=LLOYD)

    for _ in range(2):
        r = fit()
    # phase events on every fit, an event pair per E-step launch on the last one
    # (the other fits keep the EM loop's dependent launches), as in the main line
    gira.gira_profile_enable(True, launches=False)
    gira.gira_profile_read(reset=True)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    ev0.record()
    iters = 0
    for i in range(reps):
        if i == reps - 1:
            gira.gira_profile_enable(True, launches=True)
        r = fit()
        iters += r["iters_done"]
    ev1.record()
    torch.cuda.synchronize()
    prof = gira.gira_profile_read(reset=True)
    gira.gira_profile_enable(False)
    ms = ev0.elapsed_time(ev1) / reps
    kern_s = prof["estep_ms"] / max(prof["estep_launches"], 1) / 1e3
    peak = FP32_LANES_PER_SM * sms * mhz * 1e6 / D4_FP32_OPS
    locs = x[:, :3].contiguous()
    w, m, c = r["weights"], r["means"], r["covs"]
    gira.gira_gmm_conditional4(locs, w, m, c)
    gira.gira_gmm_sample(n, w, m, c, seed=1)
    torch.cuda.synchronize()
    ev0.record()
    for _ in range(reps):
        gira.gira_gmm_conditional4(locs, w, m, c)
    ev1.record()
    torch.cuda.synchronize()
    cond_ms = ev0.elapsed_time(ev1) / reps
    ev0.record()
    for _ in range(reps):
        gira.gira_gmm_sample(n, w, m, c, seed=1)
    ev1.record()
    torch.cuda.synchronize()
    samp_ms = ev0.elapsed_time(ev1) / reps
    return {"workload": f"depth frame with intensity (N={n} x 4), K={D4_K}, tol {TOL}, KInit as the main fit",
            "unit": UNIT, "value": float(n) * D4_K * iters / reps / (ms / 1e3), "ms_per_frame": ms,
            "em_ms_per_frame": prof["em_ms"] / reps, "init_ms_per_frame": prof["init_ms"] / reps,
            "iters_done": r["iters_done"], "final_loglik": r["final_loglik"],
            "kernel": prof["estep_kernel"], "kernel_ms": kern_s * 1e3,
            "kernel_units_per_s": n * D4_K / kern_s if kern_s else None,
            "frac_fp32": (n * D4_K / kern_s) / peak if kern_s else None,
            "peak_basis": f"{FP32_LANES_PER_SM} lanes x {sms} SMs x {mhz:.0f} MHz / {D4_FP32_OPS} FP32 ops per unit of "
                          "the dense step (the kernels skip pairs that are exact zeros)",
            "conditional_ms": cond_ms, "conditional_points_per_s": n / (cond_ms / 1e3),
            "sample_ms": samp_ms, "sample_points_per_s": n / (samp_ms / 1e3)}


GBMS_H = 0.05


def bench_gbms(gira, frame_pts, reps=5):
    """Mode seeking that sets K on the frame with intensity (N x 4), bandwidth 0.05:
    binned seeds, flat-kernel moves to <= 1e-3 h or 300 iterations, merge."""
    import torch
    from paper_2307_00071_gb300 import synth
    pts4 = np.concatenate([frame_pts, synth.frame_intensity(frame_pts, 1)[:, None]], axis=1)
    x = torch.as_tensor(pts4, device="cuda")
    gira.gira_gbms(x, GBMS_H)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    ev0.record()
    for _ in range(reps):
        m, c = gira.gira_gbms(x, GBMS_H)
    ev1.record()
    torch.cuda.synchronize()
    seeds = len(np.unique(np.floor(pts4.astype(np.float64) / GBMS_H + 0.5), axis=0))
    return {"workload": f"frame with intensity (N={len(pts4)} x 4), bandwidth {GBMS_H}, max_iter 300",
            "ms_per_call": ev0.elapsed_time(ev1) / reps, "K": int(len(m)), "seeds": int(seeds),
            "largest_mode_count": int(c[0])}


def bench_size_sweep(gira, frame, reps=5):
    """The paper's smaller image sizes: the frame's pixels at strides 2, 3, 4 (320x240,
    213x160, 160x120), each fitted like the main step (K=512, up to 30 iterations, tol 1e-4)."""
    import torch
    from paper_2307_00071_gb300 import synth
    out = {}
    for step, name in ((2, "320x240"), (3, "213x160"), (4, "160x120")):
        pts = synth.frame_subsampled(frame, step)
        x = torch.as_tensor(pts, device="cuda")
        fit = lambda: gira.gira_gmm_fit(x, K, iters=ITERS, tol=TOL, reg_covar=REG, seed=SEED, lloyd_iters=LLOYD)
        fit()
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        ev0.record()
        iters = 0
        for _ in range(reps):
            iters += fit()["iters_done"]
        ev1.record()
        torch.cuda.synchronize()
        ms = ev0.elapsed_time(ev1) / reps
        out[name] = {"N": len(pts), "ms_per_frame": ms, "iters": iters / reps,
                     "units_per_s": len(pts) * K * iters / reps / (ms / 1e3)}
    return out


PIPE_H = (0.05, 0.08, 0.1, 0.15)


def bench_pipeline(gira, frame_pts, reps=3):
    """The paper's timed pipeline on the frame with intensity (N x 4): mode seeking
    gives K for a bandwidth, then KInit and EM fit K components (tol 1e-4, up to
    30 iterations), one call after the other, timed together."""
    import torch
    from paper_2307_00071_gb300 import synth
    pts4 = np.concatenate([frame_pts, synth.frame_intensity(frame_pts, 1)[:, None]], axis=1)
    x = torch.as_tensor(pts4, device="cuda")
    out = {}
    for h in PIPE_H:
        def run():
            m, _ = gira.gira_gbms(x, h)
            k = min(len(m), gira.MAX_K4)
            r = gira.gira_gmm_fit4(x, k, iters=ITERS, tol=TOL, reg_covar=REG, seed=SEED, lloyd_iters=LLOYD)
            return len(m), k, r
        run()
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        ev0.record()
        for _ in range(reps):
            nm, k, r = run()
        ev1.record()
        torch.cuda.synchronize()
        out[f"h={h}"] = {"modes": nm, "K": k, "iters_done": r["iters_done"],
                         "final_loglik": r["final_loglik"], "ms_total": ev0.elapsed_time(ev1) / reps}
    return {"workload": f"frame with intensity (N={len(pts4)} x 4): mode seeking at bandwidth h, then KInit + EM "
                        f"with K = the number of modes (tol {TOL}, up to {ITERS} iterations)", "runs": out}


FRAMES_B = 8


def bench_frames_batched(gira, reps=3):
    """Throughput mode of the main workload: 8 depth frames (seeds 1-8, ~276k points
    each), K=512, the main fit's settings (k-means++ + 10 Lloyd, up to 30 EM iterations,
    tol 1e-4), as one batched call against 8 single fits; every instance stops on its
    own tolerance."""
    import torch
    from paper_2307_00071_gb300 import synth
    frames = [synth.depth_frame(seed=1 + i).points for i in range(FRAMES_B)]
    offs = np.concatenate([[0], np.cumsum([len(f) for f in frames])]).astype(np.int64)
    x = torch.as_tensor(np.concatenate(frames), device="cuda")
    ks = [K] * FRAMES_B

    def batched():
        return gira.gira_gmm_fit_batched(x, offs, ks, iters=ITERS, tol=TOL, reg_covar=REG, seed=SEED,
                                         lloyd_iters=LLOYD)

    def loop():
        return [gira.gira_gmm_fit(x[int(offs[i]):int(offs[i + 1])], K, iters=ITERS, tol=TOL, reg_covar=REG,
                                  seed=SEED, lloyd_iters=LLOYD) for i in range(FRAMES_B)]

    out = {}
    for name, fn in (("batched", batched), ("loop", loop)):
        fn()
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        ev0.record()
        for _ in range(reps):
            r = fn()
        ev1.record()
        torch.cuda.synchronize()
        out[name] = (ev0.elapsed_time(ev1) / reps, r)
    rb = out["batched"][1]
    units = float(np.sum((offs[1:] - offs[:-1]) * K * rb["iters_done"]))
    return {"workload": f"{FRAMES_B} depth frames ({int(offs[-1])} points), K={K}, KInit + up to {ITERS} EM "
                        f"iterations, tol {TOL}, per-instance stopping",
            "unit": UNIT, "value": units / (out["batched"][0] / 1e3),
            "ms_batched": out["batched"][0], "ms_per_frame_batched": out["batched"][0] / FRAMES_B,
            "ms_loop_of_single_fits": out["loop"][0], "speedup_vs_loop": out["loop"][0] / out["batched"][0],
            "iters_done": [int(v) for v in rb["iters_done"]]}


def bench_small_config(gira, reps=20):
    """The small configuration end to end on both sides: 20,000 points from a K=8 GMM,
    KInit + 20 EM iterations (tol 0): the library's fit on the GPU and the FP64 oracle's
    fit on one host core (a plain reference, not a tuned CPU implementation)."""
    import torch
    import oracle
    from paper_2307_00071_gb300 import synth
    pts = synth.gmm_cloud(20_000, 8, seed=0).points
    x = torch.as_tensor(pts, device="cuda")
    fit = lambda: gira.gira_gmm_fit(x, 8, iters=20, tol=0.0, reg_covar=REG, seed=0, lloyd_iters=LLOYD)
    fit()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    ev0.record()
    for _ in range(reps):
        fit()
    ev1.record()
    torch.cuda.synchronize()
    gpu_ms = ev0.elapsed_time(ev1) / reps
    t0 = time.perf_counter()
    oracle.gmm_fit(pts, 8, iters=20, tol=0.0, reg=REG, seed=0, lloyd_iters=LLOYD)
    cpu_ms = (time.perf_counter() - t0) * 1e3
    return {"workload": "20,000 points from a K=8 GMM, k-means++ + Lloyd + 20 EM iterations, tol 0",
            "gpu_ms_per_fit": gpu_ms, "oracle_ms_per_fit_1_core": cpu_ms, "ratio": cpu_ms / gpu_ms}


# --------------------------------------------------------------------------- gira arm
CPU_ALL_S = 10.0   # whole EM iterations over every host core until this much time has passed
CPU_ONE_ITERS = 1  # single-threaded oracle: one EM iteration of the frame (several seconds)


def cpu_baseline(frame_pts):
    """The FP64 oracle on this host: EM iterations of the full frame over every core
    (OpenMP, deterministic chunked sums), and one iteration on a single core."""
    import oracle
    n = len(frame_pts)
    w, mu, cov = oracle_start_model(frame_pts)
    t0 = time.perf_counter()
    it = 0
    while True:
        r = oracle.em_par(frame_pts, w, mu, cov, iters=1, tol=0.0, reg=REG, final=False)
        w, mu, cov = r["weights"], r["means"], r["covs"]
        it += 1
        dt = time.perf_counter() - t0
        if dt >= CPU_ALL_S or it >= 30:
            break
    t1 = time.perf_counter()
    oracle.em(frame_pts, w, mu, cov, iters=CPU_ONE_ITERS, tol=0.0, reg=REG)
    dt1 = time.perf_counter() - t1
    cores, model = host_cpu()
    threads = oracle.max_threads()
    return {"value": n * K * it / dt, "unit": UNIT, "cores": threads, "nproc": cores, "cpu_model": model,
            "kind": "oracle", "single_core_value": n * K * CPU_ONE_ITERS / dt1,
            "sample": f"{it} EM iterations (E-step + M-step, binary64) of the full {n}-point frame, K={K}, over "
                      f"{threads} OpenMP threads ({dt:.1f} s), from a seeded start model; single core: "
                      f"{CPU_ONE_ITERS} iteration of the single-threaded oracle ({dt1:.1f} s)"}


def run_gira(args):
    import torch
    rank, world, local = dist_env()
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    from paper_2307_00071_gb300 import gira, synth

    def barrier():
        if world > 1:
            import torch.distributed as dist
            dist.barrier()
        torch.cuda.synchronize()

    frame = synth.depth_frame(seed=1 + rank)
    n = len(frame.points)
    pts = torch.as_tensor(frame.points, device="cuda")
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")
    out = dict(weights=torch.empty(K, device="cuda"), means=torch.empty(K, 3, device="cuda"),
               covs=torch.empty(K, 3, 3, device="cuda"))

    def fit(p, **kw):
        return gira.gira_gmm_fit(p, K, iters=ITERS, tol=TOL, reg_covar=REG, seed=SEED, lloyd_iters=LLOYD, **kw)

    clocks = ClockSampler(local)
    for _ in range(args.warmup):
        fit(pts, **out)
    # phase events on every timed fit; an event pair around each E-step launch on
    # the last one (those pairs make the EM loop launch its kernels plainly, so
    # the other fits keep the dependent launches)
    gira.gira_profile_enable(True, launches=False)
    gira.gira_profile_read(reset=True)
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    units, iters_seen = 0, []
    barrier()
    clocks.mark_start()
    for i in range(args.steps):
        if i == args.steps - 1:
            gira.gira_profile_enable(True, launches=True)
        flush.fill_(float(i))
        ev[i][0].record()
        r = fit(pts, **out)
        ev[i][1].record()
        units += n * K * r["iters_done"]
        iters_seen.append(r["iters_done"])
    barrier()
    clocks.mark_end()
    clk = clocks.stop()
    prof = gira.gira_profile_read(reset=True)
    gira.gira_profile_enable(False)
    step_ms = [a.elapsed_time(b) for a, b in ev]
    total_s = sum(step_ms) / 1e3

    # e2e: host buffers through the C ABI, copies inside the timed region
    pinned = torch.empty((n, 3), dtype=torch.float32, pin_memory=True)
    pinned.copy_(torch.as_tensor(frame.points))
    host_out = dict(weights=np.empty(K, np.float32), means=np.empty((K, 3), np.float32),
                    covs=np.empty((K, 3, 3), np.float32))
    fit(pinned, **host_out)   # warm
    e2e_units, e2e_t = 0, 0.0
    for _ in range(max(3, args.steps // 2)):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        r = fit(pinned, **host_out)
        e2e_t += time.perf_counter() - t0
        e2e_units += n * K * r["iters_done"]
    h2d = pinned.numel() * 4
    d2h = sum(a.nbytes for a in host_out.values()) + 8 * ITERS

    # aggregate over ranks
    units_all, t_max, e2e_units_all, e2e_tmax = aggregate([units, total_s, e2e_units, e2e_t], world)

    if rank == 0:
        sms = torch.cuda.get_device_properties(local).multi_processor_count
        mhz, mhz_src = measured_peaks()
        peak_units = FP32_LANES_PER_SM * sms * mhz * 1e6 / FP32_OPS_PER_UNIT
        est_launches = max(prof["estep_launches"], 1)
        avg_estep_s = prof["estep_ms"] / est_launches / 1e3
        dense = n * K / avg_estep_s if avg_estep_s > 0 else 0.0
        # FP32 lane operations the E-step issued per launch: the pairs within reach of a
        # warp's points and the live pairs, counted by the kernel, times their op counts
        near = prof["estep_pairs_near"] / est_launches
        live = prof["estep_pairs_live"] / est_launches
        slots = max(prof["estep_pair_slots"] / est_launches, 1.0)
        ops = PT_WARP_POINTS * (PT_OPS_NEAR * near + PT_OPS_LIVE * live)
        achieved = ops / avg_estep_s if avg_estep_s > 0 else 0.0
        peak_ops = FP32_LANES_PER_SM * sms * mhz * 1e6
        tr = traffic_per_launch()
        line = {
            "metric": METRIC, "value": units_all / t_max, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1e3 * t_max / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": workload_config(n),
            "ms_per_frame": {"with_init": 1e3 * t_max / args.steps,
                             "em_only": prof["em_ms"] / args.steps, "init": prof["init_ms"] / args.steps},
            "em_only_units_per_s": n * K * prof["em_iters"] / (prof["em_ms"] / 1e3) if prof["em_ms"] else None,
            "iters_done": iters_seen,
            "roofline": {"bound": "alu", "achieved": achieved, "peak": peak_ops, "unit": "FP32 lane-op/s",
                         "frac": achieved / peak_ops, "traffic": tr,
                         "kernel": prof["estep_kernel"],
                         "launch_ms": avg_estep_s * 1e3, "launches_timed": prof["estep_launches"],
                         "peak_basis": f"{FP32_LANES_PER_SM} FP32 lanes x {sms} SMs x {mhz:.0f} MHz ({mhz_src})",
                         "achieved_basis": f"per launch {near:.0f} warp-pairs evaluated x {PT_WARP_POINTS} points x "
                                           f"{PT_OPS_NEAR} ops + {live:.0f} live warp-pairs x {PT_WARP_POINTS} "
                                           f"x {PT_OPS_LIVE} ops (counted by the kernel)",
                         "pairs_evaluated_frac": near / slots, "pairs_live_frac": live / slots,
                         "dense_equivalent": {"units_per_s": dense, "peak_units_per_s": peak_units,
                                              "frac": dense / peak_units,
                                              "basis": f"N x K per launch against {FP32_OPS_PER_UNIT} FP32 ops "
                                                       f"per unit at the dense rate"}},
            "e2e": {"value": e2e_units_all / e2e_tmax, "unit": UNIT, "h2d_bytes_per_step": h2d,
                    "d2h_bytes_per_step": d2h},
            "gpu_launches": prof["kernel_launches"],
            "clocks": clk,
        }
        if not args.no_extras:
            extras = (("grad", lambda: bench_grad(gira, frame.points, sms, mhz)),
                      ("registration", lambda: bench_registration(gira, frame.points)),
                      ("batched", lambda: bench_batched(gira)),
                      ("large_map", lambda: bench_large_map(gira)),
                      ("batched_registrations", lambda: bench_batched_registrations(gira, frame.points)),
                      ("xyz_intensity", lambda: bench_d4(gira, frame.points, sms, mhz)),
                      ("gbms", lambda: bench_gbms(gira, frame.points)),
                      ("size_sweep", lambda: bench_size_sweep(gira, frame)),
                      ("sogmm_pipeline", lambda: bench_pipeline(gira, frame.points)),
                      ("frames_batched", lambda: bench_frames_batched(gira)),
                      ("small_config", lambda: bench_small_config(gira)))
            line["extras"] = {}
            for name, fn in extras:   # a failing extra is reported, the headline line still prints
                try:
                    line["extras"][name] = fn()
                except Exception as e:  # noqa: BLE001
                    line["extras"][name] = {"error": f"{type(e).__name__}: {e}"}
        if world == 1 and not args.no_cpu_baseline:
            try:
                line["cpu_baseline"] = cpu_baseline(frame.points)
            except Exception as e:  # noqa: BLE001
                line["cpu_baseline"] = {"error": f"{type(e).__name__}: {e}"}
        print(json.dumps(line), flush=True)
    if world > 1:
        import torch.distributed as dist
        dist.barrier()
        dist.destroy_process_group()
    return 0


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    return run_gira(args)


if __name__ == "__main__":
    sys.exit(main())
