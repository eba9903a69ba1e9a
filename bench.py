#!/usr/bin/env python3
"""Benchmark of the GB300 tree-code force evaluation; prints one JSON line.

Metric: interactions per second (Ginteractions/s) and seconds per force
evaluation on the 16,777,216-particle clumpy workload (64 Hernquist clumps,
a = 0.05, masses log-uniform over one decade, + 20% uniform background;
eps = 1e-3), at the opening angle whose p99 relative force error against an
FP64 direct sum on 4096 sampled particles is 1e-3.  One step = one
leapfrog step of the orbit loop (dt = 1e-4): the whole force evaluation
(root cube, keys, sort, tree, groups, moments, walk + forces) plus the
kick-drift update, the tree rebuilt every step.  Inputs (268 MB of
particles, ~2 GB of tree workspace) exceed the 129 MB L2.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]

With --gpus N > 1 (under torchrun) every rank evaluates its own independent
system (replicas: the force evaluation has no exchange step); value is the
sum of all ranks' interactions over the slowest rank's time.
--impl reference times the FP64 CPU oracle (the same tree method and
criterion) on the host cores instead.
"""
import argparse
import hashlib
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import workloads  # noqa: E402

METRIC = "Ginteractions/s & s per force eval at N=16M, p99 rel-err 1e-3 vs FP64 direct"
UNIT = "Ginteractions/s"
TARGET_P99 = 1e-3
FLOPS_PP = 19       # FP32 flops per particle-particle / monopole particle-cell term (FMA = 2), + 1 rsqrt
FLOPS_PC_QUAD = 54  # FP32 flops per quadrupole particle-cell term (FMA = 2), + 1 rsqrt: bh_pq2, 21 FMA + 9 mul + 3 add
FP32_LANES_PER_SM = 128
SM_MAX_MHZ = 2070.0

# Operating points: the largest theta with p99 <= 1e-3 found by --calibrate on
# a GB300 (re-verified at every run; recalibrated if the check fails).
WORKLOADS = {
    "clumpy16m": dict(kind="clumpy", n=1 << 24, seed=2, eps=1e-3, leaf=16, G=96, order=2, dt=1e-4,
                      theta=0.525, desc="clumpy N=16777216: 64 Hernquist clumps (a=0.05) + 20% uniform "
                                        "background, eps=1e-3, leapfrog dt=1e-4, quadrupole"),
    "clumpy2m": dict(kind="clumpy", n=1 << 21, seed=2, eps=1e-3, leaf=16, G=96, order=2, dt=1e-4,
                     theta=0.525, desc="clumpy N=2097152 (profiling size): 64 Hernquist clumps (a=0.05) + 20% "
                                       "uniform background, eps=1e-3, quadrupole"),
    "plummer1m": dict(kind="plummer", n=1 << 20, seed=1, eps=0.01, leaf=16, G=96, order=2, dt=1e-4,
                      theta=0.6, desc="Plummer N=1048576, eps=0.01, quadrupole"),
    # the learned criterion against theta on fresh sets (seed 4, not in its training data),
    # each at its own p99 = 1e-3 point (theta searched every run)
    "clumpy4m": dict(kind="clumpy", n=1 << 22, seed=4, eps=1e-3, leaf=16, G=96, order=2, dt=1e-4,
                     theta=0.55, calibrate=True,
                     desc="clumpy N=4194304 (seed 4): 64 Hernquist clumps (a=0.05) + 20% uniform background, "
                          "eps=1e-3, quadrupole; learned criterion vs theta at matched p99"),
    "plummer4m": dict(kind="plummer", n=1 << 22, seed=4, eps=0.01, leaf=16, G=96, order=2, dt=1e-4,
                      theta=0.6, calibrate=True,
                      desc="Plummer N=4194304 (seed 4), eps=0.01, quadrupole; learned criterion vs theta "
                           "at matched p99"),
    "batched512": dict(kind="batched", nsys=512, nmin=1024, nmax=65536, seed=3, eps=0.01, theta=0.5, order=1,
                       desc="512 independent Plummer spheres, N log-uniform in [1024, 65536] (seed 3), "
                            "eps=0.01, theta=0.5, monopole; one evaluation of all systems per step"),
}
WEIGHTS = os.path.join(ROOT, "paper_1112_4539_gb300", "weights", "mac_G96_l16_o2.npz")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="clumpy16m", choices=sorted(WORKLOADS))
    ap.add_argument("--theta", type=float, default=None, help="skip the opening-angle search")
    ap.add_argument("--calibrate", action="store_true", help="always search the opening angle")
    ap.add_argument("--order", type=int, default=None)
    ap.add_argument("--group", type=int, default=None)
    ap.add_argument("--leaf", type=int, default=None)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-learned", action="store_true", help="skip the learned-criterion comparison")
    ap.add_argument("--no-extra", action="store_true",
                    help="headline run only: skip the TMA-walk, 512-system, accuracy-sweep and fresh-4M blocks")
    ap.add_argument("--cpu-sample-groups", type=int, default=6000)
    ap.add_argument("--walk", default="group", choices=["group", "particle"],
                    help="group: one warp per particle group; particle: the paper's per-particle walk (Fig. 5)")
    ap.add_argument("--walk-kernel", default="one-warp", choices=["one-warp", "paired", "tma"],
                    help="group walk kernel: one warp walks and evaluates, warp pairs (walker + evaluator), "
                         "or one warp with TMA-staged node and particle tiles")
    ap.add_argument("--curve", default="morton", choices=["morton", "hilbert"],
                    help="particle order (Sec. 5): Morton or Peano-Hilbert keys")
    ap.add_argument("--max-level", type=int, default=10, choices=[10, 21],
                    help="deepest tree level: 10 (30-bit keys) or 21 (63-bit keys)")
    ap.add_argument("--unsoftened-cells", action="store_true",
                    help="particle walk: cells without softening (the Appendix A kernel)")
    ap.add_argument("--symmetrized", action="store_true",
                    help="particle walk with individual softening lengths (log-uniform in [eps/4, 4 eps], seeded) "
                         "and the symmetrized Plummer potential")
    ap.add_argument("--cpu-report", action="store_true",
                    help="FP64 oracle on the host (1 thread and all threads) against the GPU, N=4096 and N=2^20")
    ap.add_argument("--neighbors", action="store_true",
                    help="neighbour search + SPH density on Plummer spheres (no bench line)")
    ap.add_argument("--accuracy-sweep", action="store_true",
                    help="Plummer N=2^20: errors and time over theta x group size x order (no bench line)")
    return ap.parse_args()


def dist_env():
    return (int(os.environ.get("RANK", 0)), int(os.environ.get("LOCAL_RANK", 0)),
            int(os.environ.get("WORLD_SIZE", 1)))


def whole_job(count, ms, world, device):
    """Whole-job totals of replicas (one independent system per rank): the
    sum of the counted units over ranks and the slowest rank's time.  A
    single process returns its own values; otherwise all ranks take part."""
    if world <= 1:
        return float(count), float(ms)
    import torch
    import torch.distributed as dist
    tt = torch.tensor([float(count)], dtype=torch.float64, device=device)
    dist.all_reduce(tt, op=dist.ReduceOp.SUM)
    mm = torch.tensor([float(ms)], dtype=torch.float64, device=device)
    dist.all_reduce(mm, op=dist.ReduceOp.MAX)
    return float(tt.item()), float(mm.item())


# ------------------------------------------------------------------ clocks
class ClockSampler:
    """nvidia-smi samples (SM clock and throttle reasons) while running."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.Q,
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except (OSError, ValueError):
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.15)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.t.join(timeout=2)
        sm, mx, pw, reasons = [], [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
                pw.append(float(f[3]))
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(sm),
                "power_w_max": max(pw) if pw else None}


# --------------------------------------------------------- error judging
def rel_errors(got, ref):
    """Per-target relative errors (acceleration, potential), FP64 on the device."""
    import torch
    g = got.double()
    da = torch.linalg.norm(g[:, :3] - ref[:, :3], dim=1) / torch.linalg.norm(ref[:, :3], dim=1)
    dp = (g[:, 3] - ref[:, 3]).abs() / ref[:, 3].abs()
    return da, dp


def measure_errors(ctx, x, idx_t, ref, theta, eps, acc, walk="group", unsoftened=False, soft=None):
    import torch
    if soft is not None:
        ctx.evaluate_symmetrized(x, soft, theta, acc, unsoftened)
    else:
        ctx.evaluate(x, theta, eps, acc, walk=walk, unsoftened_cells=unsoftened)
    da, dp = rel_errors(acc[idx_t], ref)
    q = torch.quantile(da, torch.tensor([0.5, 0.99], dtype=torch.float64, device=da.device))
    return dict(p50=float(q[0]), p99=float(q[1]), mean=float(da.mean()), max=float(da.max()),
                phi_mean=float(dp.mean()), phi_p99=float(torch.quantile(dp, 0.99)))


def calibrate(ctx, x, idx_t, ref, eps, acc, lo=0.2, hi=1.2, iters=9, walk="group", unsoftened=False, soft=None):
    """Largest theta (bisection) with p99 relative acceleration error <= 1e-3."""
    if measure_errors(ctx, x, idx_t, ref, hi, eps, acc, walk, unsoftened, soft)["p99"] <= TARGET_P99:
        return hi
    for _ in range(iters):
        mid = 0.5 * (lo + hi)
        if measure_errors(ctx, x, idx_t, ref, mid, eps, acc, walk, unsoftened, soft)["p99"] <= TARGET_P99:
            lo = mid
        else:
            hi = mid
    return lo


# ------------------------------------------------------------ CPU oracle
def oracle_throughput(pos, theta, eps, leaf, G, order, n_groups_sample, seed=0, walk="group",
                      unsoftened=False, curve=0, max_level=10, soft=None):
    """FP64 CPU oracle (same walk and criterion) on a bounded sample: the
    tree is built once for all particles (timed, reported apart), then the
    walk of a random sample of groups (group walk) or of n_groups_sample *
    G / 4 targets in 8 Morton-contiguous chunks (particle walk) is timed.
    value = interactions walked / walk time, as measured (the build is not
    in it; s_per_eval_estimate scales the walk to all groups and adds it)."""
    import oracle
    t0 = time.perf_counter()
    b = oracle.Built(pos, leaf, G, theta, order, curve, max_level)
    t_build = time.perf_counter() - t0
    if walk == "particle":
        n = pos.shape[0]
        chunk = max(1, min(n // 8, n_groups_sample * G // 32))
        starts = np.linspace(0, n - chunk, 8).astype(np.int64)
        I, t_walk = 0, 0.0
        eps_s = e2bar = None
        if soft is not None:
            eps_s = np.ascontiguousarray(soft[b.perm])
            e2bar = oracle.cell_softening(b.spos, eps_s, b.tree)
        for s0 in starts:
            t0 = time.perf_counter()
            res = oracle.force_particles(b.spos, b.perm, b.tree, b.mom, eps, t0=int(s0), t1=int(s0 + chunk),
                                         unsoftened_pc=unsoftened, eps_s=eps_s, e2bar=e2bar)
            t_walk += time.perf_counter() - t0
            I += int(res["n_pp"].sum() + res["n_pc"].sum())
        scale = n / (8 * chunk)
        return dict(value=I / t_walk / 1e9, t_build=t_build, t_walk=t_walk, groups=8 * chunk, ng=n,
                    interactions=I, s_per_eval_estimate=t_build + t_walk * scale, cores=oracle.num_threads())
    ng = b.g_first.shape[0]
    S = min(n_groups_sample, ng)
    rng = np.random.default_rng(seed)
    mask = np.zeros(ng, np.uint8)
    mask[rng.choice(ng, S, replace=False)] = 1
    t0 = time.perf_counter()
    res = oracle.force_groups(b.spos, b.perm, b.tree, b.mom, b.g_first, b.g_count, eps, group_mask=mask)
    t_walk = time.perf_counter() - t0
    I = int(res["n_pp"].sum() + res["n_pc"].sum())
    return dict(value=I / t_walk / 1e9, t_build=t_build, t_walk=t_walk, groups=S, ng=ng,
                interactions=I, s_per_eval_estimate=t_build + t_walk * ng / S, cores=oracle.num_threads())


def learned_comparison(bh, ctx, x, idx_t, ref, eps, theta, G, leaf, order, reps=3):
    """The learned criterion against the plain one on the same particles, each
    at its own p99 = 1e-3 operating point: whole force evaluations (build,
    moments, walk) timed with CUDA events."""
    import torch

    from paper_1112_4539_gb300 import learned
    P, fmin, fmax, meta = learned.load(WEIGHTS)
    if (meta.get("G"), meta.get("leaf"), meta.get("order")) != (G, leaf, order):
        return {"skipped": "weights were trained for another configuration"}
    tg = float(meta.get("theta_guard", 1.0))
    tau = learned.calibrate_tau(ctx, x, idx_t, ref, eps, P, fmin, fmax, theta_guard=tg)
    if tau is None:
        bh.bh_mac_set(ctx.h, None)
        return {"skipped": "no tau reaches p99 <= 1e-3"}
    acc = torch.empty_like(x)

    def timed(learned_on, th):
        if learned_on:
            bh.bh_mac_set(ctx.h, P, fmin, fmax, tau, 0.5)
        else:
            bh.bh_mac_set(ctx.h, None)
        ctx.evaluate(x, th, eps, acc)
        errs = learned.p99_error(acc, idx_t, ref)
        torch.cuda.synchronize()
        s0 = ctx.stats()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(reps):
            ctx.evaluate(x, th, eps, acc)
        e1.record()
        torch.cuda.synchronize()
        s1 = ctx.stats()
        inter = (s1["n_pp_total"] - s0["n_pp_total"] + s1["n_pc_total"] - s0["n_pc_total"]) / reps
        return {"ms_per_eval": e0.elapsed_time(e1) / reps, "interactions": inter, "p99": errs}

    plain = timed(False, theta)
    lrn = timed(True, tg)
    bh.bh_mac_set(ctx.h, None)
    return {"weights": os.path.relpath(WEIGHTS, ROOT), "tau": tau, "theta_guard": tg, "theta_fb": 0.5,
            "theta_criterion": dict(plain, theta=theta), "learned_criterion": lrn,
            "speedup": plain["ms_per_eval"] / lrn["ms_per_eval"],
            "interaction_ratio": lrn["interactions"] / plain["interactions"],
            "trained_on": "%d samples, %s" % (meta.get("samples", 0), meta.get("sets"))}


def source_hash():
    h = hashlib.sha256()
    for f in ("bh_walk.cu", "bh_walk.cuh", "bh_internal.cuh", "bh_mlp.cuh"):
        with open(os.path.join(ROOT, "paper_1112_4539_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def stored_traffic(workload):
    """DRAM bytes per walk launch from the committed ncu summary, if it was
    taken on the current walk-kernel source (else None)."""
    p = os.path.join(ROOT, "profiles", "walk_%s_traffic.txt" % workload)
    if not os.path.exists(p):
        return None
    kv = {}
    for line in open(p):
        if ":" in line:
            k, v = line.split(":", 1)
            kv[k.strip()] = v.strip()
    if kv.get("walk_source_sha256_16") != source_hash():
        return None
    try:
        return float(kv["dram_bytes_per_launch_full_size"])
    except (KeyError, ValueError):
        return None


def end_to_end(ctx, pos_np, theta, eps, steps, walk="group", unsoftened=False, world=1, dt=None, soft=None):
    """Whole steps through the public API from and to pinned host memory:
    per step an upload of the particles, the evaluation (Context.evaluate),
    the leapfrog update of the uploaded particles with device-resident
    velocities (Context.kick_drift, when dt is given) and a download of the
    forces.  Two device buffers on each side let the upload of step k+1 and
    the download of step k-1 run on copy streams while step k computes.
    Returns (ms for all steps, interactions counted by the library)."""
    import torch
    comp = torch.cuda.current_stream()
    up, down = torch.cuda.Stream(), torch.cuda.Stream()
    h_pos = torch.from_numpy(pos_np).pin_memory()
    h_acc = [torch.empty_like(h_pos).pin_memory() for _ in range(2)]
    d_pos = [torch.empty(h_pos.shape, dtype=h_pos.dtype, device="cuda") for _ in range(2)]
    d_acc = [torch.empty_like(d_pos[0]) for _ in range(2)]
    d_vel = torch.zeros_like(d_pos[0])
    ev = lambda: torch.cuda.Event(enable_timing=False)

    def run(n):
        loaded, evaluated, fetched = [ev(), ev()], [ev(), ev()], [ev(), ev()]
        for e in evaluated + fetched:
            e.record(comp)  # both buffers start free
        t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        t0.record(up)
        with torch.cuda.stream(up):
            d_pos[0].copy_(h_pos, non_blocking=True)
            loaded[0].record(up)
        for k in range(n):
            b, nb = k % 2, (k + 1) % 2
            if k + 1 < n:
                with torch.cuda.stream(up):
                    up.wait_event(evaluated[nb])   # step k-1 has finished with this buffer
                    d_pos[nb].copy_(h_pos, non_blocking=True)
                    loaded[nb].record(up)
            comp.wait_event(loaded[b])
            comp.wait_event(fetched[b])            # step k-2's forces are out of this buffer
            if soft is not None:
                ctx.evaluate_symmetrized(d_pos[b], soft, theta, d_acc[b], unsoftened)
            else:
                ctx.evaluate(d_pos[b], theta, eps, d_acc[b], walk=walk, unsoftened_cells=unsoftened)
            if dt is not None:
                ctx.kick_drift(d_pos[b], d_vel, d_acc[b], dt, dt)
            evaluated[b].record(comp)
            with torch.cuda.stream(down):
                down.wait_event(evaluated[b])
                h_acc[b].copy_(d_acc[b], non_blocking=True)
                fetched[b].record(down)
        down.wait_event(fetched[(n - 1) % 2])
        t1.record(down)
        torch.cuda.synchronize()
        return t0.elapsed_time(t1)

    run(2)
    if world > 1:
        import torch.distributed as dist
        dist.barrier()
    s0 = ctx.stats()
    ms = run(steps)
    s1 = ctx.stats()
    return ms, float((s1["n_pp_total"] - s0["n_pp_total"]) + (s1["n_pc_total"] - s0["n_pc_total"]))


# ------------------------------------------------------------------- arms
def run_reference(args, W):
    """The reference arm: the FP64 CPU oracle (same tree method, walk and
    criterion) on the host cores.  The oracle's tree of all particles is built
    once before the timed steps (its time is reported in `sample`); each step
    walks a fresh random sample of groups, and value = interactions walked in
    the timed steps / their measured time."""
    rank, _, world = dist_env()
    if rank != 0:
        return 0
    import oracle
    theta = args.theta if args.theta is not None else W["theta"]
    pos = workloads.make(W["kind"], W["n"], W["seed"])
    t0 = time.perf_counter()
    b = oracle.Built(pos, W["leaf"], W["G"], theta, W["order"])
    t_build = time.perf_counter() - t0
    ng = b.g_first.shape[0]
    S = min(args.cpu_sample_groups, ng)
    rng = np.random.default_rng(0)
    inter, times = [], []
    for step in range(args.warmup + args.steps):
        mask = np.zeros(ng, np.uint8)
        mask[rng.choice(ng, S, replace=False)] = 1
        t0 = time.perf_counter()
        res = oracle.force_groups(b.spos, b.perm, b.tree, b.mom, b.g_first, b.g_count, W["eps"],
                                  group_mask=mask)
        tw = time.perf_counter() - t0
        if step >= args.warmup:
            inter.append(int(res["n_pp"].sum() + res["n_pc"].sum()))
            times.append(tw)
    value = sum(inter) / sum(times) / 1e9
    ms_step = 1e3 * sum(times) / len(times)
    sample = ("FP64 oracle group walk, theta=%.4g, %d threads: each step walks %d random groups of the %d "
              "(%.3g interactions, %.2f s); the oracle's tree of all %d particles was built once before the "
              "timed steps (%.2f s, not in the rate); a whole evaluation at this rate: about %.0f s"
              % (theta, oracle.num_threads(), S, ng, float(np.mean(inter)), ms_step * 1e-3, W["n"], t_build,
                 t_build + ms_step * 1e-3 * ng / S))
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_step,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": W["desc"], "n": W["n"], "theta": theta,
                                            "leaf": W["leaf"], "group": W["G"], "order": W["order"],
                                            "step": "walk of %d random groups (bounded sample)" % S},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": oracle.num_threads(),
                             "kind": "oracle", "sample": sample},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


def run_ours(args, W):
    import torch

    import paper_1112_4539_gb300 as bh

    rank, local, world = dist_env()
    if world != args.gpus:
        print("warning: --gpus %d but WORLD_SIZE %d" % (args.gpus, world), file=sys.stderr)
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    bh.lib()

    order = args.order or W["order"]
    G = args.group or W["G"]
    leaf = args.leaf or W["leaf"]
    eps, dt, n = W["eps"], W["dt"], W["n"]
    # each rank evaluates its own independent system
    pos_np = workloads.make(W["kind"], n, W["seed"] + rank)
    x0 = torch.from_numpy(pos_np).to(dev)
    x = x0.clone()
    vel = torch.zeros_like(x)
    acc = torch.empty_like(x)
    curve = bh.CURVE_HILBERT if args.curve == "hilbert" else bh.CURVE_MORTON
    variant = {"paired": bh.WALK_PAIRED, "tma": bh.WALK_TMA}.get(args.walk_kernel, bh.WALK_ONE_WARP)
    ctx = bh.Context(n, device=local, leaf_size=leaf, group_size=G, order=order, curve=curve,
                     max_level=args.max_level, walk_variant=variant)
    stream = torch.cuda.current_stream()

    # individual softening lengths (symmetrized potential; the per-particle walk)
    soft = None
    if args.symmetrized:
        args.walk = "particle"
        soft = torch.from_numpy(workloads.softening_lengths(n, eps, seed=17 + rank)).to(dev)

    # FP64 direct sum on 4096 seeded targets: the error judge
    idx = workloads.sample_targets(n, 4096, seed=101)
    idx_t = torch.from_numpy(idx).to(dev)
    ref = torch.empty((idx.size, 4), dtype=torch.float64, device=dev)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    if soft is not None:
        rc = bh.direct_force_sym(x, soft, x[idx_t].contiguous(), soft[idx_t].contiguous(), idx_t, ref, 64)
    else:
        rc = bh.direct_force(x, x[idx_t].contiguous(), idx_t, eps, ref, 64)
    torch.cuda.synchronize()
    t_judge = time.perf_counter() - t0
    assert rc == 0, rc

    theta = args.theta if args.theta is not None else W["theta"]
    walk, uns = args.walk, args.unsoftened_cells
    errs = measure_errors(ctx, x, idx_t, ref, theta, eps, acc, walk, uns, soft)
    calibrated = False
    if args.theta is None and (args.calibrate or W.get("calibrate") or errs["p99"] > TARGET_P99 or
                               soft is not None):
        theta = calibrate(ctx, x, idx_t, ref, eps, acc, walk=walk, unsoftened=uns, soft=soft)
        errs = measure_errors(ctx, x, idx_t, ref, theta, eps, acc, walk, uns, soft)
        calibrated = True
    st = ctx.status()
    assert st == 0, st

    # kick-drift-kick leapfrog from rest, the two half kicks between forces
    # merged: the first step kicks by dt/2, every later one by dt
    kicks = [0]

    def step(walk_ev=None):
        ctx.build(x)
        if soft is not None:
            ctx.softening(soft)
        ctx.moments(theta)
        if walk_ev is not None:
            walk_ev[0].record(stream)
        if walk == "group":
            ctx.force(eps, acc)
        else:
            ctx.force_particles(eps, acc, uns, individual_softening=soft is not None)
        if walk_ev is not None:
            walk_ev[1].record(stream)
        ctx.kick_drift(x, vel, acc, dt / 2 if kicks[0] == 0 else dt, dt)
        kicks[0] += 1

    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    s0 = ctx.stats()
    clocks = ClockSampler(local)
    clocks.start()
    time.sleep(0.3)
    walk_evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
                for _ in range(args.steps)]
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record(stream)
    for k in range(args.steps):
        step(walk_evs[k])
    e1.record(stream)
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    clk = clocks.stop()
    s1 = ctx.stats()
    assert s1["status"] == 0, s1["status"]
    t_ms = e0.elapsed_time(e1)
    walk_ms = float(np.mean([a.elapsed_time(b) for a, b in walk_evs]))
    n_pp = s1["n_pp_total"] - s0["n_pp_total"]
    n_pc = s1["n_pc_total"] - s0["n_pc_total"]
    inter = n_pp + n_pc
    launches = s1["launches"] - s0["launches"]
    # whole job: sum of interactions over ranks / slowest rank
    tot_inter, max_ms = whole_job(inter, t_ms, world, dev)
    value = tot_inter / (max_ms * 1e-3) / 1e9

    # end to end through the public API with host buffers (pinned), copies timed: every step uploads its
    # particles and downloads its forces; with two buffers per side the copies of neighbouring steps run on
    # their own streams while a step evaluates
    e2e_steps = max(3, args.steps // 2)
    e2e_ms, e2e_inter = end_to_end(ctx, pos_np, theta, eps, e2e_steps, walk, uns, world, dt=dt, soft=soft)
    e2e_inter, e2e_max = whole_job(e2e_inter, e2e_ms, world, dev)
    e2e_value = e2e_inter / (e2e_max * 1e-3) / 1e9
    h_pos_bytes = int(pos_np.size * 4)

    # roofline of the dominant kernel (the walk): FP32 CUDA-core arithmetic
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    steps = args.steps
    pc_flops = FLOPS_PC_QUAD if order >= 2 else FLOPS_PP
    flops_per_launch = (n_pp * FLOPS_PP + n_pc * pc_flops) / steps
    achieved = flops_per_launch / (walk_ms * 1e-3) / 1e12
    peak = sms * FP32_LANES_PER_SM * 2 * SM_MAX_MHZ * 1e6 / 1e12
    roofline = {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
                "traffic": stored_traffic(args.workload) if walk == "group" else None,
                "kernel": "bh_walk_kernel" if walk == "group" else "bh_pwalk_kernel",
                "walk_ms": walk_ms, "walk_share": walk_ms * steps / t_ms,
                "peak_basis": "%d SMs x 128 FP32 lanes x 2 x %.0f MHz (max SM clock)" % (sms, SM_MAX_MHZ),
                "frac_at_measured_clock": (achieved / (peak * clk["sm_mhz"] / SM_MAX_MHZ)) if clk.get("sm_mhz")
                else None,
                "flops_per_interaction": {"pp_and_monopole_pc": FLOPS_PP, "quadrupole_pc": FLOPS_PC_QUAD}}

    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": steps,
            "warmup": args.warmup, "ms_per_step": max_ms / steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": W["desc"], "n": n, "theta": theta, "theta_calibrated": calibrated,
                       "leaf": leaf, "group": G, "order": order, "walk": walk, "walk_kernel": args.walk_kernel,
                       "curve": args.curve,
                       "max_level": args.max_level,
                       "unsoftened_cells": uns if walk == "particle" else None,
                       "softening": ("individual, log-uniform in [eps/4, 4 eps], symmetrized" if soft is not None
                                     else "eps for every particle"),
                       "errors_vs_fp64_direct_4096": errs, "judge_s": t_judge,
                       "interactions_per_step": inter / steps, "pp_per_step": n_pp / steps,
                       "pc_per_step": n_pc / steps, "l2": "inputs larger than L2 (no flush)",
                       "parallelism": "replicas" if world > 1 else "single"},
            "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": h_pos_bytes,
                    "d2h_bytes_per_step": h_pos_bytes, "steps": e2e_steps,
                    "ms_per_step": e2e_max / e2e_steps,
                    "step": "upload particles, build + moments + walk, kick-drift (device velocities), download "
                            "forces; copies overlapped with neighbouring steps (2 buffers)"},
            "gpu_launches": launches, "roofline": roofline, "clocks": clk}

    if not args.no_learned and walk == "group" and os.path.exists(WEIGHTS):
        line["learned_mac"] = learned_comparison(bh, ctx, x0, idx_t, ref, eps, theta, G, leaf, order)
    if args.workload == "clumpy16m" and walk == "group" and world == 1 and not args.no_extra:
        # the other configurations of the benchmark, measured in the same run
        ref_out = torch.empty_like(x0)
        ctx.evaluate(x0, theta, eps, ref_out)
        if args.walk_kernel == "one-warp":
            line["tma_walk"] = tma_block(bh, local, x0, theta, eps, leaf, G, order, ref_out)
            line["tma_walk"]["one_warp_walk_ms"] = walk_ms
        ctx.close()
        ctx = None
        torch.cuda.empty_cache()
        line["batched512"] = batched_block(local)
        line["accuracy_sweep_plummer1m"] = accuracy_sweep(local)
        if not args.no_learned and os.path.exists(WEIGHTS):
            line["learned_fresh4m"] = {name: learned_fresh_block(bh, local, name)
                                       for name in ("clumpy4m", "plummer4m")}

    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cb = oracle_throughput(pos_np, theta, eps, leaf, G, order, args.cpu_sample_groups, walk=walk,
                               unsoftened=uns, curve=curve, max_level=args.max_level,
                               soft=None if soft is None else soft.cpu().numpy())
        unit_s = "groups" if walk == "group" else "targets"
        line["cpu_baseline"] = {"value": cb["value"], "unit": UNIT, "cores": cb["cores"], "kind": "oracle",
                                "sample": "FP64 oracle %s walk on the same particles and theta: %d of %d %s "
                                          "walked in %.2f s (the measured rate); its tree of all particles was "
                                          "built before, in %.2f s (not in the rate); a whole evaluation at this "
                                          "rate: about %.0f s" % (walk, cb["groups"], cb["ng"], unit_s, cb["t_walk"],
                                                                  cb["t_build"], cb["s_per_eval_estimate"])}
    if ctx is not None:
        ctx.close()
    if rank == 0:
        print(json.dumps(line))
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


def batched_measure(W, local, rank, steps, warmup, world=1, dev=None):
    """All systems per step in one graph replay (tuned launch configuration),
    against a loop of per-system evaluations with plain launches, and end to
    end with host copies.  Returns a dict of the measurements."""
    import torch

    import paper_1112_4539_gb300 as bh
    from paper_1112_4539_gb300 import autotune

    dev = dev or torch.device("cuda", local)
    pos_np, offs = workloads.batched_plummer(W["nsys"], W["nmin"], W["nmax"], seed=W["seed"] + rank)
    n, nsys = pos_np.shape[0], W["nsys"]
    x = torch.from_numpy(pos_np).to(dev)
    out = torch.empty_like(x)
    theta, eps, order = W["theta"], W["eps"], W["order"]
    cfg, table = autotune.tune_batched(x, offs, theta, eps, order=order)
    ctx = bh.Context(n, device=local, order=order, max_systems=nsys, **cfg)
    bh._check(bh.bh_batch_layout(ctx.h, offs), "bh_batch_layout")
    l0 = ctx.stats()["launches"]
    graph = bh.BatchedGraph(ctx, x, theta, eps, out)
    per_eval_launches = ctx.stats()["launches"] - l0
    for _ in range(warmup):
        graph.launch()
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    s0 = ctx.stats()
    clocks = ClockSampler(local)
    clocks.start()
    time.sleep(0.3)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    for _ in range(steps):
        graph.launch()
    e1.record()
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    clk = clocks.stop()
    s1 = ctx.stats()
    assert s1["status"] == 0, s1["status"]
    t_ms = e0.elapsed_time(e1)
    n_pp = s1["n_pp_total"] - s0["n_pp_total"]
    n_pc = s1["n_pc_total"] - s0["n_pc_total"]
    inter = float(n_pp + n_pc)
    # the per-system loop of plain launches (same configuration)
    single = bh.Context(int(np.max(np.diff(offs))), device=local, order=order, **cfg)
    xs = [x[offs[k]:offs[k + 1]].contiguous() for k in range(nsys)]
    os_ = [torch.empty_like(v) for v in xs]
    for k in range(nsys):
        single.evaluate(xs[k], theta, eps, os_[k])
    torch.cuda.synchronize()
    f0, f1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    f0.record()
    for k in range(nsys):
        single.evaluate(xs[k], theta, eps, os_[k])
    f1.record()
    torch.cuda.synchronize()
    loop_ms = f0.elapsed_time(f1)
    same = all(torch.equal(os_[k], out[offs[k]:offs[k + 1]]) for k in range(nsys))
    single.close()
    # end to end: host particles in, host forces out, through the graph
    h_pos = torch.from_numpy(pos_np).pin_memory()
    h_out = torch.empty_like(h_pos).pin_memory()
    g0, g1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    g0.record()
    for _ in range(steps):
        x.copy_(h_pos, non_blocking=True)
        graph.launch()
        h_out.copy_(out, non_blocking=True)
    g1.record()
    torch.cuda.synchronize()
    e2e_ms = g0.elapsed_time(g1)
    graph.close()
    ctx.close()
    return dict(t_ms=t_ms, n_pp=n_pp, n_pc=n_pc, inter=inter, n=n, nsys=nsys, cfg=cfg, table=table,
                per_eval_launches=per_eval_launches, loop_ms=loop_ms, same=same, e2e_ms=e2e_ms,
                h2d=int(h_pos.numel() * 4), d2h=int(h_out.numel() * 4), clocks=clk)


def run_batched(args, W):
    """All systems per step in one graph replay; prints the JSON line."""
    import torch

    rank, local, world = dist_env()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    m = batched_measure(W, local, rank, args.steps, args.warmup, world, dev)
    tot_inter, max_ms = whole_job(m["inter"], m["t_ms"], world, dev)
    value = tot_inter / (max_ms * 1e-3) / 1e9
    sms = torch.cuda.get_device_properties(dev).multi_processor_count
    order = W["order"]
    flops = (m["n_pp"] * FLOPS_PP + m["n_pc"] * (FLOPS_PC_QUAD if order >= 2 else FLOPS_PP)) / args.steps
    achieved = flops / (m["t_ms"] / args.steps * 1e-3) / 1e12
    peak = sms * FP32_LANES_PER_SM * 2 * SM_MAX_MHZ * 1e6 / 1e12
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": max_ms / args.steps, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": W["desc"], "n_total": m["n"], "n_systems": m["nsys"], "theta": W["theta"],
                       "order": order, "tuned": m["cfg"], "tuning_table": m["table"],
                       "interactions_per_step": m["inter"] / args.steps,
                       "l2": "inputs 126 MB, tree work arrays > L2 (no flush)"},
            "per_system_loop": {"ms_per_step": m["loop_ms"], "launches": m["nsys"] * 30,
                                "identical_results": m["same"],
                                "speedup_of_graph": m["loop_ms"] / (max_ms / args.steps)},
            "e2e": {"value": m["inter"] / (m["e2e_ms"] * 1e-3) / 1e9, "unit": UNIT, "h2d_bytes_per_step": m["h2d"],
                    "d2h_bytes_per_step": m["d2h"], "ms_per_step": m["e2e_ms"] / args.steps},
            "gpu_launches": m["per_eval_launches"] * args.steps,
            "roofline": {"bound": "alu", "achieved": achieved, "peak": peak, "unit": "TFLOP/s", "frac": achieved / peak,
                         "traffic": None, "kernel": "whole batched evaluation (graph replay)"},
            "clocks": m["clocks"]}
    if rank == 0:
        print(json.dumps(line))
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


def batched_block(local):
    """The 512-system workload as a block of the headline line: one graph
    replay of all systems per evaluation against the per-system loop."""
    W = WORKLOADS["batched512"]
    steps = 10
    m = batched_measure(W, local, 0, steps, 3)
    ms = m["t_ms"] / steps
    return {"workload": W["desc"], "n_total": m["n"], "n_systems": m["nsys"], "tuned": m["cfg"],
            "ms_per_eval": ms, "ginteractions_per_s": m["inter"] / (m["t_ms"] * 1e-3) / 1e9,
            "per_system_loop_ms": m["loop_ms"], "speedup_of_graph": m["loop_ms"] / ms,
            "identical_results": m["same"], "e2e_ms_per_eval": m["e2e_ms"] / steps, "steps": steps,
            "clocks": m["clocks"]}


def learned_fresh_block(bh, local, name):
    """The learned criterion against theta on a fresh 4,194,304-particle set
    (seed 4, not in the training data): theta and tau each bisected to
    p99 = 1e-3 against the FP64 direct judge, then whole evaluations timed."""
    import torch
    W = WORKLOADS[name]
    dev = torch.device("cuda", local)
    pos = workloads.make(W["kind"], W["n"], W["seed"])
    x = torch.from_numpy(pos).to(dev)
    ctx = bh.Context(W["n"], device=local, leaf_size=W["leaf"], group_size=W["G"], order=W["order"])
    idx = workloads.sample_targets(W["n"], 4096, seed=101)
    idx_t = torch.from_numpy(idx).to(dev)
    ref = torch.empty((idx.size, 4), dtype=torch.float64, device=dev)
    assert bh.direct_force(x, x[idx_t].contiguous(), idx_t, W["eps"], ref, 64) == 0
    acc = torch.empty_like(x)
    clocks = ClockSampler(local)
    clocks.start()
    theta = calibrate(ctx, x, idx_t, ref, W["eps"], acc)
    res = learned_comparison(bh, ctx, x, idx_t, ref, W["eps"], theta, W["G"], W["leaf"], W["order"])
    res["clocks"] = clocks.stop()
    res["workload"] = W["desc"]
    ctx.close()
    return res


def tma_block(bh, local, x, theta, eps, leaf, G, order, ref_out):
    """The TMA-staged walk kernel on the headline particles: whole evaluations
    and walk time, and whether its forces carry the one-warp kernel's bits."""
    import torch
    ctx = bh.Context(x.shape[0], device=local, leaf_size=leaf, group_size=G, order=order, walk_variant=bh.WALK_TMA)
    acc = torch.empty_like(x)
    ctx.evaluate(x, theta, eps, acc)
    same = bool(torch.equal(acc, ref_out))
    walk, tot = [], []
    for _ in range(4):
        e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        e0.record()
        ctx.build(x)
        ctx.moments(theta)
        e1.record()
        ctx.force(eps, acc)
        e2.record()
        torch.cuda.synchronize()
        walk.append(e1.elapsed_time(e2))
        tot.append(e0.elapsed_time(e2))
    assert ctx.status() == 0
    ctx.close()
    return {"kernel": "bh_walk_tma_kernel", "ms_per_eval": float(np.median(tot)), "walk_ms": float(np.median(walk)),
            "same_bits_as_one_warp": same,
            "staging": "node walk records per sibling range and leaf-particle batches by cp.async.bulk into "
                       "shared memory (mbarrier completion)"}


def accuracy_sweep(local=0, reps=3):
    """Force errors against the FP64 direct sum (4096 seeded targets) and the
    evaluation time over theta in {0.3, 0.5, 0.75} x group size in {32, 64,
    128, 256} x {monopole, quadrupole} on a Plummer sphere of 2^20 particles
    (seed 1, eps = 0.01, leaf 16).  Returns a dict."""
    import torch

    import paper_1112_4539_gb300 as bh
    bh.lib()
    dev = torch.device("cuda", local)
    n, eps, leaf = 1 << 20, 0.01, 16
    x = torch.from_numpy(workloads.make("plummer", n, 1)).to(dev)
    idx = workloads.sample_targets(n, 4096, seed=101)
    idx_t = torch.from_numpy(idx).to(dev)
    ref = torch.empty((idx.size, 4), dtype=torch.float64, device=dev)
    assert bh.direct_force(x, x[idx_t].contiguous(), idx_t, eps, ref, 64) == 0
    acc = torch.empty_like(x)
    rows = []
    clocks = ClockSampler(local)
    clocks.start()
    for order in (1, 2):
        for G in (32, 64, 128, 256):
            ctx = bh.Context(n, device=local, leaf_size=leaf, group_size=G, order=order)
            for theta in (0.3, 0.5, 0.75):
                errs = measure_errors(ctx, x, idx_t, ref, theta, eps, acc)
                s0 = ctx.stats()
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record()
                for _ in range(reps):
                    ctx.evaluate(x, theta, eps, acc)
                e1.record()
                torch.cuda.synchronize()
                s1 = ctx.stats()
                assert s1["status"] == 0, s1["status"]
                inter = (s1["n_pp_total"] - s0["n_pp_total"] + s1["n_pc_total"] - s0["n_pc_total"]) / reps
                rows.append(dict(order=order, G=G, theta=theta, p50=errs["p50"], p99=errs["p99"],
                                 mean=errs["mean"], max=errs["max"], phi_p99=errs["phi_p99"],
                                 ms_per_eval=e0.elapsed_time(e1) / reps, interactions=inter))
            ctx.close()
    return {"sweep": "Plummer N=1048576 (seed 1), eps=0.01, leaf 16; errors vs FP64 direct on 4096 targets "
                     "(seed 101); time = whole evaluation (build, moments, walk)",
            "rows": rows, "clocks": clocks.stop()}


def run_accuracy_sweep(args):
    """The accuracy sweep alone; prints one JSON object."""
    import torch
    out = accuracy_sweep()
    out["gpu"] = torch.cuda.get_device_name()
    print(json.dumps(out))
    return 0


def run_neighbors(args):
    """Neighbour search and SPH density (the general tree walk of Sec. 4.3)
    on Plummer spheres of 2^20 and 2^24 particles, radii for ~64 neighbours:
    time of tree_build + tree_neighbors per evaluation (CUDA events), pairs
    tested and neighbours found.  Prints one JSON object."""
    import torch

    import paper_1112_4539_gb300 as bh
    bh.lib()
    rows = []
    for n, G, leaf in ((1 << 20, 64, 16), (1 << 20, 32, 16), (1 << 24, 64, 16), (1 << 24, 32, 16)):
        pos = workloads.make("plummer", n, 1)
        x = torch.from_numpy(pos).cuda()
        h = torch.from_numpy(workloads.plummer_search_radii(pos, 64).astype(np.float32)).cuda()
        ctx = bh.Context(n, leaf_size=leaf, group_size=G)
        cnt = torch.empty(n, dtype=torch.int32, device="cuda")
        rho = torch.empty(n, dtype=torch.float32, device="cuda")
        for _ in range(3):
            ctx.build(x)
            bh._check(bh.tree_neighbors(ctx.h, h, cnt, rho), "tree_neighbors")
        torch.cuda.synchronize()
        s0 = ctx.stats()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        reps = 5
        for _ in range(reps):
            ctx.build(x)
            bh.tree_neighbors(ctx.h, h, cnt, rho)
        e1.record()
        torch.cuda.synchronize()
        s1 = ctx.stats()
        assert s1["status"] == 0, s1["status"]
        ms = e0.elapsed_time(e1) / reps
        tested = (s1["n_pp_total"] - s0["n_pp_total"]) / reps
        found = float(cnt.sum().item())
        rows.append(dict(n=n, G=G, leaf=leaf, ms_per_eval=ms, pairs_tested=tested, neighbours=found,
                         mean_neighbours=found / n, pairs_tested_per_s=tested / (ms * 1e-3),
                         particles_per_s=n / (ms * 1e-3), median_neighbours=float(cnt.median().item())))
        ctx.close()
    print(json.dumps({"neighbors": "Plummer spheres (seed 1), radii from the analytic density for ~64 "
                                   "neighbours; time = tree_build + tree_neighbors", "gpu": torch.cuda.get_device_name(),
                      "rows": rows}))
    return 0


def run_cpu_report(args):
    """The FP64 oracle on this machine's host cores against the GPU path, on
    the small Plummer configuration (N=4096, monopole, theta 0.5, leaf 8,
    G 64) and on Plummer N=2^20 (quadrupole, theta 0.6, leaf 16, G 96):
    whole tree evaluations (build + group walk) with one thread and with all
    threads, the FP64 direct sum on the 4096 seeded targets (one thread: a
    512-target subset, scaled), and the GPU's whole evaluation.  Prints one
    JSON object."""
    import os as _os

    import torch

    import oracle
    import paper_1112_4539_gb300 as bh
    bh.lib()
    cores = oracle.num_threads()
    rows = []
    for name, n, theta, order, leaf, G in (("plummer4096", 4096, 0.5, 1, 8, 64),
                                           ("plummer1m", 1 << 20, 0.6, 2, 16, 96)):
        pos = workloads.make("plummer", n, 0 if n == 4096 else 1)
        eps = 0.01
        row = dict(config=name, n=n, theta=theta, order=order, leaf=leaf, G=G)
        for threads in (1, cores):
            oracle.set_threads(threads)
            t0 = time.perf_counter()
            res, _ = oracle.tree_force(pos, theta, eps, n_leaf=leaf, G=G, order=order)
            row["oracle_tree_s_%dthreads" % threads] = time.perf_counter() - t0
            row["interactions"] = int(res["n_pp"].sum() + res["n_pc"].sum())
            idx = workloads.sample_targets(n, 4096, seed=101)
            sub = idx if threads > 1 else idx[:512]
            t0 = time.perf_counter()
            oracle.direct(pos, pos[sub], sub.astype(np.int64), eps)
            row["oracle_direct_4096_s_%dthreads" % threads] = (time.perf_counter() - t0) * idx.size / sub.size
        oracle.set_threads(cores)
        x = torch.from_numpy(pos).cuda()
        ctx = bh.Context(n, leaf_size=leaf, group_size=G, order=order)
        acc = torch.empty_like(x)
        for _ in range(3):
            ctx.evaluate(x, theta, eps, acc)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(10):
            ctx.evaluate(x, theta, eps, acc)
        e1.record()
        torch.cuda.synchronize()
        row["gpu_s"] = e0.elapsed_time(e1) / 10 * 1e-3
        row["gpu_speedup_vs_1thread"] = row["oracle_tree_s_1threads"] / row["gpu_s"]
        row["gpu_speedup_vs_%dthreads" % cores] = row["oracle_tree_s_%dthreads" % cores] / row["gpu_s"]
        ctx.close()
        rows.append(row)
    print(json.dumps({"cpu_report": "FP64 oracle (group walk, same criterion) vs the GPU path; whole evaluations",
                      "host_cores": cores, "nproc": _os.cpu_count(), "gpu": torch.cuda.get_device_name(),
                      "rows": rows}))
    return 0


def main():
    args = parse()
    if args.cpu_report:
        return run_cpu_report(args)
    if args.accuracy_sweep:
        return run_accuracy_sweep(args)
    if args.neighbors:
        return run_neighbors(args)
    W = WORKLOADS[args.workload]
    if args.impl == "reference":
        if W["kind"] == "batched":
            print(json.dumps({"impl": "reference", "unavailable": "the reference arm times the headline workload"}))
            return 0
        return run_reference(args, W)
    if W["kind"] == "batched":
        return run_batched(args, W)
    return run_ours(args, W)


if __name__ == "__main__":
    sys.exit(main())
