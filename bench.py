#!/usr/bin/env python3
"""Benchmark of the SLK-BO hot path on one GB300 (one JSON line on stdout).

A step is one whole solve (kNN graph, sigma, and Algorithm 1's outer loop:
unary term, bound iterations, mode update, energy, until the modes stop
changing) of the default workload: 1e6 points x 128 features on curved
8-dim manifolds, L = 100 clusters with Zipf(1.1) sizes, k = 10 heat-kernel
affinity, bfloat16 tensor-core distance tiles with the exact float32 rerank
(synthetic; see paper_1810_13044_gb300/inputs.py).  The metric is solves/s;
the bound iterations are also reported as N*L*iterations/s.  The same line
carries the 70000 x 784, L = 10, k = 5 MNIST-shaped workload under
"workloads" (its own device and end-to-end figures).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl slk|reference]
                  [--workload manifolds|mnist_like|ms|batched|serving]

--impl reference times the FP64 CPU oracle (the reference arm of this
project) on a bounded sample of the same workload, the sample the main arm's
cpu_baseline also times.  Under torchrun each rank solves its own copy of
the workload (replicas: weak scaling), rank 0 prints.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "SLK N·L·iter/s and solves/s vs plain FP32 GPU at equal labels; p50/p99 latency"
WORKLOADS = {
    # the precision form: curved 8-dim manifolds, Zipf(1.1) cluster sizes, heat affinity
    "manifolds": dict(name="manifolds_1000000x128_L100", N=1_000_000, D=128, L=100, k=10, lam=1.0,
                      affinity="heat", gen="manifolds", sample_rows=32, sample_sub=20000),
    # the MNIST-shaped plain form
    "mnist_like": dict(name="mnist_like_70000x784_L10", N=70000, D=784, L=10, k=5, lam=1.0,
                       affinity="binary", gen="mnist_like", sample_rows=16, sample_sub=7000),
}
WORKLOAD = dict(WORKLOADS["manifolds"])
PEAKS_PATH = os.path.join(ROOT, "MEASURED_PEAKS.json")
FP32_LANES_PER_SM = 128      # FP32 FMA units per SM (4 sub-partitions x 32)
SEED = 1810

# DRAM traffic (dram__bytes_read.sum + dram__bytes_write.sum) of one launch of
# a kernel on a workload, from a one-pass ncu capture, with the SHA-256 at capture
# time of the kernel's own part of its source file, from the line that begins it
# to the end of the kernel: a changed kernel reports null.
NCU_TRAFFIC = {
    ("bound_staged_kernel", "manifolds_1000000x128_L100"): {
        "bytes": 6510319872 + 2380906240,
        "source": "paper_1810_13044_gb300/csrc/bound.cu",
        "begin": "// ------------------------------------- staged form for large N",
        "sha256": "165c1bbdfebb48dffb55511dd7dd8fbf69aa9587daa23efcadb476c7a59ec108",
    },
}


# What the distance tiles' figures say: the algorithm's N^2 pairs over the time
# of the whole candidate phase, not a rate of the tensor cores.
SWEEP_NOTE = ("achieved counts all N^2 pairs; tiles that cannot hold a neighbour are left out above "
              "a work size, so it is an all-pairs equivalent, not a share of the peak")


def ncu_traffic(kernel, workload):
    """Per-launch DRAM bytes of `kernel` on `workload` if its source is unchanged."""
    rec = NCU_TRAFFIC.get((kernel, workload))
    if rec is None:
        return None
    import hashlib
    path = os.path.join(ROOT, rec["source"])
    if not os.path.exists(path):
        return None
    with open(path) as f:
        text = f.read()
    at = text.find(rec["begin"])
    end = text.find("\n}\n", text.find(kernel + "(", max(at, 0)))
    if at < 0 or end < 0 or hashlib.sha256(text[at:end].encode()).hexdigest() != rec["sha256"]:
        return None
    return rec["bytes"]


def parse(argv=None):
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["slk", "reference"], default="slk")
    ap.add_argument("--precision", choices=["fp32", "bf16_rerank"], default="bf16_rerank")
    ap.add_argument("--no-fp32-compare", action="store_true",
                    help="skip timing the plain float32 solve beside the main arm")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-nested", action="store_true",
                    help="skip the second (70000 x 784) workload carried in the default line")
    ap.add_argument("--workload", choices=["manifolds", "mnist_like", "batched", "serving", "ms"],
                    default="manifolds",
                    help="manifolds: one 1e6 x 128, L=100, k=10 heat-affinity solve per step; "
                         "mnist_like: one 70000 x 784, L=10, k=5 solve per step; ms: the "
                         "70000 x 784 problem solved by SLK-MS (mean-shift modes); batched: 256 "
                         "uneven problems per step (slk_solve_batched); serving: a Poisson "
                         "request stream")
    ap.add_argument("--instances", type=int, default=256)
    ap.add_argument("--requests", type=int, default=2000, help="serving: requests in the stream")
    ap.add_argument("--rate", type=float, default=200.0, help="serving: mean Poisson arrival rate (req/s)")
    ap.add_argument("--rate-search", action="store_true",
                    help="serving: also search the highest sustainable arrival rate")
    ap.add_argument("--rows", type=int, default=None,
                    help="generate the workload with this many points (profiling captures)")
    args = ap.parse_args(argv)
    base = "mnist_like" if args.workload in ("mnist_like", "ms") else "manifolds"
    WORKLOAD.clear()
    WORKLOAD.update(WORKLOADS[base])
    if args.rows:
        WORKLOAD["N"] = args.rows
        WORKLOAD["name"] = f"{WORKLOAD['gen']}_{args.rows}x{WORKLOAD['D']}_L{WORKLOAD['L']}"
        WORKLOAD["sample_sub"] = min(WORKLOAD["sample_sub"], args.rows)
    return args


def whole_job(ms_local, units_per_rank, world, device=None):
    """Max of the ranks' timed milliseconds (all_reduce MAX when world > 1) and
    the whole-job throughput: units of every rank / that time (replicas: each
    rank solves its own copy, so per-rank work is fixed as ranks are added)."""
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(ms_local)], dtype=torch.float64, device=device)
    if world > 1:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    ms_max = float(t.item())
    return ms_max, world * units_per_rank / (ms_max / 1e3)


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def make_points(W):
    """The workload's seeded points (float32, N x D)."""
    from paper_1810_13044_gb300 import inputs
    if W["gen"] == "manifolds":
        X, _ = inputs.manifolds(N=W["N"], D=W["D"], n_clusters=W["L"])
    else:
        X, _ = inputs.mnist_like(N=W["N"], D=W["D"])
    return X


def seeds_gpu(W, Xd, ctx):
    """K-means++ seeds (Section 4.2) of the workload, drawn on the GPU from the
    seeded draws of inputs.kmeanspp_draws (equal to inputs.kmeanspp)."""
    from paper_1810_13044_gb300 import inputs, slk
    first, u = inputs.kmeanspp_draws(W["N"], W["L"], SEED)
    return slk.kmeanspp(Xd, W["L"], first, u, ctx=ctx)


# ------------------------------------------------------------------ clocks

class ClockSampler:
    """nvidia-smi samples (200 ms) of SM clock and throttle reasons while running."""

    FIELDS = ["clocks.sm", "clocks.max.sm", "power.draw", "clocks_event_reasons.hw_slowdown",
              "clocks_event_reasons.hw_thermal_slowdown", "clocks_event_reasons.sw_thermal_slowdown",
              "clocks_event_reasons.sw_power_cap"]

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.index}", "--query-gpu=" + ",".join(self.FIELDS),
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except (OSError, FileNotFoundError):
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *a):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()

    def summary(self):
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) != len(self.FIELDS):
                continue
            try:
                sm.append(float(parts[0]))
                mx.append(float(parts[1]))
            except ValueError:
                continue
            for n, v in zip(names, parts[3:]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["unsampled"], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


# ------------------------------------------------------------------ oracle sample

class OracleSample:
    """The bounded CPU sample of one solve that both the main arm's
    cpu_baseline and the reference arm time, with the FP64 oracle as it
    stands on all host cores:

    * kNN: the exact kNN rows of `sample_rows` points of the full problem
      (each against all N points), scaled to N rows;
    * Algorithm 1: a whole solve (exact kNN graph, median sigma, K-means++
      seeds, outer loop to convergence with tol 1e-6 / max_inner 100) of the
      first `sample_sub` points (a uniform subsample: points are stored in a
      seeded random order), scaled linearly to N rows (unary, z-updates, mode
      update and energy are linear in N at fixed L, k).

    The subsample's own kNN graph, sigma and seeds are prepared once and not
    timed (their cost is covered by the kNN leg)."""

    def __init__(self, W, X):
        import oracle
        from paper_1810_13044_gb300 import inputs
        self.W, self.X = W, X
        N, k, L = W["N"], W["k"], W["L"]
        self.rows = np.linspace(0, N - 1, W["sample_rows"]).astype(np.int64)
        n = min(W["sample_sub"], N)
        self.Xs = np.ascontiguousarray(X[:n])
        idx, d2 = oracle.knn(self.Xs, k)
        self.sig = oracle.sigma(d2, "median")
        self.rp = np.arange(n + 1, dtype=np.int64) * k
        self.ci = idx.reshape(-1)
        self.w = oracle.heat_weights(d2.reshape(-1), self.sig) if W["affinity"] == "heat" else None
        first, u = inputs.kmeanspp_draws(n, min(L, n), SEED)
        self.m0 = oracle.kmeanspp(self.Xs, min(L, n), first, u)
        self.cores = oracle.threads()

    def run(self):
        """Seconds per solve of the full problem, extrapolated from the sample."""
        import oracle
        W, N = self.W, self.W["N"]
        n = self.Xs.shape[0]
        t0 = time.perf_counter()
        oracle.knn(self.X, W["k"], rows=self.rows)
        t_knn = (time.perf_counter() - t0) * N / len(self.rows)
        t0 = time.perf_counter()
        ref = oracle.solve_graph(self.Xs, len(self.m0), self.rp, self.ci, self.w, self.sig, W["lam"],
                                 self.m0)
        t_solve = (time.perf_counter() - t0) * N / n
        self.last = ref
        return t_knn + t_solve

    def describe(self):
        W = self.W
        n = self.Xs.shape[0]
        r = getattr(self, "last", None)
        it = f" ({r['outer']} outer iterations, {r['inner_total']} z-updates)" if r else ""
        return (f"FP64 oracle on {self.cores} threads: exact kNN rows of {len(self.rows)} of the "
                f"{W['N']} points scaled x{W['N'] / len(self.rows):.0f}, plus a whole Algorithm-1 "
                f"solve of a {n}-point subsample on its own exact kNN graph{it} scaled "
                f"x{W['N'] / n:.1f}")


# ------------------------------------------------------------------ arms

def run_reference(args, rank, world):
    if rank != 0:
        return
    X = make_points(WORKLOAD)
    sample = OracleSample(WORKLOAD, X)
    for _ in range(args.warmup):
        sample.run()
    times = [sample.run() for _ in range(args.steps)]
    sec = statistics.median(times)
    value = 1.0 / sec
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": "solves/s", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": sec * 1e3,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic", "config": {"workload": WORKLOAD["name"], **{k: WORKLOAD[k] for k in
                                                                          ("N", "D", "L", "k")}},
        "cpu_baseline": {"value": value, "unit": "solves/s", "cores": sample.cores, "kind": "oracle",
                         "sample": sample.describe()},
        "e2e": {"value": value, "unit": "solves/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)


def _events(torch):
    return torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)


def measure_workload(W, args, ctx, dev, world, stream, main: bool):
    """Time one workload's solves and the figures around them.  Returns the
    per-workload dict (device value, e2e, rooflines, plain float32 solve)
    plus the clock summary and launch count of its timed region."""
    import torch
    import torch.distributed as dist

    from paper_1810_13044_gb300 import slk

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    N, D, L, k, lam = (W[x] for x in ("N", "D", "L", "k", "lam"))
    heat = W["affinity"] == "heat"
    X = make_points(W)
    Xd = torch.from_numpy(X).to(dev)
    m0d = seeds_gpu(W, Xd, ctx)
    params = slk.default_params(knn_precision=args.precision, affinity=W["affinity"])
    out = (torch.empty(N, L, device=dev), torch.empty(N, dtype=torch.int32, device=dev),
           torch.empty(L, dtype=torch.int32, device=dev))

    def step():
        return slk.solve(Xd, L, k, lam, m0d, params=params, ctx=ctx, out=out)

    for _ in range(args.warmup):
        _, _, _, stats = step()
    barrier()
    ev0, ev1 = _events(torch)
    ctx.profile(True)
    with ClockSampler(dev.index) as clk:
        barrier()
        ev0.record(stream)
        for _ in range(args.steps):
            _, _, _, stats = step()
        ev1.record(stream)
        barrier()
    ms_phase, calls, launches = ctx.profile_read()
    ctx.profile(False)
    ms_max, value = whole_job(ev0.elapsed_time(ev1), args.steps, world, dev)

    labels_main = out[1].clone()
    modes_main = out[2].clone()
    plain = None
    if not args.no_fp32_compare and args.precision != "fp32":
        # the plain float32 GPU solve at equal labels (same workload, own timing)
        p32 = slk.default_params(knn_precision="fp32", affinity=W["affinity"])
        out32 = (torch.empty(N, L, device=dev), torch.empty(N, dtype=torch.int32, device=dev),
                 torch.empty(L, dtype=torch.int32, device=dev))
        slk.solve(Xd, L, k, lam, m0d, params=p32, ctx=ctx, out=out32)
        barrier()
        f0, f1 = _events(torch)
        steps32 = min(args.steps, 5) if N <= 100000 else 1   # float32 tiles at 1e6 rows take seconds
        f0.record(stream)
        for _ in range(steps32):
            slk.solve(Xd, L, k, lam, m0d, params=p32, ctx=ctx, out=out32)
        f1.record(stream)
        barrier()
        plain = {"value": steps32 / (f0.elapsed_time(f1) / 1e3), "unit": "solves/s", "knn": "fp32",
                 "steps": steps32,
                 "equal_labels": bool(torch.equal(out32[1], labels_main)),
                 "equal_modes": bool(torch.equal(out32[2], modes_main))}

    # bound iterations alone on this solve's graph: N*L*iter/s (fixed 50 updates)
    g = slk.knn_graph(Xd, k, precision=args.precision, ctx=ctx, affinity=W["affinity"],
                      sigma=stats["sigma"])
    gw = g.w if heat else None
    A, Z0 = slk.unary(Xd, out[2], stats["sigma"], ctx=ctx)
    Zb, Zp = Z0.clone(), torch.empty_like(Z0)
    slk.bound_iterate(A, g.row_ptr, g.col_idx, gw, lam, Zb, Zp, 50, tol=-1.0, ctx=ctx)
    e0, e1 = _events(torch)
    reps = 5
    e0.record(stream)
    for _ in range(reps):
        Zb.copy_(Z0)
        slk.bound_iterate(A, g.row_ptr, g.col_idx, gw, lam, Zb, Zp, 50, tol=-1.0, ctx=ctx)
    e1.record(stream)
    torch.cuda.synchronize()
    bound_ms = e0.elapsed_time(e1) / reps
    del g, A, Z0, Zb, Zp

    # starting modes (Section 4.2) on the same data, timed alone: N x N float32
    # distance tiles with the kernel-density epilogue
    init_ms = None
    if N <= 200000:
        slk.initial_modes(Xd, m0d, stats["sigma"], ctx=ctx)
        i0, i1 = _events(torch)
        i0.record(stream)
        slk.initial_modes(Xd, m0d, stats["sigma"], ctx=ctx)
        i1.record(stream)
        torch.cuda.synchronize()
        init_ms = i0.elapsed_time(i1)

    # e2e through the host-buffer entry point (pinned X in, labels + modes out)
    Xh = torch.from_numpy(X).pin_memory()
    m0h = m0d.cpu()
    hout = (None, torch.empty(N, dtype=torch.int32).pin_memory(),
            torch.empty(L, dtype=torch.int32).pin_memory())
    slk.solve_host(Xh, L, k, lam, m0h, params=params, ctx=ctx, out=hout)
    barrier()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        slk.solve_host(Xh, L, k, lam, m0h, params=params, ctx=ctx, out=hout)
    barrier()
    _, e2e_value = whole_job((time.perf_counter() - t0) * 1e3, args.steps, world, dev)

    peaks = json.load(open(PEAKS_PATH)) if os.path.exists(PEAKS_PATH) else {}
    sm_mhz = peaks.get("sm_max_mhz", 2070.0)
    fp32_peak = 152 * FP32_LANES_PER_SM * 2 * sm_mhz * 1e6 / 1e12
    # the distance tiles of the kNN graph
    cand_ms = ms_phase["knn_cand"] / max(1, calls["knn_cand"])
    Dp = ((D + 15) // 16) * 16
    flops = 2.0 * N * N * D
    if args.precision == "fp32":
        roof = {"bound": "alu", "kernel": "knn_cand_fp32_kernel",
                "achieved": flops / (cand_ms / 1e3) / 1e12, "peak": fp32_peak, "unit": "TFLOP/s",
                "peak_source": "derived: 152 SMs x 128 FP32 lanes x 2 flop x max SM clock",
                "traffic": None}
    else:
        peak = peaks.get("bf16_tflops", 1900.0)
        roof = {"bound": "tensor", "kernel": "knn_sweep_kernel", "note": SWEEP_NOTE,
                "achieved": flops / (cand_ms / 1e3) / 1e12, "peak": peak, "unit": "TFLOP/s",
                "peak_source": ("of measured bf16_tflops (burst)" if "bf16_tflops" in peaks
                                else "of fallback"),
                "traffic": ncu_traffic("knn_sweep_kernel", W["name"])}
    roof["frac"] = None if "note" in roof else roof["achieved"] / roof["peak"]
    roof["launch_ms"] = cand_ms
    roof["algorithmic"] = f"2*N*N*D = {flops:.3e} flop per launch (Dp={Dp})"
    # bound iterations: per row and update row_ptr 8 + col 4k (+ w 4k) + a, z_old, z_new 12L
    # bytes (each neighbour row of Z counted once, the ideal reuse)
    b_row = 8 + 4 * k + (4 * k if heat else 0) + 12 * L
    hbm = peaks.get("hbm_gbs", 6800.0)
    upd = max(1, stats["inner_iters_total"]) * args.steps
    gbs = N * b_row * upd / (ms_phase["bound"] / 1e3) / 1e9
    # the z-update kernel bound_launch picks for this shape (fixed degree k)
    if N >= 100000 and 64 < L <= 128 and L % 4 == 0:
        bkern = "bound_staged_kernel"
    elif N * (4 * L + 4 * k + (4 * k if heat else 0)) <= 96 * 1024 * 2 * 152:
        bkern = "bound_cached_kernel"
    else:
        bkern = "bound_persistent_kernel"
    roof_bound = {"bound": "hbm", "kernel": bkern, "achieved": gbs,
                  "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
                  "peak_source": "of measured hbm_gbs" if "hbm_gbs" in peaks else "of fallback",
                  "traffic": ncu_traffic(bkern, W["name"]),
                  "traffic_note": "per launch = the z-updates of one outer iteration",
                  "algorithmic": f"N*(8+4k{'+4k' if heat else ''}+12L) = {N * b_row / 1e6:.1f} MB "
                                 f"per update; the solve's bound phase over its "
                                 f"{stats['inner_iters_total']} updates",
                  "launch_ms": ms_phase["bound"] / max(1, calls["bound"]),
                  "rows_sorted_by_mode": N * L * 4 > (64 << 20),
                  "l2_resident": N * b_row < 100e6,
                  "fixed_50_updates_gbs": N * b_row * 50 / (bound_ms / 1e3) / 1e9}
    fb_ms = ms_phase["knn_fallback"] / max(1, calls["knn_fallback"])
    fb_rows = stats["knn_fallback_rows"]
    if ms_phase["knn_fallback"] > max(ms_phase["knn_cand"], ms_phase["bound"]) and fb_rows > 0:
        fflops = 2.0 * fb_rows * N * D
        roof = {"bound": "alu", "kernel": "knn_fallback_batch_kernel",
                "achieved": fflops / (fb_ms / 1e3) / 1e12, "peak": fp32_peak, "unit": "TFLOP/s",
                "peak_source": "derived: 152 SMs x 128 FP32 lanes x 2 flop x max SM clock",
                "traffic": None, "launch_ms": fb_ms,
                "algorithmic": f"2*rows*N*D = {fflops:.3e} flop per launch ({fb_rows} rows)"}
        roof["frac"] = roof["achieved"] / roof["peak"]
    elif ms_phase["bound"] > ms_phase["knn_cand"]:
        roof = dict(roof_bound)
    res = {
        "value": value, "unit": "solves/s", "ms_per_step": ms_max / args.steps,
        "config": {"workload": W["name"], "N": N, "D": D, "L": L, "k": k, "lambda": lam,
                   "sigma": "median kNN distance", "affinity": W["affinity"],
                   "seeds": "K-means++ (Section 4.2) drawn on the GPU from seeded draws",
                   "knn": ("float32 SIMT distance tiles" if args.precision == "fp32" else
                           "bfloat16 tcgen05 distance tiles for candidates, exact float32 "
                           "rerank with rounding certificate (same graph as float32)"),
                   "parallelism": f"replicas{world}" if world > 1 else "single",
                   "l2": f"inputs larger than L2 (X is {N * D * 4 / 1e6:.0f} MB, L2 129 MB)",
                   "outer_iters": stats["outer_iters"],
                   "inner_iters_total": stats["inner_iters_total"]},
        "nl_iter_per_s": N * L * 50 / (bound_ms / 1e3), "bound_ms_per_50_updates": bound_ms,
        "initial_modes": None if init_ms is None else {
            "ms": init_ms, "bound": "alu",
            "achieved_tflops": 2.0 * N * N * D / (init_ms / 1e3) / 1e12, "peak_tflops": fp32_peak,
            "algorithmic": "2*N*N*D flop (float32 distance tiles) + N*N exp; all pairs counted, the "
                           "tiles that cannot hold a cluster's maximiser are left out"},
        "phase_ms_per_step": {k_: v / args.steps for k_, v in ms_phase.items()},
        "roofline": roof,
        "roofline_bound": roof_bound,
        "plain_fp32_gpu": plain,
        "e2e": {"value": e2e_value, "unit": "solves/s", "h2d_bytes_per_step": N * D * 4 + L * 4,
                "d2h_bytes_per_step": N * 4 + L * 4},
        "energy": stats["energy"], "knn_fallback_rows": stats["knn_fallback_rows"],
        "knn_rows_by_stage": {"left_open_by_first_certificate": stats["knn_fallback_rows"],
                              "to_float32_stage": stats["knn_float32_rows"],
                              "exact_rescan": stats["knn_exact_rows"]},
    }
    return res, clk.summary(), launches, X


def run_slk(args, rank, world, local):
    import torch
    import torch.distributed as dist

    from paper_1810_13044_gb300 import slk

    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    dev = torch.device("cuda", local)
    ctx = slk.context(local)
    stream = torch.cuda.current_stream(dev)
    res, clocks, launches, X = measure_workload(WORKLOAD, args, ctx, dev, world, stream, main=True)
    nested = {}
    if (not args.no_nested and WORKLOAD["gen"] == "manifolds" and not args.rows):
        W2 = WORKLOADS["mnist_like"]
        r2, c2, l2, _ = measure_workload(W2, args, ctx, dev, world, stream, main=False)
        r2["clocks"] = c2
        r2["gpu_launches"] = l2
        nested[W2["name"]] = r2
    if rank == 0:
        line = {
            "metric": METRIC, "value": res["value"], "unit": "solves/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": res["ms_per_step"],
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": res["config"],
        }
        line.update({k_: v for k_, v in res.items() if k_ not in line and k_ != "config"})
        line["gpu_launches"] = launches
        line["clocks"] = clocks
        if nested:
            line["workloads"] = nested
        if not args.no_cpu_baseline:
            sample = OracleSample(WORKLOAD, X)
            sec = sample.run()
            line["cpu_baseline"] = {"value": 1.0 / sec, "unit": "solves/s", "cores": sample.cores,
                                    "kind": "oracle", "sample": sample.describe()}
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


def oracle_ms_sample(X, m0, sig, rows=2000, ms_iters=1):
    """Seconds of one Eq. (mean-shift) iteration of the FP64 oracle on the
    full problem, from one iteration on `rows` rows scaled to N rows."""
    import oracle
    N, L = WORKLOAD["N"], WORKLOAD["L"]
    Xs = X[:rows]
    M0 = X[m0].astype(np.float64)
    A = oracle.unary_vec(Xs, M0, sig)
    t0 = time.perf_counter()
    oracle.mean_shift(Xs, oracle.log_z(A), M0, sig, ms_iters, -1.0)
    return (time.perf_counter() - t0) / ms_iters * N / rows


def run_ms(args, rank, world, local):
    """SLK-MS (modes by Eq. mean-shift) on the 70000 x 784, L=10, k=5 problem."""
    import torch
    import torch.distributed as dist

    from paper_1810_13044_gb300 import slk

    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    X = make_points(WORKLOAD)
    N, D, L, k, lam = (WORKLOAD[x] for x in ("N", "D", "L", "k", "lam"))
    dev = torch.device("cuda", local)
    Xd = torch.from_numpy(X).to(dev)
    params = slk.default_params(knn_precision=args.precision)
    ctx = slk.context(local)
    m0d = seeds_gpu(WORKLOAD, Xd, ctx)
    out = (torch.empty(N, L, device=dev), torch.empty(N, dtype=torch.int32, device=dev),
           torch.empty(L, D, device=dev))

    def step():
        return slk.solve_ms(Xd, L, k, lam, m0d, params=params, ctx=ctx, out=out)

    for _ in range(args.warmup):
        _, _, _, stats = step()
    torch.cuda.synchronize()

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    stream = torch.cuda.current_stream(dev)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ctx.profile(True)
    with ClockSampler(local) as clk:
        barrier()
        ev0.record(stream)
        for _ in range(args.steps):
            _, _, _, stats = step()
        ev1.record(stream)
        barrier()
    ms_phase, calls, launches = ctx.profile_read()
    ctx.profile(False)
    ms_max, value = whole_job(ev0.elapsed_time(ev1), args.steps, world, dev)

    # e2e through the public API: pinned host X in, labels + modes out, every step
    Xh = torch.from_numpy(X).pin_memory()
    lab_h = torch.empty(N, dtype=torch.int32).pin_memory()
    M_h = torch.empty(L, D, dtype=torch.float32).pin_memory()
    Xe = torch.empty_like(Xd)

    def e2e_step():
        Xe.copy_(Xh, non_blocking=True)
        slk.solve_ms(Xe, L, k, lam, m0d, params=params, ctx=ctx, out=out)
        lab_h.copy_(out[1], non_blocking=True)
        M_h.copy_(out[2], non_blocking=True)

    e2e_step()
    barrier()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        e2e_step()
    barrier()
    _, e2e_value = whole_job((time.perf_counter() - t0) * 1e3, args.steps, world, dev)

    if rank == 0:
        peaks = json.load(open(PEAKS_PATH)) if os.path.exists(PEAKS_PATH) else {}
        sm_mhz = peaks.get("sm_max_mhz", 2070.0)
        fp32_peak = 152 * FP32_LANES_PER_SM * 2 * sm_mhz * 1e6 / 1e12
        ms_iters = stats["ms_iters_total"]
        ms_launch_ms = ms_phase["mean_shift"] / max(1, calls["mean_shift"])
        # Eq. (mean-shift): per (point, label, feature) a difference, a square-add
        # (distance) and a multiply-add (weighted sum) = 5 flop
        ms_flops = 5.0 * N * L * D * ms_iters / max(1, stats["outer_iters"])
        roof_ms = {"bound": "alu", "kernel": "ms_persistent_kernel",
                   "achieved": ms_flops / (ms_launch_ms / 1e3) / 1e12, "peak": fp32_peak,
                   "unit": "TFLOP/s",
                   "peak_source": "derived: 152 SMs x 128 FP32 lanes x 2 flop x max SM clock",
                   "traffic": None, "launch_ms": ms_launch_ms,
                   "algorithmic": f"5*N*L*D flop per mean-shift iteration x "
                                  f"{ms_iters / max(1, stats['outer_iters']):.1f} iterations per launch"}
        roof_ms["frac"] = roof_ms["achieved"] / roof_ms["peak"]
        cand_ms = ms_phase["knn_cand"] / max(1, calls["knn_cand"])
        flops = 2.0 * N * N * D
        peak = peaks.get("bf16_tflops", 1900.0)
        roof_knn = {"bound": "tensor", "kernel": "knn_sweep_kernel", "note": SWEEP_NOTE,
                    "achieved": flops / (cand_ms / 1e3) / 1e12, "peak": peak, "unit": "TFLOP/s",
                    "peak_source": "measured bf16_tflops" if "bf16_tflops" in peaks else "fallback",
                    "traffic": None, "launch_ms": cand_ms,
                    "algorithmic": f"2*N*N*D = {flops:.3e} flop per launch"}
        roof_knn["frac"] = None
        # the dominant kernel of the step by device time
        dominant = roof_ms if ms_phase["mean_shift"] >= ms_phase["knn_cand"] else roof_knn
        line = {
            "metric": METRIC, "value": value, "unit": "solves/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_max / args.steps,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": WORKLOAD["name"] + "_slk_ms", "N": N, "D": D, "L": L, "k": k,
                       "lambda": lam, "sigma": "median kNN distance", "modes": "mean-shift (SLK-MS)",
                       "knn": args.precision, "parallelism": f"replicas{world}" if world > 1 else "single",
                       "l2": f"inputs larger than L2 (X is {N * D * 4 / 1e6:.0f} MB, L2 129 MB)",
                       "outer_iters": stats["outer_iters"],
                       "inner_iters_total": stats["inner_iters_total"],
                       "ms_iters_total": ms_iters,
                       "max_ms": params.max_ms, "tol_ms": params.tol_ms, "tol_modes": params.tol_modes},
            "phase_ms_per_step": {k_: v / args.steps for k_, v in ms_phase.items()},
            "roofline": dominant,
            "roofline_mean_shift": roof_ms,
            "e2e": {"value": e2e_value, "unit": "solves/s", "h2d_bytes_per_step": N * D * 4,
                    "d2h_bytes_per_step": N * 4 + L * D * 4},
            "gpu_launches": launches,
            "clocks": clk.summary(),
            "energy": stats["energy"],
        }
        if not args.no_cpu_baseline:
            import oracle
            from paper_1810_13044_gb300 import inputs
            sample = OracleSample(WORKLOAD, X)
            sec = sample.run()
            first, u = inputs.kmeanspp_draws(N, L, SEED)
            m0 = oracle.kmeanspp(X, L, first, u)
            t_ms = oracle_ms_sample(X, m0, sample.sig)
            line["cpu_baseline"] = {"value": 1.0 / (sec + t_ms * ms_iters), "unit": "solves/s",
                                    "cores": sample.cores, "kind": "oracle",
                                    "sample": sample.describe() + f"; mean-shift: one iteration on "
                                              f"2000 rows scaled x{N // 2000} rows and x{ms_iters} "
                                              f"iterations"}
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


def make_batch(count, seed=1810):
    """The batched workload: N ~ U[500, 20000], D in {9, 64, 256}, L ~ U[5, 50],
    imbalanced Gaussian mixtures (largest cluster 60-80 %), k = 5, K-means++ seeds."""
    from paper_1810_13044_gb300 import inputs
    g = inputs.rng(seed)
    probs = []
    for i in range(count):
        N = int(g.integers(500, 20001))
        D = int(g.choice([9, 64, 256]))
        L = int(g.integers(5, 51))
        X, _ = inputs.mixture(N, D, L, seed=seed * 7919 + i)
        m0 = inputs.kmeanspp(X, L, seed=seed * 7919 + i)
        probs.append(dict(X=X, m0=m0, N=N, D=D, L=L, k=5, lam=1.0))
    return probs


def run_batched(args, rank, world, local):
    import torch
    import torch.distributed as dist

    from paper_1810_13044_gb300 import slk

    torch.cuda.set_device(local)
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    dev = torch.device("cuda", local)
    probs = make_batch(args.instances)
    for pr in probs:
        pr["Xd"] = torch.from_numpy(pr["X"]).to(dev)
        pr["m0d"] = torch.from_numpy(pr["m0"]).to(dev)
    params = slk.default_params(knn_precision=args.precision)
    ctx = slk.context(local)
    batch = [dict(X=pr["Xd"], L=pr["L"], k=pr["k"], lam=pr["lam"], init_modes=pr["m0d"]) for pr in probs]
    outs = [(torch.empty(pr["N"], pr["L"], device=dev), torch.empty(pr["N"], dtype=torch.int32, device=dev),
             torch.empty(pr["L"], dtype=torch.int32, device=dev)) for pr in probs]

    def step():
        return slk.solve_batched(batch, params=params, ctx=ctx, outs=outs)

    for _ in range(args.warmup):
        res = step()

    def barrier():
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    stream = torch.cuda.current_stream(dev)
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ctx.profile(True)
    with ClockSampler(local) as clk:
        barrier()
        ev0.record(stream)
        for _ in range(args.steps):
            res = step()
        ev1.record(stream)
        barrier()
    ms_phase, _, launches = ctx.profile_read()
    ctx.profile(False)
    n = len(probs)
    ms_max, value = whole_job(ev0.elapsed_time(ev1), n * args.steps, world, dev)
    outer = [r[3]["outer_iters"] for r in res]
    inner = [r[3]["inner_iters_total"] for r in res]
    # the plain per-instance GPU solve of the same problems, and label agreement
    single = []
    barrier()
    f0, f1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    f0.record(stream)
    for pr in probs:
        single.append(slk.solve(pr["Xd"], pr["L"], pr["k"], pr["lam"], pr["m0d"], params=params, ctx=ctx))
    f1.record(stream)
    barrier()
    ms1 = f0.elapsed_time(f1)
    equal = sum(int(torch.equal(a[1], b[1]) and torch.equal(a[2], b[2])) for a, b in zip(res, single))
    if rank == 0:
        rows = sum(pr["N"] for pr in probs)
        line = {
            "metric": METRIC, "value": value, "unit": "solves/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_max / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": f"batched_{n}_mixtures", "instances": n, "rows_total": rows,
                       "N": "U[500,20000]", "D": "{9,64,256}", "L": "U[5,50]", "k": 5, "lambda": 1.0,
                       "knn": args.precision, "l2": "inputs larger than L2 (all problems' X together)"},
            "plain_per_instance_gpu": {"value": n / (ms1 / 1e3), "unit": "solves/s",
                                       "equal_labels_and_modes": f"{equal}/{n}"},
            "gpu_launches": launches, "clocks": clk.summary(),
            "phase_ms_per_step": {k_: v / args.steps for k_, v in ms_phase.items() if v},
            "outer_iters": {"max": max(outer), "mean": sum(outer) / n},
            "inner_iters_total": {"max": max(inner), "mean": sum(inner) / n},
        }
        print(json.dumps(line), flush=True)
    if world > 1:
        dist.destroy_process_group()


def make_request_pool(count, dev, seed=1810):
    """Serving requests: N log-uniform in [1e3, 2e5], D in {64, 512, 4096},
    L ~ U[5, 100], k ~ U[5, 10].  Features like the 70000 x 784 workload's,
    drawn on the device (seeded): per cluster a 10-dim latent Gaussian
    u ~ N(mu_c, I), mu_c ~ N(0, 9 I), pushed through a fixed random map
    x = W2 ReLU(W1 u + b1) (256 hidden units), so that the D-dim features have
    low intrinsic dimension, as image features do.  Initial modes: seeded
    random distinct points.  A stream draws its requests from this pool."""
    import torch
    from paper_1810_13044_gb300 import inputs
    g = inputs.rng(seed)
    reqs = []
    for i in range(count):
        N = int(np.exp(g.uniform(np.log(1e3), np.log(2e5))))
        D = int(g.choice([64, 512, 4096]))
        L = int(g.integers(5, 101))
        k = int(g.integers(5, 11))
        tg = torch.Generator(device=dev).manual_seed(seed * 100003 + i)
        mu = torch.randn(L, 10, generator=tg, device=dev) * 3.0
        lab = torch.randint(0, L, (N,), generator=tg, device=dev)
        U = mu[lab] + torch.randn(N, 10, generator=tg, device=dev)
        W1 = torch.randn(256, 10, generator=tg, device=dev) / np.sqrt(10)
        b1 = torch.randn(256, generator=tg, device=dev)
        W2 = torch.randn(D, 256, generator=tg, device=dev) / np.sqrt(256)
        X = (torch.relu(U @ W1.T + b1) @ W2.T).contiguous()
        m0 = torch.randperm(N, generator=tg, device=dev)[:L].to(torch.int32).contiguous()
        reqs.append(dict(X=X, L=L, k=k, lam=1.0, init_modes=m0, N=N, D=D))
    return reqs


def serve_stream(slk, ctx, params, pool, seq, arrivals, budget, keep=0):
    """Serve the requests pool[seq[i]] arriving at arrivals[i] (seconds from
    the start) on a fresh server; returns (completion times, wall seconds,
    (Z, labels, modes) of the first `keep` requests, the largest number of
    requests in the system while the first and while the second half of the
    stream arrived)."""
    srv = slk.Server(max_slots=64, quantum=10, memory_bytes=budget, params=params, ctx=ctx)
    done_at, tickets, pending, kept = {}, {}, set(), {}
    nxt, in_sys = 0, [0, 0]
    t0 = time.perf_counter()
    while nxt < len(seq) or pending:
        now = time.perf_counter() - t0
        while nxt < len(seq) and arrivals[nxt] <= now:
            tk = srv.submit(pool[seq[nxt]])
            tickets[tk] = nxt
            pending.add(tk)
            nxt += 1
        half = 0 if nxt <= len(seq) // 2 else 1
        in_sys[half] = max(in_sys[half], len(pending))
        if not pending:
            time.sleep(max(0.0, min(0.002, arrivals[nxt] - now)))
            continue
        srv.step()
        now = time.perf_counter() - t0
        for tk in list(pending):
            st, res = srv.poll(tk)
            if st == srv.DONE:
                i = tickets[tk]
                done_at[i] = now
                if i < keep:
                    kept[i] = (res[0].clone(), res[1].clone(), res[2].clone())
                pending.discard(tk)
    wall = time.perf_counter() - t0
    srv.close()
    return np.array([done_at[i] for i in range(len(seq))]), wall, kept, in_sys


def run_serving(args, rank, world, local):
    """A fixed-length Poisson stream through the continuous-batching server:
    p50/p99 latency (from arrival), solves/s, the highest sustainable arrival
    rate, and the plain per-instance slk_solve loop on the same requests."""
    import torch

    from paper_1810_13044_gb300 import slk

    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    pool = make_request_pool(64, dev)
    g = np.random.Generator(np.random.PCG64(77))
    n = args.requests
    seq = g.integers(0, len(pool), size=n)
    arrivals = np.cumsum(g.exponential(1.0 / args.rate, size=n))
    params = slk.default_params(knn_precision=args.precision)
    free = torch.cuda.mem_get_info(dev)[0]
    budget = int(min(free * 0.5, 120 << 30))
    ctx = slk.context(local)
    # warm-up: every pool request once through a throw-away server
    serve_stream(slk, ctx, params, pool, np.arange(len(pool)), np.zeros(len(pool)), budget)
    torch.cuda.synchronize()
    keep = min(n, 200)
    ctx.profile(True)
    with ClockSampler(local) as clk:
        done, wall, kept, in_sys = serve_stream(slk, ctx, params, pool, seq, arrivals, budget,
                                                keep=keep)
    _, _, launches = ctx.profile_read()
    ctx.profile(False)
    lat = (done - arrivals) * 1e3
    ms_max, value = whole_job(wall * 1e3, n, world, dev)
    # the plain per-instance GPU solve of the same requests, one after another
    # (all n of them, timed), then the first `keep` again against the server's
    # results (untimed)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for i in range(n):
        pr = pool[seq[i]]
        slk.solve(pr["X"], pr["L"], pr["k"], pr["lam"], pr["init_modes"], params=params, ctx=ctx)
    torch.cuda.synchronize()
    plain = n / (time.perf_counter() - t0)
    equal, dz_max, differing = 0, 0.0, []
    for i in range(keep):
        pr = pool[seq[i]]
        Z1, lab1, m1, _ = slk.solve(pr["X"], pr["L"], pr["k"], pr["lam"], pr["init_modes"],
                                    params=params, ctx=ctx)
        same = torch.equal(lab1, kept[i][1]) and torch.equal(m1, kept[i][2])
        equal += int(same)
        dz_max = max(dz_max, (Z1 - kept[i][0]).abs().max().item())
        if not same:
            differing.append(int(seq[i]))
    # the highest arrival rate the server sustains: a stream of 400 requests
    # at each rate; sustained when the queue stays bounded -- the most
    # requests in the system while the second half arrives is within 1.5x
    # (+ 8) of that while the first half arrives -- and the completions keep
    # pace with the arrivals (served per second over the arrival span >= 90 %)
    search = []
    if args.rate_search:
        for rate in (10.0, 20.0, 30.0, 40.0, 50.0, 60.0, 80.0):
            gs = np.random.Generator(np.random.PCG64(1000 + int(rate)))
            m = 400
            sq = gs.integers(0, len(pool), size=m)
            arr = np.cumsum(gs.exponential(1.0 / rate, size=m))
            d, wl, _, ins = serve_stream(slk, ctx, params, pool, sq, arr, budget)
            la = (d - arr) * 1e3
            span = arr[-1]
            done_in_span = int((d <= span).sum())
            ok = ins[1] <= 1.5 * ins[0] + 8 and done_in_span >= 0.9 * np.sum(arr <= span) - 8
            search.append({"rate": rate, "served_per_s": m / wl, "p50_ms": float(np.percentile(la, 50)),
                           "p99_ms": float(np.percentile(la, 99)), "in_system_max_by_half": ins,
                           "sustained": bool(ok)})
    sustainable = max([r["rate"] for r in search if r["sustained"]], default=None)
    if rank == 0:
        line = {
            "metric": METRIC, "value": value, "unit": "solves/s", "n_gpus": world,
            "steps": n, "warmup": 1, "ms_per_step": ms_max / n,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": f"serving_poisson{int(args.rate)}_{n}req",
                       "N": "log-uniform [1e3, 2e5]", "D": "{64, 512, 4096}", "L": "U[5,100]",
                       "k": "U[5,10]", "knn": args.precision, "arrivals": f"Poisson, mean {args.rate}/s",
                       "requests": f"{n} drawn from a pool of {len(pool)} (seeded)",
                       "memory_budget_gb": round(budget / 2**30, 1), "slots": 64, "quantum": 10,
                       "offered_rate": args.rate, "l2": "inputs larger than L2",
                       "admission": "FIFO; a request starts when a slot is free and its peak device "
                                    "state fits the arena; waiting requests queue (no dropping), "
                                    "so latency is measured from arrival"},
            "latency_ms": {"p50": float(np.percentile(lat, 50)), "p99": float(np.percentile(lat, 99)),
                           "max": float(lat.max())},
            "in_system_max_by_half": in_sys,
            "plain_per_instance_gpu": {"value": plain, "unit": "solves/s", "requests": n,
                                       "equal_labels_and_modes": f"{equal}/{keep} (the first {keep})",
                                       "max_abs_dz": dz_max,
                                       "differing_pool_requests": sorted(set(differing)),
                                       "note": "requests of 1e5 rows or more with 64 < L <= 128 run "
                                               "their z-updates alone on the staged kernel, whose "
                                               "soft-max rounds differently from the segmented "
                                               "kernel the server uses; labels then differ only at "
                                               "near-ties"},
            "rate_search": search, "max_sustainable_rate": sustainable,
            "rows_total": int(sum(pool[i]["N"] for i in seq)),
            "gpu_launches": launches, "clocks": clk.summary(),
        }
        print(json.dumps(line), flush=True)


def main():
    args = parse()
    rank, world, local = dist_env()
    if args.impl == "reference":
        run_reference(args, rank, world)
    elif args.workload == "batched":
        run_batched(args, rank, world, local)
    elif args.workload == "serving":
        run_serving(args, rank, world, local)
    elif args.workload == "ms":
        run_ms(args, rank, world, local)
    else:
        run_slk(args, rank, world, local)


if __name__ == "__main__":
    main()
