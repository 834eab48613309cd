"""Benchmark: milliseconds to a certified F2M optimum, with the roofline of the
dominant kernel (the pricing scan's tensor rate or the GDP sweep's GB/s).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--workload c1|c2|c3|c4|c5]
    python bench.py --impl reference ...     # the CPU oracle on the same workload
    python bench.py --max-iters 1000000      # every GDP phase to its fixed point
    python bench.py --pricing 2              # scans skip tile pairs that cannot hold z < 0
    python bench.py --update classes --shift 1   # class-by-class GDP sweeps (variant)
    python bench.py --degrees 1:4                # fractional b-matching, b_v in 1..4 (variant)

A step is one full f2m_solve from lambda = 0 on a fresh context: GDP phases
(128 sweeps at most each, by default), pricing scans over all n(n-1)/2 pairs,
CSR merges, sign extraction and the exact finisher, until the solution is
certified optimal for the complete graph.  Contexts are created before the timed region; L2 is flushed (a 256 MB
device write) before every timed step.  Each step is bracketed by CUDA events
on the stream the library runs on.

Default workload (the headline configuration): n = 100,000 points uniform in
[0, 10^6]^2, seed 0, k = 10 symmetrised nearest-neighbour candidate CSR.
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

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

WORKLOADS = {
    "c1": dict(kind="uniform", n=1000, k=10, seed=0),
    "c2": dict(kind="uniform", n=100_000, k=10, seed=0),
    "c3": dict(kind="mixture", n=200_000, k=12, seed=0),
    "c4": dict(kind="batch", n=0, k=10, seed=0, count=256, nmin=1000, nmax=20000),
    "c5": dict(kind="warm", n=0, k=0, seed=0, sizes=(("mixture", 100_000, 10), ("mixture", 200_000, 12))),
}


def batch_specs(w, rank=0):
    """Instance i: seed i (+ 1000 * rank), n = round(exp(U[ln nmin, ln nmax])) from a
    SplitMix64 draw of seed 0, uniform if i is even, clustered if odd."""
    import instances as I
    key = I.stream_key(w["seed"] + 1000 * rank, 77)
    u = I.draws(key, 0, w["count"]) >> np.uint64(11)
    frac = u.astype(np.float64) * (2.0 ** -53)
    lo, hi = np.log(w["nmin"]), np.log(w["nmax"])
    ns = np.floor(np.exp(lo + frac * (hi - lo)) + 0.5).astype(int)
    return [("uniform" if i % 2 == 0 else "mixture", int(ns[i]), i + 1000 * rank, w["k"])
            for i in range(w["count"])]
METRIC = "ms to certified F2M optimum"
GDP_BYTES_PER_ENTRY = 8   # {col, cost} streamed per directed entry
GDP_BYTES_PER_NODE = 12   # row_ptr + lambda read + lambda write
PRICING_FLOPS_PER_PAIR = 16  # the filter's inner product: 8 multiply-adds (mma.sync m16n8k8)
PRICING_PAIRS_PER_CYCLE = 64  # per SM: 128 pairs an mma.sync, one per 8 cycles and SM quarter (microbenchmark)


def workload_name(w):
    if w["kind"] == "warm":
        return ("learned warm start vs cold start: mixture n=100000 k=10 and n=200000 k=12, seed 0, "
                "network trained on 2000 solved n=20000 instances (paper_2011_08170_gb300/warm_start_mlp.npy), "
                "both solves certified optimal on all pairs")
    if w["kind"] == "batch":
        return (f"batch of {w['count']} instances, n log-uniform in [{w['nmin']}, {w['nmax']}], "
                f"uniform/clustered alternating, k={w['k']}, int32 rounded-Euclidean costs, "
                f"full O(n^2) pricing per instance, all certified")
    return (f"{w['kind']} n={w['n']} k={w['k']} seed={w['seed']}, int32 rounded-Euclidean costs, "
            f"full O(n^2) pricing, certified")


def load_peaks():
    try:
        return json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except Exception:
        return {"hbm_gbs": 6800.0, "sm_max_mhz": 2070.0, "_fallback": True}


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 200 ms."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index=0):
        self.index = index
        self.rows = []
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None
            return
        # nvidia-smi's start-up (NVML initialisation) takes CPU time and driver
        # locks: let it finish before the timed region begins
        t0 = time.perf_counter()
        while not self.rows and self.proc.poll() is None and time.perf_counter() - t0 < 5.0:
            time.sleep(0.01)

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append([x.strip() for x in line.split(",")])

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        rows = [r for r in self.rows if len(r) >= 8]
        sm = [float(r[0]) for r in rows if r[0].replace(".", "").isdigit()]
        mx = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[4 + i].lower() == "active"})
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons, "samples": len(rows)}


def dist_env():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def replica_seed(w, rank):
    """Replicas: rank r solves its own instance of the workload, seed + r."""
    return w["seed"] + rank


def max_over_ranks(dist, value, device="cuda"):
    """The largest value over the ranks (the job's time is its slowest rank's)."""
    if not dist:
        return value
    import torch
    t = torch.tensor([value], device=device, dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def cpu_oracle_estimate(d, gpu_counts, budget_s=12.0):
    """Time the CPU oracle on bounded samples of the same instance and scale.

    Samples: oracle GDP sweeps on the full instance from lambda = 0 (as many as
    fit in ~40% of the budget, at most the solve's sweep count), the oracle
    finisher from the lambda those sweeps reach, and the oracle pricing scan
    over the first rows (~40% of the budget).  Sweeps and pairs are scaled by
    the sweep count and pricing-round count of the solve.  Single thread.
    """
    import oracle
    xy, rp, col = d["xy"], d["row_ptr"], d["col"]
    n = rp.size - 1
    cost = oracle.cost_table(xy, rp, col)
    lam = np.zeros(n, np.int32)
    t0 = time.perf_counter()
    sweeps = 0
    while (time.perf_counter() - t0 < 0.4 * budget_s and sweeps < gpu_counts["iterations"]) or sweeps < 2:
        st, lam, _, _ = oracle.sweep(rp, col, cost, lam, 8, 2)
        sweeps += 1
    t_sweep = (time.perf_counter() - t0) / sweeps
    t1 = time.perf_counter()
    fst, _, _, fin_aug = oracle.finisher(rp, col, cost, lam, 8)
    t_fin = time.perf_counter() - t1
    rows, pairs, t_pr = 0, 0, 0.0
    step = max(1, n // 400)
    while t_pr < 0.4 * budget_s and rows < n:
        t1 = time.perf_counter()
        oracle.pricing(xy, rp, col, lam, 8, rows=(rows, min(n, rows + step)), cap=0)
        t_pr += time.perf_counter() - t1
        pairs += sum(n - 1 - u for u in range(rows, min(n, rows + step)))
        rows += step
    t_pair = t_pr / max(pairs, 1)
    total_pairs = n * (n - 1) / 2
    est_ms = 1e3 * (gpu_counts["iterations"] * t_sweep
                    + gpu_counts["pricing_rounds"] * total_pairs * t_pair + t_fin)
    sample = (f"{sweeps} oracle sweeps on the full instance ({t_sweep * 1e3:.1f} ms each), the oracle "
              f"finisher from the lambda they reach ({t_fin * 1e3:.0f} ms, {fin_aug} augmentations, "
              f"status {fst}) and {pairs:.3g} oracle pricing pairs over rows 0..{rows} "
              f"({t_pair * 1e9:.2f} ns/pair), scaled to {gpu_counts['iterations']} sweeps and "
              f"{gpu_counts['pricing_rounds']} full scans")
    return est_ms, sample


def run_reference(args, w, rank):
    """--impl reference: the CPU oracle (unmodified) on the same workload."""
    if rank != 0:
        return 0
    import instances as I
    import oracle
    oracle.build()
    mi = args.max_iters or 128  # the oracle's default, the library's too
    if w["kind"] in ("batch", "warm"):
        return run_reference_multi(args, w, mi)
    d = I.make_instance(w["kind"], w["n"], w["seed"], w["k"])
    # the oracle's own counts are not affordable at this size; the sweep and
    # round counts of the method are those the oracle would take (the GPU path
    # is bit-exact with it), fixed here per workload from the solve record
    counts = REFERENCE_COUNTS.get((args.workload, "fixed point" if mi >= 10 ** 5 else mi))
    if counts is None:
        r = oracle.solve(d["xy"], d["row_ptr"], d["col"], max_iters=mi)
        counts = {"iterations": r.iterations, "pricing_rounds": r.pricing_rounds}
    times = []
    sample = ""
    for i in range(args.warmup + args.steps):
        est, sample = cpu_oracle_estimate(d, counts, budget_s=args.ref_budget)
        if i >= args.warmup:
            times.append(est)
    v = statistics.median(times)
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "ms",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup, "ms_per_step": v,
            "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "int32",
            "data": "synthetic", "config": {"workload": workload_name(w), "n": w["n"], "k": w["k"],
                                            "max_iters": mi},
            "cpu_baseline": {"value": v, "unit": "ms", "cores": 1, "kind": "oracle", "sample": sample},
            "e2e": {"value": v, "unit": "ms", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    # one complete oracle solve of the same instance, timed here, outside the
    # sampled steps (about a minute at n = 100,000; skipped for larger n)
    if not args.no_ref_whole and w["n"] <= 100_000:
        t0 = time.perf_counter()
        r = oracle.solve(d["xy"], d["row_ptr"], d["col"], max_iters=mi)
        t_whole = (time.perf_counter() - t0) * 1e3
        line["cpu_baseline"]["whole_solve"] = {
            "ms": t_whole, "status": int(r.status), "certified": int(r.certified),
            "iterations": int(r.iterations), "pricing_rounds": int(r.pricing_rounds),
            "note": "one complete oracle solve of the workload (all phases, scans, merges, finisher), "
                    "single thread, timed once after the sampled steps"}
    print(json.dumps(line), flush=True)
    return 0


def run_reference_multi(args, w, mi):
    """--impl reference on the batch and warm-start workloads.  Batch: the
    oracle solves the instances whole, in order, until the budget is spent; the
    time is scaled to all instances by the sum of n^2 (the pricing scans
    dominate).  Warm start: the oracle has no network, so both instances are
    estimated cold, as for the single-instance workloads."""
    import instances as I
    import oracle
    times, sample = [], ""
    for step in range(args.warmup + args.steps):
        if w["kind"] == "batch":
            specs = batch_specs(w)
            t0 = time.perf_counter()
            done, t_solve = [], 0.0
            for sp in specs:
                if done and time.perf_counter() - t0 > args.ref_budget:
                    break
                d = I.make_instance(*sp)
                t1 = time.perf_counter()
                r = oracle.solve(d["xy"], d["row_ptr"], d["col"], max_iters=mi)
                t_solve += time.perf_counter() - t1
                assert r.status == 0 and r.certified == 2
                done.append(sp[1])
            scale = sum(float(sp[1]) ** 2 for sp in specs) / sum(float(n) ** 2 for n in done)
            est = 1e3 * t_solve * scale
            sample = (f"{len(done)} of {len(specs)} instances (n = {min(done)}..{max(done)}) solved whole by "
                      f"the oracle in {t_solve:.1f} s, scaled by the sum of n^2 over all instances")
        else:
            est, parts = 0.0, []
            for kind, n, k in w["sizes"]:
                d = I.make_instance(kind, n, w["seed"], k)
                e, s = cpu_oracle_estimate(d, {"iterations": mi, "pricing_rounds": 2},
                                           budget_s=args.ref_budget / len(w["sizes"]))
                est += e
                parts.append(f"{kind} n={n}: {s}")
            sample = "cold start (the oracle has no network); " + "; ".join(parts)
        if step >= args.warmup:
            times.append(est)
    v = statistics.median(times)
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "ms",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup, "ms_per_step": v,
            "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "int32",
            "data": "synthetic", "config": {"workload": workload_name(w), "max_iters": mi},
            "cpu_baseline": {"value": v, "unit": "ms", "cores": 1, "kind": "oracle", "sample": sample},
            "e2e": {"value": v, "unit": "ms", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# Sweep and pricing-round counts of the certified solve of each workload, at
# 128 sweeps per GDP phase (the oracle's own counts, recorded with its solve in
# tests/golden/full_size_solves.json) and with every phase run to its fixed
# point.  They only scale the CPU reference arm's bounded samples (a full
# oracle solve at n = 1e5 takes a minute or more).  c1 is small enough for the
# oracle to solve outright.
REFERENCE_COUNTS: dict = {
    ("c2", 128): {"iterations": 128, "pricing_rounds": 2},
    ("c3", 128): {"iterations": 128, "pricing_rounds": 2},
    ("c2", "fixed point"): {"iterations": 3064, "pricing_rounds": 2},
    ("c3", "fixed point"): {"iterations": 3169, "pricing_rounds": 2},
}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--workload", default="c2", choices=sorted(WORKLOADS))
    ap.add_argument("--impl", default="gdp", choices=["gdp", "reference"])
    ap.add_argument("--ref-budget", type=float, default=6.0)
    ap.add_argument("--no-ref-whole", action="store_true",
                    help="--impl reference: skip the one complete oracle solve after the sampled steps")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-c3", action="store_true",
                    help="default workload: leave out the n = 200,000 object of the line")
    ap.add_argument("--instances", type=int, default=None,
                    help="batch workloads: solve only the first N instances (profiling)")
    ap.add_argument("--pricing", type=int, default=1, choices=[1, 2],
                    help="1: full scan of all pairs (the headline); 2: the scan with far tile pairs skipped")
    ap.add_argument("--pricing-tensor", action="store_true",
                    help="full scan with the tensor-core filter instead of the fp32 filter on the CUDA cores")
    ap.add_argument("--batch-shape", type=int, default=-1,
                    help="batch workloads: fixed kernel shape instead of the autotuner's")
    ap.add_argument("--finisher", default="host", choices=["host", "gpu"],
                    help="where the finisher's first phase runs (the host threads by default, one warp "
                         "per block of 2,048 nodes on the GPU)")
    ap.add_argument("--batch-clusters", action="store_true",
                    help="batch workloads: one thread-block cluster per instance instead of the streaming kernels")
    ap.add_argument("--update", default="jacobi", choices=["jacobi", "classes"],
                    help="single instance: Jacobi sweeps (Section 5.1, the headline) or class-by-class sweeps")
    ap.add_argument("--shift", type=int, default=2, help="damping shift of the GDP step")
    ap.add_argument("--max-iters", type=int, default=None,
                    help="sweeps per GDP phase (default: the library's, 128); 1000000 runs every phase "
                         "to its fixed point")
    ap.add_argument("--degrees", default=None,
                    help="single instance: degree requirements b_v drawn uniformly from LO:HI (capped at "
                         "deg(v) - 1), the fractional b-matching LP instead of F2M")
    args = ap.parse_args()
    w = WORKLOADS[args.workload]
    rank, world, local = dist_env()
    if args.impl == "reference":
        return run_reference(args, w, rank)
    if w["kind"] == "batch":
        return run_batch(args, w, rank, world, local)
    if w["kind"] == "warm":
        return run_warm(args, w, rank, world, local)

    import torch
    import paper_2011_08170_gb300 as f2m
    from paper_2011_08170_gb300 import build as B

    B.build()
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    line = single_line(args, args.workload, w, rank, world, local, dist, f2m, torch)
    # the headline metric is quoted at n = 100k and 200k: the default line
    # carries the 200k workload too, timed the same way
    if args.workload == "c2" and line.get("_plain") and not args.no_c3:
        line["c3"] = single_line(args, "c3", WORKLOADS["c3"], rank, world, local, dist, f2m, torch,
                                 nested=True)
    line.pop("_plain", None)
    if rank == 0:
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()
    return 0


def recorded_whole_solve(w):
    """The oracle's complete solve of this instance, as recorded with its
    counters by tests/golden/make_full_size_solves.py (timed on the machine
    that wrote the record, one core)."""
    p = os.path.join(ROOT, "tests", "golden", "full_size_solves.json")
    name = f"{w['kind']}_n{w['n']}_k{w['k']}_seed{w['seed']}"
    try:
        rec = json.load(open(p))[name]
    except Exception:
        return None
    return {"ms": 1e3 * rec["oracle_seconds"], "record": f"tests/golden/full_size_solves.json[{name}]",
            "note": "one complete oracle solve (all phases, scans, merges, finisher), timed once on the "
                    "machine that wrote the record, single thread; not re-run here"}


def single_line(args, wname, w, rank, world, local, dist, f2m, torch, nested=False):
    """Times args.steps solves of one single-instance workload and returns its
    JSON object (the bench line, or the nested object of a second size)."""
    import instances as I
    # replicas: every rank solves its own instance of the same workload (seed + rank)
    d = I.make_instance(w["kind"], w["n"], replica_seed(w, rank), w["k"])
    n, nnz0 = w["n"], int(d["row_ptr"][-1])
    stream = torch.cuda.current_stream()
    flush = torch.empty(256 * 1024 * 1024, dtype=torch.uint8, device="cuda")
    flush.fill_(0)  # the fill kernel is loaded here, not in the first timed step
    torch.cuda.synchronize()

    # variants: class-by-class sweeps, degree requirements
    flags = f2m.F2M_FLAG_CLASS_SWEEPS if args.update == "classes" else 0
    b = None
    if args.degrees:
        lo, hi = (int(t) for t in args.degrees.split(":"))
        key = I.stream_key(replica_seed(w, rank), 91)
        draw = (I.draws(key, 0, n) % np.uint64(hi - lo + 1)).astype(np.int64) + lo
        b = np.minimum(draw, np.diff(d["row_ptr"]) - 1).astype(np.int32)
    variant = args.update != "jacobi" or b is not None or args.shift != 2

    def make_ctx(xy, rp, col):
        c = f2m.f2m_create(xy, rp, col, params=params, stream=stream)
        if b is not None:
            f2m.f2m_set_degrees(c, b)
        return c

    # warm-up solves (also load the module, JIT nothing)
    params = f2m.f2m_default_params(pricing=args.pricing, flags=flags | finisher_flag(f2m, args),
                                    damping_shift=args.shift)
    if args.max_iters:
        params.max_iters = args.max_iters
    for _ in range(args.warmup):
        ctx = make_ctx(d["xy"], d["row_ptr"], d["col"])
        f2m.f2m_solve(ctx)
        f2m.f2m_destroy(ctx)
    ctxs = [make_ctx(d["xy"], d["row_ptr"], d["col"]) for _ in range(args.steps)]
    clocks = ClockSampler(local)
    clocks.start()
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    launches0 = f2m.f2m_kernel_launches()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
           for _ in range(args.steps)]
    infos = []
    host = []  # per step: host ms of the flush enqueue, of f2m_solve, of the info read-out
    torch.cuda.synchronize()
    t_wall = time.perf_counter()
    for i in range(args.steps):
        t0 = time.perf_counter()
        flush.fill_(i & 0xFF)
        evs[i][0].record(stream)
        t1 = time.perf_counter()
        inf = f2m.f2m_solve(ctxs[i])
        t2 = time.perf_counter()
        evs[i][1].record(stream)
        infos.append(inf.as_dict())
        t3 = time.perf_counter()
        host.append(((t1 - t0) * 1e3, (t2 - t1) * 1e3, (t3 - t2) * 1e3))
    torch.cuda.synchronize()
    wall_ms = (time.perf_counter() - t_wall) * 1e3
    launches = f2m.f2m_kernel_launches() - launches0
    step_ms = [a.elapsed_time(b) for a, b in evs]
    if dist:
        dist.barrier()
    clk = clocks.stop()
    for c in ctxs:
        f2m.f2m_destroy(c)
    ms = sum(step_ms) / len(step_ms)
    ms = max_over_ranks(dist, ms)
    for inf in infos:
        assert inf["status"] == 0 and inf["certified"] == 2, inf

    # end to end through the C ABI with host buffers: create (upload + cost
    # table) + solve + read back x, the CSR and lambda, from and to pinned host
    # memory (the output buffers are the caller's, allocated once, like the inputs)
    xy_h = torch.from_numpy(d["xy"]).pin_memory()
    rp_h = torch.from_numpy(d["row_ptr"]).pin_memory()
    col_h = torch.from_numpy(d["col"]).pin_memory()
    cap = max(inf["nnz"] for inf in infos) * 9 // 8 + 1024
    out_x = (torch.empty(n + 1, dtype=torch.int32).pin_memory(), torch.empty(cap, dtype=torch.int32).pin_memory(),
             torch.empty(cap, dtype=torch.uint8).pin_memory(), torch.empty(cap, dtype=torch.int32).pin_memory())
    out_lam = torch.empty(n, dtype=torch.int32).pin_memory()
    e2e_ms = []
    h2d = d["xy"].nbytes + d["row_ptr"].nbytes + d["col"].nbytes
    d2h = 0
    for i in range(args.steps):
        flush.fill_(i & 0xFF)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ctx = make_ctx(xy_h, rp_h, col_h)
        info = f2m.f2m_solve(ctx)
        res_x = f2m.f2m_get_x(ctx, out=out_x)
        lam_o, _ = f2m.f2m_get_lambda(ctx, out=out_lam)
        torch.cuda.synchronize()
        e2e_ms.append((time.perf_counter() - t0) * 1e3)
        d2h = sum(t.numel() * t.element_size() for t in (*res_x, lam_o))
        f2m.f2m_destroy(ctx)
    e2e = statistics.median(e2e_ms)
    e2e = max_over_ranks(dist, e2e)

    peaks = load_peaks()
    inf0 = infos[0]
    iters = statistics.median(i["iterations"] for i in infos)
    ms_gdp = statistics.median(i["ms_gdp"] for i in infos)
    ms_pr = statistics.median(i["ms_pricing"] for i in infos)
    gdp_bytes = iters * (GDP_BYTES_PER_ENTRY * nnz0 + GDP_BYTES_PER_NODE * n)
    gdp_gbs = gdp_bytes / (ms_gdp * 1e-3) / 1e9
    # pairs the scans evaluated: n(n-1)/2 a full scan, rows x n the scan that
    # certifies the finisher's lambda (only rows whose lambda rose)
    pr_pairs = inf0.get("pricing_pairs") or inf0["pricing_rounds"] * n * (n - 1) / 2
    sm_mhz = clk.get("sm_mhz") or peaks.get("sm_max_mhz", 2070.0)
    num_sms = torch.cuda.get_device_properties(local).multi_processor_count
    pr_rate = pr_pairs / (ms_pr * 1e-3) if ms_pr > 0 else 0.0  # pairs/s
    pr_tflops = pr_rate * PRICING_FLOPS_PER_PAIR / 1e12
    pr_frac_pipe = pr_rate / (num_sms * PRICING_PAIRS_PER_CYCLE * sm_mhz * 1e6)
    traffic = load_traffic(wname)
    gdp_kernel = "gdp_classes_kernel" if args.update == "classes" else "gdp_ring_reg_kernel"
    if ms_gdp >= ms_pr:
        roofline = {"kernel": gdp_kernel, "bound": "hbm", "achieved": gdp_gbs,
                    "peak": peaks["hbm_gbs"], "unit": "GB/s", "frac": gdp_gbs / peaks["hbm_gbs"],
                    "traffic": traffic.get(gdp_kernel),
                    "note": "algorithmic bytes of the sweep over its time; the working set is shared-memory "
                            "and L2 resident, so this is an effective rate (DRAM sees the CSR once per phase)"}
    else:
        roofline = {"kernel": "pricing_kernel", "bound": "tensor", "achieved": pr_tflops, "peak": peaks["bf16_tflops"],
                    "unit": "TFLOP/s", "frac": pr_tflops / peaks["bf16_tflops"],
                    "traffic": traffic.get("pricing_kernel"),
                    "work": f"{PRICING_FLOPS_PER_PAIR} flops per pair (8 multiply-adds of the exact integer "
                            f"filter) x the pairs the scans evaluated",
                    "frac_pipe": pr_frac_pipe,
                    "frac_pipe_work": f"pairs against the issue rate of mma.sync m16n8k8, {PRICING_PAIRS_PER_CYCLE} "
                                      f"pairs a cycle and SM"}
    roofline["peak_source"] = "MEASURED_PEAKS.json" if not peaks.get("_fallback") else "fallback"
    roofline["peak_note"] = "bf16_tflops of MEASURED_PEAKS.json" \
        if roofline["kernel"] == "pricing_kernel" else "hbm_gbs of MEASURED_PEAKS.json"
    if args.pricing == 2 and roofline["kernel"] == "pricing_kernel":
        roofline["effective"] = True
        roofline["note"] = ("culled scan: the rate counts all n(n-1)/2 pairs per scan, but tile pairs that "
                            "cannot hold z < 0 are not evaluated, so it is an effective rate and can exceed "
                            "the peak")
    roofline["gdp_sweep_gbs"] = gdp_gbs
    roofline["gdp_sweep_frac_of_hbm"] = gdp_gbs / peaks["hbm_gbs"]
    roofline["gdp_working_set_mb"] = (GDP_BYTES_PER_ENTRY * nnz0 + GDP_BYTES_PER_NODE * n) / 1e6
    roofline["pricing_tflops"] = pr_tflops
    roofline["pricing_frac_pipe"] = pr_frac_pipe

    host_ms = {"flush_enqueue": statistics.median(h[0] for h in host),
               "f2m_solve": statistics.median(h[1] for h in host),
               "info_readout": statistics.median(h[2] for h in host),
               "per_step": [round(sum(h), 3) for h in host],
               "event_ms_per_step": [round(x, 3) for x in step_ms]}
    line = {"metric": METRIC, "value": ms, "unit": "ms", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": False,
            "scaling": "weak", "vs_baseline": None, "dtype": "int32", "data": "synthetic",
            "config": {"workload": workload_name(w) + ("" if args.pricing == 1 else
                                                       "; pricing skips tile pairs too far apart to hold z < 0"),
                       "pricing": "full" if args.pricing == 1 else "culled", "n": n, "k": w["k"], "nnz": nnz0,
                       "update": args.update, "damping_shift": args.shift, "max_iters": int(params.max_iters),
                       "degrees": ("2 (F2M)" if b is None else
                                   f"b_v uniform in {args.degrees.replace(':', '..')}, capped at deg(v)-1"),
                       "l2": "flushed before every timed step (256 MB device write)",
                       "parallelism": f"replicas x{world}"},
            "breakdown_ms": {k: statistics.median(i[k] for i in infos)
                             for k in ("ms_gdp", "ms_pricing", "ms_merge", "ms_extract", "ms_finish",
                                       "ms_total")},
            "solve": {k: inf0[k] for k in ("iterations", "phases", "pricing_rounds", "edges_added",
                                           "finisher_calls", "augmentations", "bound2", "frac_bits",
                                           "certified", "nnz")},
            "finisher_split": {
                "ms_prep": statistics.median(i["ms_finish_prep"] for i in infos),
                "ms_phase": [statistics.median(i["ms_finish_phase"][k] for i in infos) for k in range(3)],
                "ms_scatter": statistics.median(i["ms_finish_scatter"] for i in infos),
                "aug_phase": inf0["finish_aug_phase"], "threads": inf0["finish_threads"],
                "phase1_gpu": inf0["finish_phase1_gpu"],
                "ms_prep_per_step": [round(i["ms_finish_prep"], 3) for i in infos]},
            "sweep_edges_per_s": iters * nnz0 / (ms_gdp * 1e-3),
            "wall_ms_timed_region": wall_ms,
            "host_ms": host_ms,
            "e2e": {"value": e2e, "unit": "ms", "h2d_bytes_per_step": int(h2d),
                    "d2h_bytes_per_step": int(d2h)},
            "roofline": roofline, "clocks": clk, "gpu_launches": int(launches)}
    if nested:
        for k in ("metric", "unit", "n_gpus", "warmup", "higher_is_better", "scaling", "vs_baseline",
                  "dtype", "data"):
            line.pop(k)
    if rank == 0 and not args.no_cpu_baseline and not variant and not nested:
        est, sample = cpu_oracle_estimate(d, {"iterations": inf0["iterations"],
                                              "pricing_rounds": inf0["pricing_rounds"]})
        line["cpu_baseline"] = {"value": est, "unit": "ms", "cores": 1, "kind": "oracle",
                                "sample": sample}
        whole = recorded_whole_solve(w)
        if whole:
            line["cpu_baseline"]["whole_solve_recorded"] = whole
    line["_plain"] = not variant and args.pricing == 1 and not args.max_iters
    if nested:
        line.pop("_plain")
    return line


def run_batch(args, w, rank, world, local):
    """Batch workload: one step = f2m_solve_batch over all instances, from lambda = 0."""
    import torch
    import instances as I
    import paper_2011_08170_gb300 as f2m
    from paper_2011_08170_gb300 import build as B

    B.build()
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    specs = batch_specs(w, rank)
    if args.instances:
        specs = specs[:args.instances]
    ds = [I.make_instance(*sp) for sp in specs]
    params = f2m.f2m_default_params(batch_shape=args.batch_shape, pricing=args.pricing,
                                    flags=(f2m.F2M_FLAG_BATCH_CLUSTERS if args.batch_clusters else 0) |
                                    finisher_flag(f2m, args))
    if args.max_iters:
        params.max_iters = args.max_iters
    insts = [(d["xy"], d["row_ptr"], d["col"]) for d in ds]
    ns = np.array([d["xy"].shape[0] for d in ds])
    nnzs = np.array([int(d["row_ptr"][-1]) for d in ds])
    stream = torch.cuda.current_stream()
    flush = torch.empty(256 * 1024 * 1024, dtype=torch.uint8, device="cuda")
    flush.fill_(0)  # the fill kernel is loaded here, not in the first timed step
    torch.cuda.synchronize()
    for _ in range(args.warmup):
        b = f2m.f2m_create_batch(insts, params=params, stream=stream)
        f2m.f2m_solve_batch(b)
        f2m.f2m_destroy_batch(b)
    bs = [f2m.f2m_create_batch(insts, params=params, stream=stream) for _ in range(args.steps)]
    clocks = ClockSampler(local)
    clocks.start()
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    launches0 = f2m.f2m_kernel_launches()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
           for _ in range(args.steps)]
    res = []
    torch.cuda.synchronize()
    for i in range(args.steps):
        flush.fill_(i & 0xFF)
        evs[i][0].record(stream)
        res.append(f2m.f2m_solve_batch(bs[i]))
        evs[i][1].record(stream)
    torch.cuda.synchronize()
    launches = f2m.f2m_kernel_launches() - launches0
    clk = clocks.stop()
    step_ms = [a.elapsed_time(b) for a, b in evs]
    for b in bs:
        f2m.f2m_destroy_batch(b)
    ms = sum(step_ms) / len(step_ms)
    ms = max_over_ranks(dist, ms)
    infos, tot = res[0]
    assert tot.status == 0 and tot.certified == 2, tot.as_dict()
    # end to end: create from host arrays, solve, read every instance back
    # into the caller's pinned buffers (allocated once: one block per array,
    # a slice per instance)
    ns_b = [len(r) - 1 for _, r, _ in insts]
    caps = [inf.nnz * 9 // 8 + 64 for inf in infos]
    o_n = np.concatenate([[0], np.cumsum(ns_b)]).astype(np.int64)
    o_e = np.concatenate([[0], np.cumsum(caps)]).astype(np.int64)
    pin_rp = torch.empty(int(o_n[-1]) + len(insts), dtype=torch.int32).pin_memory()
    pin_lam = torch.empty(int(o_n[-1]), dtype=torch.int32).pin_memory()
    pin_col = torch.empty(int(o_e[-1]), dtype=torch.int32).pin_memory()
    pin_x2 = torch.empty(int(o_e[-1]), dtype=torch.uint8).pin_memory()
    outs = [((pin_rp[o_n[j] + j:o_n[j + 1] + j + 1], pin_col[o_e[j]:o_e[j + 1]], pin_x2[o_e[j]:o_e[j + 1]]),
             pin_lam[o_n[j]:o_n[j + 1]]) for j in range(len(insts))]
    e2e_ms = []
    h2d = sum(x.nbytes + r.nbytes + c.nbytes for x, r, c in insts)
    d2h = 0
    for i in range(args.steps):
        flush.fill_(i & 0xFF)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        b = f2m.f2m_create_batch(insts, params=params, stream=stream)
        f2m.f2m_solve_batch(b)
        d2h = 0
        for j in range(len(insts)):
            lam, _ = f2m.f2m_batch_get_lambda(b, j, out=outs[j][1])
            rp, col, x2 = f2m.f2m_batch_get_x(b, j, out=outs[j][0])
            d2h += sum(t.numel() * t.element_size() for t in (lam, rp, col, x2))
        torch.cuda.synchronize()
        e2e_ms.append((time.perf_counter() - t0) * 1e3)
        f2m.f2m_destroy_batch(b)
    e2e = max_over_ranks(dist, statistics.median(e2e_ms))
    peaks = load_peaks()
    sweeps = np.array([i.iterations for i in infos])
    gdp_bytes = float(np.sum(sweeps * (GDP_BYTES_PER_ENTRY * nnzs + GDP_BYTES_PER_NODE * ns)))
    ms_gdp = statistics.median(r[1].ms_gdp for r in res)
    ms_pr = statistics.median(r[1].ms_pricing for r in res)
    gdp_gbs = gdp_bytes / (ms_gdp * 1e-3) / 1e9
    pairs = float(sum(int(i.pricing_rounds) * n * (n - 1) / 2 for i, n in zip(infos, ns)))
    sm_mhz = clk.get("sm_mhz") or peaks.get("sm_max_mhz", 2070.0)
    num_sms = torch.cuda.get_device_properties(local).multi_processor_count
    pr_rate = pairs / (ms_pr * 1e-3) if ms_pr > 0 else 0.0
    tiles = tot.gdp_kernel == 8  # F2M_GDP_KERNEL_BATCH_TILES
    roofline = {"kernel": "gdp_ring_reg_kernel" if tiles else "gdp_batch_kernel", "bound": "hbm", "achieved": gdp_gbs,
                "peak": peaks["hbm_gbs"], "unit": "GB/s", "frac": gdp_gbs / peaks["hbm_gbs"],
                "traffic": None if tiles else load_traffic(args.workload).get("gdp_batch_kernel"),
                "note": "algorithmic bytes of the sweeps over their time" +
                        ("; the tiles' rows stay in registers for a phase, so this is an effective rate (DRAM sees "
                         "the graph once per phase)" if tiles else ""),
                "peak_source": "MEASURED_PEAKS.json" if not peaks.get("_fallback") else "fallback",
                "gdp_working_set_mb": float(np.sum(GDP_BYTES_PER_ENTRY * nnzs + GDP_BYTES_PER_NODE * ns)) / 1e6,
                "pricing_tflops": pr_rate * PRICING_FLOPS_PER_PAIR / 1e12,
                "pricing_frac_pipe": pr_rate / (num_sms * PRICING_PAIRS_PER_CYCLE * sm_mhz * 1e6)}
    line = {"metric": METRIC + " (all instances of the batch)", "value": ms, "unit": "ms",
            "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms,
            "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "int32",
            "data": "synthetic",
            "config": {"workload": workload_name(w) if not args.instances else
                       workload_name(w) + f" (first {len(ns)} instances)", "instances": int(len(ns)),
                       "sum_n": int(ns.sum()), "kernel_shape": int(tot.batch_shape), "graph": bool(tot.batch_graph),
                       "gdp_path": {8: "tiles", 6: "clusters"}.get(int(tot.gdp_kernel), "streaming"),
                       "max_iters": int(params.max_iters),
                       "sum_nnz": int(nnzs.sum()), "l2": "working set larger than L2; flushed before every step",
                       "parallelism": f"replicas x{world}"},
            "breakdown_ms": {k: statistics.median(getattr(r[1], k) for r in res)
                             for k in ("ms_gdp", "ms_pricing", "ms_merge", "ms_extract", "ms_finish", "ms_total")},
            "finisher_split": {
                "ms_prep": statistics.median(r[1].ms_finish_prep for r in res),
                "ms_phase": [statistics.median(r[1].ms_finish_phase[k] for r in res) for k in range(3)],
                "ms_scatter": statistics.median(r[1].ms_finish_scatter for r in res),
                "aug_phase": list(tot.finish_aug_phase), "phase1_gpu": int(tot.finish_phase1_gpu)},
            "solve": {"sweeps_total": int(sweeps.sum()), "sweeps_max": int(sweeps.max()),
                      "phases": int(tot.phases), "pricing_scans": int(tot.pricing_rounds),
                      "edges_added": int(tot.edges_added), "finisher_calls": int(tot.finisher_calls),
                      "augmentations": int(tot.augmentations)},
            "e2e": {"value": e2e, "unit": "ms", "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h)},
            "roofline": roofline, "clocks": clk, "gpu_launches": int(launches)}
    if rank == 0:
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()
    return 0


def run_warm(args, w, rank, world, local):
    """Warm-start workload: per instance, a cold solve (lambda = 0) and a warm one
    (features + network + rounding, then the same solve), both certified.  The
    value is the warm solve's ms summed over the instances, the network's time
    included; the cold sum is reported beside it."""
    import torch
    import instances as I
    import paper_2011_08170_gb300 as f2m
    from paper_2011_08170_gb300 import build as B
    from paper_2011_08170_gb300 import warm_start as W

    B.build()
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    ds = [I.make_instance(kind, n, replica_seed(w, rank), k) for kind, n, k in w["sizes"]]
    stream = torch.cuda.current_stream()
    flush = torch.empty(256 * 1024 * 1024, dtype=torch.uint8, device="cuda")
    flush.fill_(0)  # the fill kernel is loaded here, not in the first timed step
    torch.cuda.synchronize()
    m = f2m.f2m_mlp_create(W.load_weights(), stream=stream)
    params = f2m.f2m_default_params()
    if args.max_iters:
        params.max_iters = args.max_iters

    def one(d, warm):
        ctx = f2m.f2m_create(d["xy"], d["row_ptr"], d["col"], params=params, stream=stream)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        flush.fill_(1)
        e0.record(stream)
        wms = f2m.f2m_warm_start(ctx, m) if warm else 0.0
        info = f2m.f2m_solve(ctx).as_dict()
        e1.record(stream)
        torch.cuda.synchronize()
        f2m.f2m_destroy(ctx)
        assert info["status"] == 0 and info["certified"] == 2, info
        return e0.elapsed_time(e1), wms, info

    for _ in range(args.warmup):
        for d in ds:
            one(d, False)
            one(d, True)
    clocks = ClockSampler(local)
    clocks.start()
    launches0 = f2m.f2m_kernel_launches()
    per = {i: {"cold": [], "warm": [], "net": []} for i in range(len(ds))}
    infos = {}
    for _ in range(args.steps):
        for i, d in enumerate(ds):
            tc, _, ic = one(d, False)
            tw, wms, iw = one(d, True)
            per[i]["cold"].append(tc)
            per[i]["warm"].append(tw)
            per[i]["net"].append(wms)
            infos[i] = (ic, iw)
    launches = f2m.f2m_kernel_launches() - launches0
    clk = clocks.stop()
    warm_ms = max_over_ranks(dist, sum(statistics.median(per[i]["warm"]) for i in per))
    cold_ms = max_over_ranks(dist, sum(statistics.median(per[i]["cold"]) for i in per))
    rows = []
    for i, (kind, n, k) in enumerate(w["sizes"]):
        ic, iw = infos[i]
        same = ic["bound2"] / 2.0 ** ic["frac_bits"] == iw["bound2"] / 2.0 ** iw["frac_bits"]
        assert same, (ic, iw)
        rows.append({"instance": f"{kind} n={n} k={k}", "cold_ms": statistics.median(per[i]["cold"]),
                     "warm_ms": statistics.median(per[i]["warm"]), "network_ms": statistics.median(per[i]["net"]),
                     "cold_sweeps": ic["iterations"], "warm_sweeps": iw["iterations"],
                     "cold_phases": ic["phases"], "warm_phases": iw["phases"], "same_optimum": same})
    # end to end through the ABI with host buffers: create, warm start, solve,
    # read back into the caller's pinned buffers (allocated once per instance)
    e2e = 0.0
    h2d = d2h = 0
    for i, d in enumerate(ds):
        nd = len(d["row_ptr"]) - 1
        cap = infos[i][1]["nnz"] * 9 // 8 + 1024
        out_x = (torch.empty(nd + 1, dtype=torch.int32).pin_memory(), torch.empty(cap, dtype=torch.int32).pin_memory(),
                 torch.empty(cap, dtype=torch.uint8).pin_memory(), torch.empty(cap, dtype=torch.int32).pin_memory())
        out_lam = torch.empty(nd, dtype=torch.int32).pin_memory()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ctx = f2m.f2m_create(d["xy"], d["row_ptr"], d["col"], params=params, stream=stream)
        f2m.f2m_warm_start(ctx, m)
        f2m.f2m_solve(ctx)
        res_x = f2m.f2m_get_x(ctx, out=out_x)
        lam_o, _ = f2m.f2m_get_lambda(ctx, out=out_lam)
        torch.cuda.synchronize()
        e2e += (time.perf_counter() - t0) * 1e3
        h2d += d["xy"].nbytes + d["row_ptr"].nbytes + d["col"].nbytes
        d2h += sum(t.numel() * t.element_size() for t in (*res_x, lam_o))
        f2m.f2m_destroy(ctx)
    e2e = max_over_ranks(dist, e2e)
    line = {"metric": METRIC + " (learned warm start, sum over the instances)", "value": warm_ms, "unit": "ms",
            "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "ms_per_step": warm_ms + cold_ms,
            "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "int32",
            "data": "synthetic",
            "config": {"workload": workload_name(w), "l2": "flushed before every solve (256 MB device write)",
                       "max_iters": int(params.max_iters), "parallelism": f"replicas x{world}"},
            "cold_start_ms": cold_ms, "instances": rows,
            "e2e": {"value": e2e, "unit": "ms", "h2d_bytes_per_step": int(h2d), "d2h_bytes_per_step": int(d2h)},
            "clocks": clk, "gpu_launches": int(launches)}
    if rank == 0:
        print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()
    return 0


def finisher_flag(f2m, args):
    fl = {"host": 0, "gpu": f2m.F2M_FLAG_FINISHER_GPU}[args.finisher]
    return fl | (f2m.F2M_FLAG_PRICING_TENSOR if args.pricing_tensor else 0)


def load_traffic(workload):
    """DRAM bytes per launch from the committed ncu summary, if any."""
    p = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        return json.load(open(p)).get(workload, {})
    except Exception:
        return {}


if __name__ == "__main__":
    sys.exit(main())
