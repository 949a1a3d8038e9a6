"""Benchmark of the t-SGNE layout loop on GB300.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Workload (the paper-scale single layout): stochastic block model with 300,000
nodes in 50 Zipf(1.2)-sized blocks, 1,000,000 edges before 10 % are rewired
at random, a 128-d embedding of block centres plus noise, perplexity 30,
exact all-pairs repulsion.  One step = one t-SGNE iteration (attraction over
P, all-pairs repulsion with FP64 Z, gains / momentum update) through
``tsgne_step``.  The affinity build runs once before the timed region and is
reported as ``build_ms``.

Printed: one JSON line (rank 0).  ``value`` = iterations/s over the K timed
steps (device time, CUDA events on the library's stream, L2 flushed before
every step); ``e2e`` = the same metric for a whole layout through the C ABI
from pinned host buffers (build from host CSR + X, K_e2e iterations, layout
copied back), copies inside the timed region; ``roofline`` = the repulsion
kernel (the dominant one) against the FP32 ALU peak; ``cpu_baseline`` = the
FP64 oracle timed on a bounded sample of the same workload.

``--impl reference`` times the oracle itself (there is no runnable reference
implementation of the paper) on the host cores, each step a bounded sample of
repulsion rows of the same workload, and prints the same metric.
"""

from __future__ import annotations

import argparse
import hashlib
import json
import os
import re
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import tsgne_synth as synth  # noqa: E402

METRIC = "t-SGNE iters/sec @300K nodes/1M edges (% FP32/HBM roofline); served layouts/s + p50/p99"
UNIT = "iters/s"
WORKLOAD = "zipf300k"
WORKLOADS = ("zipf300k", "zipf100k", "sbm2k")
WORKLOAD_DESC = ("stochastic block model, 300,000 nodes, 50 Zipf(1.2) blocks, 1,000,000 edges before 10% rewiring, "
                 "128-d FP32 embedding (block centre N(0,4I) + N(0,I)), perplexity 30, Y0 ~ N(0,1e-4^2), "
                 "exact all-pairs repulsion, FP32 with FP64 Z")
# FP32 ALU peak of GB300: 152 SMs x 128 FP32 lanes x 2 flop (FMA) x 2.07 GHz max SM clock
FP32_PEAK_TFLOPS = 152 * 128 * 2 * 2.070e9 / 1e12
FLOPS_PER_UNORDERED_PAIR = 16  # 2 sub, 3 for d^2+1, w^2, Z add, 8 for the two force FMAs pairs
# sources of the dominant (symmetric repulsion) kernel; the committed DRAM
# traffic figure is used only if it was captured on exactly these sources
REPULSION_SRCS = [os.path.join(ROOT, "paper_2310_11186_gb300", "csrc", f)
                  for f in ("repulsion_sym.cu", "sym_unit.cuh", "f32x2.cuh", "zsum.cuh")]
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "repulsion_zipf300k.md")
PIPES_FILE = os.path.join(ROOT, "profiles", "repulsion_sym_zipf100k_full.md")


def repulsion_source_sha() -> str:
    h = hashlib.sha256()
    for f in REPULSION_SRCS:
        h.update(open(f, "rb").read())
    return h.hexdigest()


def log(*a):
    print(*a, file=sys.stderr, flush=True)


# ------------------------------------------------------------------ helpers

class ClockSampler:
    """Samples nvidia-smi clocks / throttle reasons while running."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
              "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
              "clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        self.lines = []
        self.t = None

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "100"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except Exception:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *exc):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
            if self.t:
                self.t.join(timeout=2)

    def summary(self):
        sm, mx, pw, reasons = [], [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 8:
                continue
            try:
                sm.append(float(parts[0]))
                mx.append(float(parts[1]))
                pw.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[4:8]):
                if v.lower() == "active":
                    reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": 0}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "power_w_max": max(pw),
                "reasons": sorted(reasons), "samples": len(sm)}


def traffic_per_launch():
    """DRAM bytes per repulsion launch from the committed ncu summary, if it was
    taken on the current kernel source (else None)."""
    try:
        txt = open(TRAFFIC_FILE).read()
    except OSError:
        return None
    m_sha = re.search(r"source_sha256:\s*([0-9a-f]{64})", txt)
    m_b = re.search(r"traffic_bytes_per_launch:\s*([0-9.eE+]+)", txt)
    if not m_sha or not m_b:
        return None
    return float(m_b.group(1)) if repulsion_source_sha() == m_sha.group(1) else None


ATTRACT_SRCS = [os.path.join(ROOT, "paper_2310_11186_gb300", "csrc", f)
                for f in ("attract_plan.cu", "row_update.cuh", "storage.cuh", "zsum.cuh")]
ATTRACT_TRAFFIC_FILE = os.path.join(ROOT, "profiles", "attract_rmat21.md")


def attraction_traffic():
    """DRAM bytes per attraction+update launch at R-MAT 2^21 from the
    committed ncu summary, if it was taken on the current kernel source."""
    try:
        txt = open(ATTRACT_TRAFFIC_FILE).read()
    except OSError:
        return None
    m_sha = re.search(r"source_sha256:\s*([0-9a-f]{64})", txt)
    m_b = re.search(r"traffic_bytes_per_launch:\s*([0-9.eE+]+)", txt)
    if not m_sha or not m_b:
        return None
    h = hashlib.sha256()
    for f in ATTRACT_SRCS:
        h.update(open(f, "rb").read())
    return float(m_b.group(1)) if h.hexdigest() == m_sha.group(1) else None


def pipe_utilisation():
    """FMA / MUFU pipe activity of the repulsion kernel from the committed ncu
    summary (--set full on the 100K case), if it was taken on the current
    kernel source (else None)."""
    try:
        txt = open(PIPES_FILE).read()
    except OSError:
        return None
    m_sha = re.search(r"source_sha256:\s*([0-9a-f]{64})", txt)
    m_f = re.search(r"fma_pipe_active_pct:\s*([0-9.]+)", txt)
    m_x = re.search(r"xu_pipe_active_pct:\s*([0-9.]+)", txt)
    if not (m_sha and m_f and m_x) or repulsion_source_sha() != m_sha.group(1):
        return None
    return {"fma_pipe_active_pct": float(m_f.group(1)), "mufu_pipe_active_pct": float(m_x.group(1)),
            "target_fma_pct": 60.0, "source": os.path.relpath(PIPES_FILE, ROOT)}


def oracle_sample(Y, n, target_s: float, threads: int = 1):
    """Times the FP64 oracle's repulsion rows on a growing row block (split
    over `threads` host threads) until the sample takes about target_s;
    returns (seconds per iteration extrapolated to all n rows, rows timed,
    seconds spent)."""
    import oracle

    oracle.build()
    Yd = np.ascontiguousarray(Y, np.float64)
    rows = 16 * threads
    spent = 0.0
    while True:
        t = time.perf_counter()
        if threads == 1:
            oracle.repulsion_rows(Yd, 0, rows)
        else:
            oracle.repulsion_all(Yd, threads=threads, i0=0, i1=rows)
        dt = time.perf_counter() - t
        spent += dt
        if dt >= target_s or rows >= n:
            return dt * n / rows, rows, spent
        rows = min(n, int(rows * max(2.0, min(16.0, 1.2 * target_s / max(dt, 1e-4)))))


def aggregate_ranks(local_seconds: float, units_per_rank: float):
    """Whole-job throughput of N replicas: every rank's units over the slowest
    rank's time (max over ranks; no collective when running alone).
    Returns (max_seconds, units_per_second)."""
    import torch
    import torch.distributed as dist

    ws = dist.get_world_size() if dist.is_available() and dist.is_initialized() else 1
    t = local_seconds
    if ws > 1:
        dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
        tt = torch.tensor([local_seconds], dtype=torch.float64, device=dev)
        dist.all_reduce(tt, op=dist.ReduceOp.MAX)
        t = float(tt.item())
    return t, ws * units_per_rank / t


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


# --------------------------------------------------------------- reference

def run_reference(args):
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    g, X = synth.workload(args.workload)
    Y = synth.y_init(g.n)
    import oracle

    oracle.build()
    cores = os.cpu_count() or 1
    # size one step (a block of repulsion rows over all host cores) to about
    # ref_step_seconds of CPU time
    per_iter, _, _ = oracle_sample(Y, g.n, 0.5, threads=cores)
    rows = int(min(g.n, max(16 * cores, g.n * args.ref_step_seconds / per_iter)))
    Yd = np.ascontiguousarray(Y, np.float64)
    for _ in range(args.warmup):
        oracle.repulsion_all(Yd, threads=cores, i0=0, i1=rows)
    times = []
    for _ in range(args.steps):
        t = time.perf_counter()
        oracle.repulsion_all(Yd, threads=cores, i0=0, i1=rows)
        times.append(time.perf_counter() - t)
    step_s = statistics.mean(times)
    frac = rows / g.n  # one step is this fraction of an iteration's repulsion
    value = frac / step_s
    sample = (f"FP64 oracle repulsion rows 0..{rows} of {g.n} (F_rep and row Z sums, {rows * g.n:.3g} pair "
              f"evaluations per step = {frac:.4f} of an iteration), rows split over {cores} host threads; "
              f"value = iterations/s = that fraction / the measured step time")
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": step_s * 1e3,
        "iteration_fraction_per_step": frac, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": args.workload, "description": WORKLOAD_DESC if args.workload == WORKLOAD else
                   args.workload, "nodes": g.n, "edges": g.m // 2},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


# -------------------------------------------------------------------- ours

def run_ours(args):
    import torch

    import paper_2310_11186_gb300 as pkg
    from paper_2310_11186_gb300 import build as pbuild
    from paper_2310_11186_gb300 import quality

    ws, rank, local = dist_env()
    if ws > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    pbuild.build()
    pkg.lib()

    t0 = time.perf_counter()
    g, X = synth.workload(args.workload, seed=args.seed)
    Y0 = synth.y_init(g.n, seed=args.seed)
    log(f"[bench] workload {WORKLOAD}: n={g.n} edges={g.m // 2} ({time.perf_counter() - t0:.1f}s)")

    # ---- device-timed iterations (profile mode: per-kernel CUDA events).
    # With several ranks the one layout's repulsion units are divided over
    # them (strong scaling) and summed by an NCCL all-reduce each iteration.
    if ws > 1:
        from paper_2310_11186_gb300 import shard

        slay = shard.ShardedLayout(profile=1)
        lay = slay.layout
        step = slay.step
        build = slay.build_P
    else:
        slay = None
        lay = pkg.Layout(profile=1)
        step = lay.step
        build = lay.build_P
    s = lay.stream
    tb = time.perf_counter()
    build(g.row_ptr, g.col, X)
    build_ms = (time.perf_counter() - tb) * 1e3
    lay.init_Y(Y0)
    # the library's autotuner over the exact pass's shapes (symmetric 1 or 2
    # warps x 8 or 16 i-points per lane, or the ordered-pair kernel); the
    # sharded path keeps the symmetric default
    tune = None
    if ws == 1 and not args.no_autotune:
        chosen, tms = lay.autotune(3)
        tune = {"chosen": {"tile_warps": chosen[0], "i_per_lane": chosen[1], "symmetric": bool(chosen[2])},
                "ms_per_pass": tms}
        log(f"[bench] autotune: {chosen} {tms}")
    shape = lay.repulsion_shape()
    for _ in range(args.warmup):
        step()
    lay.sync()
    lay.kernel_times(reset=True)
    flush = torch.empty(320 * 2 ** 20 // 4, dtype=torch.float32, device="cuda")  # > 129 MB L2
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    if ws > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    with ClockSampler(local) as clk:
        for k in range(args.steps):
            with torch.cuda.stream(s):
                flush.fill_(float(k))
            starts[k].record(s)
            step()
            ends[k].record(s)
        lay.sync()
        torch.cuda.synchronize()
    if ws > 1:
        torch.distributed.barrier()
    step_ms = [a.elapsed_time(b) for a, b in zip(starts, ends)]
    total_s = sum(step_ms) / 1e3
    kt = lay.kernel_times(reset=True)
    # kernel launches in the timed region: one per timed section, plus the L2
    # prefetch of the layout that the attraction section issues before its
    # kernel when the (FP32) layout holds at least 1 MiB
    launches = sum(v[1] for v in kt.values()) + (kt["attract_update"][1] if 8 * g.n >= 1 << 20 else 0)
    rep_ms = kt["repulsion"][0] / max(kt["repulsion"][1], 1)
    upd_ms = kt["attract_update"][0] / max(kt["attract_update"][1], 1)
    n = g.n
    flops = FLOPS_PER_UNORDERED_PAIR * n * (n - 1) / 2.0
    achieved = flops / (rep_ms / 1e3) / 1e12
    Yt = lay.get_Y()
    nnz_P = lay.sizes()[1]
    lay.close()

    total_s, value = aggregate_ranks(total_s, args.steps)
    if ws > 1:
        value = args.steps / total_s  # one layout: iterations/s, not a sum over replicas

    # ---- end to end: whole layout from pinned host buffers through the C ABI
    e2e_iters = args.e2e_iters
    rp_h = torch.from_numpy(g.row_ptr).pin_memory()
    col_h = torch.from_numpy(g.col).pin_memory()
    X_h = torch.from_numpy(X).pin_memory()
    Y0_h = torch.from_numpy(Y0).pin_memory()
    Y_out = torch.empty((n, 2), dtype=torch.float32).pin_memory()
    lay2 = shard.ShardedLayout() if ws > 1 else pkg.Layout()
    torch.cuda.synchronize()
    if ws > 1:
        torch.distributed.barrier()
    te = time.perf_counter()
    lay2.build_P(rp_h, col_h, X_h)
    lay2.init_Y(Y0_h)
    lay2.run(e2e_iters)
    lay2.get_Y(Y_out)
    e2e_s, _ = aggregate_ranks(time.perf_counter() - te, e2e_iters)
    kl_final = lay2.kl()
    lay2.close()
    # the paper's embedding step: ShortestPath to 128 random targets (Sec. 2.3)
    targets = (synth.splitmix64(args.seed, 5, 0, 128) % np.uint64(n)).astype(np.int32)
    pkg.tsgne_shortest_path_embedding(g.row_ptr, g.col, targets)  # warm
    ts = time.perf_counter()
    pkg.tsgne_shortest_path_embedding(g.row_ptr, g.col, targets)
    sp_s = time.perf_counter() - ts
    h2d = rp_h.numel() * 8 + col_h.numel() * 4 + X_h.numel() * 4 + Y0_h.numel() * 4
    d2h = Y_out.numel() * 4
    Yf = Y_out.numpy()
    labels = g.labels
    q_nmi = quality.layout_nmi(Yf, labels, restarts=2)
    q_aq = quality.aq(Yf, labels)

    # ---- CPU baseline: the FP64 oracle on a bounded sample (rank 0 only)
    cpu = None
    if rank == 0 and not args.no_cpu_baseline:
        cores = os.cpu_count() or 1
        per_iter, rows, spent = oracle_sample(Yt, n, args.cpu_seconds / 2, threads=cores)
        per_iter1, rows1, spent1 = oracle_sample(Yt, n, args.cpu_seconds / 2, threads=1)
        cpu = {"value": 1.0 / per_iter, "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": (f"FP64 oracle repulsion rows 0..{rows} of {n} at the timed layout, rows split over "
                          f"{cores} host threads ({rows * n:.3g} pair evaluations, {spent:.1f} s), "
                          f"extrapolated to all rows"),
               "single_thread": {"value": 1.0 / per_iter1, "rows": rows1, "seconds": spent1}}

    batched = None
    serving = None
    if rank == 0 and not args.no_batched:
        batched = bench_batched(args, pkg)
    if rank == 0 and not args.no_serving:
        serving = bench_serving(args, pkg)
    rmat_res = bench_rmat(args, pkg) if (rank == 0 and not args.no_rmat) else None
    tree_res = bench_tree(args, pkg, g, X, Y0, Yt) if (rank == 0 and not args.no_tree) else None
    rw_res = bench_random_walk(args, pkg, g, X) if (rank == 0 and not args.no_tree) else None
    scale_res = bench_scale(args, pkg) if (rank == 0 and not args.no_scale) else None
    cfg0_res = bench_config0(args, pkg) if (rank == 0 and not args.no_config0) else None

    if rank != 0:
        return 0
    tr = traffic_per_launch()
    clocks = clk.summary()
    line = {
        "metric": METRIC,
        "value": value,
        "unit": UNIT,
        "n_gpus": ws,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": total_s * 1e3 / args.steps,
        "higher_is_better": True,
        "scaling": "strong" if ws > 1 else "weak",
        "vs_baseline": None,
        "dtype": "f32",
        "data": "synthetic",
        "config": {
            "workload": args.workload,
            "description": WORKLOAD_DESC if args.workload == WORKLOAD else args.workload,
            "nodes": n,
            "edges": g.m // 2,
            "nnz_P": int(nnz_P),
            "l2": "flushed (320 MB write) before every timed step",
            "parallelism": (f"one layout over {ws} GPUs: repulsion tile pairs divided, int64 forces and Z "
                            f"partials summed by an NCCL all-reduce per iteration" if ws > 1 else "single GPU"),
            "repulsion_launch": shape,
            "repulsion_autotune": tune,
        },
        "roofline": {
            "bound": "alu",
            "kernel": "repulsion",
            "achieved": achieved,
            "peak": FP32_PEAK_TFLOPS,
            "unit": "TFLOP/s",
            "frac": achieved / FP32_PEAK_TFLOPS,
            "traffic": tr,
            "pipes_ncu": pipe_utilisation(),
            "flops_per_launch": flops,
            "ms_per_launch": rep_ms,
            "peak_source": "152 SMs x 128 FP32 lanes x 2 flop x 2.07 GHz (unit counts and max clock)",
        },
        "roofline_hbm": roofline_hbm(rmat_res, n, nnz_P, upd_ms),
        "kernels_ms_per_step": {"repulsion": rep_ms, "attract_update": upd_ms},
        "cpu_baseline": cpu,
        "e2e": {"value": e2e_iters / e2e_s, "unit": UNIT,
                "h2d_bytes_per_step": h2d / e2e_iters, "d2h_bytes_per_step": d2h / e2e_iters,
                "iters": e2e_iters, "wall_s": e2e_s,
                "note": "build_P from host CSR+X, init_Y from host, run, layout back to host (pinned)"},
        "gpu_launches": launches,
        "clocks": clocks,
        "build_ms": build_ms,
        "shortest_path_embedding": {"ms": sp_s * 1e3, "targets": 128,
                                    "note": "host CSR in, 300000 x 128 distances back to the host"},
        "paper_pipeline_s": {"shortest_path_plus_tsgne": sp_s + e2e_s, "iters": e2e_iters,
                             "paper": "under 5 min (4:57) on a 32-core Xeon Gold 6338, Table 2"},
        "quality": {"kl": kl_final, "nmi": q_nmi, "aq": q_aq, "iters": e2e_iters},
        "serving": serving,
        "batched": batched,
        "rmat": rmat_res,
        "tree": tree_res,
        "random_walk_P": rw_res,
        "scale": scale_res,
        "config0": cfg0_res,
        "paper_context": "300K nodes / 1M edges in under 5 min (ShortestPath + t-SGNE, 32-core Xeon Gold 6338)",
    }
    print(json.dumps(line), flush=True)
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def roofline_hbm(rmat_res, n, nnz, att_ms):
    """The attraction+update kernel (S3+S5, HBM-bound) against the measured
    HBM copy bandwidth: at R-MAT 2^21 (P and its structure larger than L2:
    the measurement) when that section ran, with the 300K benchmark's figure
    beside it for context (its 22 MB mostly stay in L2)."""
    peak, src = hbm_peak()
    b300 = attraction_bytes(n, nnz, 0)
    ctx = {"bytes_per_launch": b300, "ms_per_launch": att_ms,
           "achieved": b300 / (att_ms * 1e-3) / 1e9 if att_ms > 0 else None}
    if rmat_res is None or "fp32" not in rmat_res:
        return {"bound": "hbm", "kernel": "attract_update (S3+S5)", "achieved": ctx["achieved"], "peak": peak,
                "unit": "GB/s", "frac": (ctx["achieved"] / peak) if ctx["achieved"] else None, "traffic": None,
                "peak_source": src, "workload": "zipf300k (R-MAT section skipped)"}
    r = rmat_res["fp32"]["attraction_roofline"]
    return {"bound": "hbm", "kernel": "attract_update (S3+S5)", "achieved": r["achieved"], "peak": peak,
            "unit": "GB/s", "frac": r["achieved"] / peak, "traffic": attraction_traffic(),
            "peak_source": src, "workload": "R-MAT 2^21 nodes / 2^24 edges, FP32",
            "bytes_per_launch": r["bytes_per_launch"], "ms_per_launch": r["ms_per_launch"],
            "zipf300k_context": ctx}


def bench_config0(args, pkg, log_fn=log):
    """Config 0 (the 2,000-node SBM, 1,000 iterations, exact repulsion): the
    whole layout on the GPU (tsgne_run) and in the FP64 oracle (one host
    thread, the whole run), their final KL against the stated 1e-3
    tolerance, and the paper's two quality measures for both layouts."""
    import torch
    import oracle
    from paper_2310_11186_gb300 import quality

    iters = 1000
    g, X = synth.workload("sbm2k")
    Y0 = synth.y_init(g.n, seed=0)
    with pkg.Layout() as warm:  # graph capture and module load outside the timed run
        warm.build_P(g.row_ptr, g.col, X)
        warm.init_Y(Y0)
        warm.run(10)
    with pkg.Layout() as lay:
        lay.build_P(g.row_ptr, g.col, X)
        lay.init_Y(Y0)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        lay.run(iters)
        gpu_s = time.perf_counter() - t0
        Yg = lay.get_Y()
        kl = lay.kl()
    rp, col, P = oracle.build_P(g.n, g.row_ptr, g.col, X, 30.0)
    t0 = time.perf_counter()
    Yo, _, _ = oracle.optimize(g.n, rp, col, P, Y0.astype(np.float64), iters)
    cpu_s = time.perf_counter() - t0
    okl, _ = oracle.kl(g.n, rp, col, P, Yo)
    out = {
        "workload": "stochastic block model, 2,000 nodes, 10 blocks, p_in 0.05, p_out 0.0005, 128-d X, "
                    "perplexity 30, Y0 ~ N(0, 1e-4^2), exact repulsion",
        "iters": iters,
        "gpu": {"seconds": gpu_s, "iters_per_s": iters / gpu_s, "kl": kl,
                "nmi": quality.layout_nmi(Yg, g.labels, restarts=2), "aq": quality.aq(Yg, g.labels)},
        "oracle": {"seconds": cpu_s, "iters_per_s": iters / cpu_s, "cores": 1, "kl": okl,
                   "nmi": quality.layout_nmi(Yo, g.labels, restarts=2), "aq": quality.aq(Yo, g.labels)},
        "kl_rel_diff": abs(kl - okl) / okl,
        "kl_tolerance": 1e-3,
    }
    log_fn(f"[bench] config 0: GPU {iters} it in {gpu_s:.3f} s, oracle {cpu_s:.1f} s; KL {kl:.5f} vs {okl:.5f} "
           f"(rel {out['kl_rel_diff']:.1e})")
    return out


def bench_tree(args, pkg, g, X, Y0, Yt, log_fn=log):
    """The tree-code repulsion (an approximation beyond the paper's exact sum)
    on the same workload: device-timed steps, a whole 1,000-iteration layout,
    and its distance from the exact path (gradient at the timed layout, KL of
    the final layouts both scored exactly)."""
    import torch

    theta = args.tree_theta
    lay = pkg.Layout(profile=1, repulsion=1, theta=theta)
    lay.build_P(g.row_ptr, g.col, X)
    lay.init_Y(Y0)
    for _ in range(args.warmup):
        lay.step()
    lay.sync()
    lay.kernel_times(reset=True)
    flush = torch.empty(320 * 2 ** 20 // 4, dtype=torch.float32, device="cuda")
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    torch.cuda.synchronize()
    ms = 0.0
    for k in range(args.steps):
        with torch.cuda.stream(lay.stream):
            flush.fill_(float(k))
        ev[0].record(lay.stream)
        lay.step()
        ev[1].record(lay.stream)
        ev[1].synchronize()
        ms += ev[0].elapsed_time(ev[1])
    kt = lay.kernel_times(reset=True)
    # gradient, tree vs exact, at a spread layout (block centres N(0, 30^2 I),
    # the scale of a converged layout) and at the exact path's timed layout
    Ysp = synth.spread_layout(g.labels, scale=30.0, seed=args.seed + 1)
    lay.set_state(Ysp)
    Gt, Zt = lay.gradient(1.0)
    lay.set_state(Yt)
    Gt2, Zt2 = lay.gradient(1.0)
    lay.close()
    with pkg.Layout() as ex:
        ex.build_P(g.row_ptr, g.col, X)
        ex.set_state(Ysp)
        Ge, Ze = ex.gradient(1.0)
        ex.set_state(Yt)
        Ge2, Ze2 = ex.gradient(1.0)
        # whole layout with the tree code, then scored by the exact KL
        with pkg.Layout(repulsion=1, theta=theta) as lt:
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            lt.build_P(g.row_ptr, g.col, X)
            lt.init_Y(Y0)
            lt.run(args.e2e_iters)
            Yf = lt.get_Y()
            wall = time.perf_counter() - t0
        ex.init_Y(Yf)
        kl_tree = ex.kl()

    def per(name):
        return kt[name][0] / max(kt[name][1], 1)

    out = {
        "theta": theta,
        "iters_per_s": args.steps / (ms / 1e3),
        "ms_per_step": ms / args.steps,
        "kernels_ms_per_step": {"tree_build": per("tree_build"), "tree_walk": per("repulsion"),
                                "attract_update": per("attract_update")},
        "grad_rel_l2_vs_exact": float(np.linalg.norm(Gt - Ge) / np.linalg.norm(Ge)),
        "Z_rel_vs_exact": abs(Zt - Ze) / Ze,
        "error_layout": "spread layout: block centres N(0, 30^2 I) plus N(0, I) per point",
        "at_timed_layout": {"grad_rel_l2_vs_exact": float(np.linalg.norm(Gt2 - Ge2) / np.linalg.norm(Ge2)),
                            "Z_rel_vs_exact": abs(Zt2 - Ze2) / Ze2,
                            "layout": f"the exact path's layout after {args.warmup + args.steps} iterations"},
        "layout_s": wall,
        "layout_iters": args.e2e_iters,
        "kl_exact_of_tree_layout": kl_tree,
        "note": ("approximate repulsion (not the paper's exact Eq. 4 sum); parity: the exact sums under the "
                 "derived per-row error bound of the monopole approximation"),
    }
    log_fn(f"[bench] tree theta={theta}: {out['iters_per_s']:.1f} it/s, build {out['kernels_ms_per_step']['tree_build']:.3f} ms, "
           f"walk {out['kernels_ms_per_step']['tree_walk']:.3f} ms, grad err {out['grad_rel_l2_vs_exact']:.2e}")
    return out


def bench_random_walk(args, pkg, g, X, log_fn=log):
    """One-time cost of the random-walk estimate of P (Eq. 6) on the same
    graph, next to the perplexity bisection's, and the size of the P it
    produces (walk pairs reach beyond the graph's edges)."""
    import torch

    out = {"walks": args.rw_walks, "length": args.rw_length}
    for name, cfg in (("bisection", {}), ("random_walk", {"p_walks": args.rw_walks,
                                                          "p_walk_length": args.rw_length})):
        with pkg.Layout(**cfg) as lay:
            lay.build_P(g.row_ptr, g.col, X)  # warm (allocations, module load)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            lay.build_P(g.row_ptr, g.col, X)
            out[name] = {"build_ms": (time.perf_counter() - t0) * 1e3, "nnz_P": int(lay.sizes()[1])}
    log_fn(f"[bench] P build: bisection {out['bisection']['build_ms']:.1f} ms, random walks "
           f"{out['random_walk']['build_ms']:.1f} ms (nnz {out['random_walk']['nnz_P']})")
    return out


def bench_scale(args, pkg, log_fn=log):
    """Whole layouts at the sizes of the paper's largest graphs with the
    tree-code repulsion, end to end from pinned host buffers: P build,
    1,000 iterations, layout back to the host."""
    import torch

    cases = (("zipf3m", "3,000,000 nodes, 200 Zipf(1.2) blocks, 4.94M edges (10 % rewired), 64-d X",
              "LFR 3M / 4,937,941 edges: t-SGNE 0:49:02 on an 8-core Apple M2 (context)"),
             ("zipf4m", "3,997,962 nodes, 500 Zipf(1.2) blocks, 34.7M edges (10 % rewired), 32-d X",
              "LiveJournal 3,997,962 / 34,681,189 edges: t-SGNE 2:05:51 on an 8-core Apple M2 (context)"))
    out = {}
    for name, desc, paper in cases:
        t0 = time.perf_counter()
        g, X = synth.workload(name, seed=args.seed)
        log_fn(f"[bench] scale {name}: n={g.n} edges={g.m // 2} ({time.perf_counter() - t0:.1f}s)")
        rp_h = torch.from_numpy(g.row_ptr).pin_memory()
        col_h = torch.from_numpy(g.col).pin_memory()
        X_h = torch.from_numpy(X).pin_memory()
        Y_out = torch.empty((g.n, 2), dtype=torch.float32).pin_memory()
        with pkg.Layout(repulsion=1, theta=args.tree_theta) as lay:
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            lay.build_P(rp_h, col_h, X_h)
            tb = time.perf_counter()
            lay.init_Y(None)
            lay.run(args.e2e_iters)
            lay.get_Y(Y_out)
            t1 = time.perf_counter()
            kl = lay.kl()
        out[name] = {"workload": f"{name}: {desc}, perplexity 30", "theta": args.tree_theta,
                     "iters": args.e2e_iters, "build_P_s": tb - t0, "layout_s": t1 - t0,
                     "iters_per_s": args.e2e_iters / (t1 - tb), "kl_tree_Z": kl, "paper": paper}
        log_fn(f"[bench] scale {name}: build {tb - t0:.2f} s, layout {t1 - t0:.2f} s "
               f"({out[name]['iters_per_s']:.0f} it/s)")
        del g, X, rp_h, col_h, X_h, Y_out
    return out


def bench_batched(args, pkg, log_fn=log):
    """256 block-model graphs advanced together (one batch, autotuned tile)
    against one context per graph run one after the other."""
    import time as _t

    graphs = synth.sbm_mixed_batch(args.batch_graphs, 500, 50_000, 4, 12, 5, 40, 64, seed=args.seed)
    Y0s = [synth.y_init(g.n, seed=args.seed * 7919 + k) for k, (g, _) in enumerate(graphs)]
    n_tot = sum(g.n for g, _ in graphs)
    pairs = sum(0.5 * g.n * (g.n - 1) for g, _ in graphs)
    log_fn(f"[bench] batched: {len(graphs)} graphs, {n_tot} nodes, {pairs:.3g} pairs/iter")
    iters = args.batch_iters
    with pkg.Batch() as b:
        for (g, X), Y0 in zip(graphs, Y0s):
            b.add(g.row_ptr, g.col, X, Y0)
        chosen, tune = b.autotune_shapes(trial_iters=2)
        b.run(2)
        t0 = _t.perf_counter()
        b.run(iters)
        batched_s = (_t.perf_counter() - t0) / iters
    per_graph = 0.0
    for (g, X), Y0 in zip(graphs, Y0s):
        with pkg.Layout() as lay:
            lay.build_P(g.row_ptr, g.col, X)
            lay.init_Y(Y0)
            lay.run(2)
            t0 = _t.perf_counter()
            lay.run(iters)
            per_graph += (_t.perf_counter() - t0) / iters
    L = len(graphs)
    return {
        "workload": (f"{L} stochastic block models, n log-uniform in [500, 50000] (total {n_tot}), mean degree "
                     f"U[4, 12], 5-40 equal blocks, 10% rewired, 64-d embeddings, perplexity 30"),
        "iters_timed": iters,
        "tile_shape": {"tile_warps": chosen[0], "i_per_lane": chosen[1]},
        "autotune_ms_per_iter": tune,
        "batched_ms_per_iter": batched_s * 1e3,
        "one_context_per_graph_ms_per_iter": per_graph * 1e3,
        "speedup": per_graph / batched_s,
        "layouts_per_s_at_1000_iters": {"batched": L / (1000 * batched_s), "one_per_graph": L / (1000 * per_graph)},
        "pairs_per_s_batched": pairs / batched_s,
        "note": "wall-clock per iteration after warm-up, both arms synchronised; layouts/s = members / (1000 x s/iter)",
    }


def bench_serving(args, pkg, log_fn=log):
    """Poisson arrivals of block-model layout requests served by continuous
    batching, against the same trace served one layout at a time."""
    from paper_2310_11186_gb300 import serve

    count = args.serve_requests
    arr = synth.poisson_arrivals(count, args.serve_rate, seed=args.seed + 11)
    ns = synth.log_uniform_ints(count, 1_000, 300_000, seed=args.seed + 12)
    reqs, spec = [], []
    for k in range(count):
        n = int(ns[k])
        blocks = int(min(50, max(5, n // 5000)))
        g = synth.sbm_zipf(n, blocks, 3 * n, zipf_s=0.0, rewire=0.10, seed=args.seed * 1000 + 500 + k)
        X = synth.block_embedding(g.labels, 128, seed=args.seed * 1000 + 500 + k)
        spec.append((g, X))
    mk = lambda: [serve.Request(k, float(arr[k]), spec[k][0].row_ptr, spec[k][0].col, spec[k][1],
                                synth.y_init(spec[k][0].n, seed=k)) for k in range(count)]
    log_fn(f"[bench] serving: {count} requests at {args.serve_rate}/s, n in [{ns.min()}, {ns.max()}]")
    cfg = pkg.tsgne_config_default(theta=args.tree_theta)
    srv = serve.LayoutServer(iters=args.serve_iters, tick_iters=10, budget_bytes=80 * 2 ** 30, tile_warps=2,
                             policy="srpt", config=cfg, tree_min_n=args.serve_tree_min_n)
    try:
        served = srv.serve(mk())
    finally:
        srv.close()
    serial = serve.serial_baseline(mk(), args.serve_iters, config=cfg, tree_min_n=args.serve_tree_min_n)
    n_tree = int((ns >= args.serve_tree_min_n).sum()) if args.serve_tree_min_n > 0 else 0
    # capacity: the same requests all present at time 0 (the offered rate no
    # longer caps the served arm)
    sat = None
    if args.serve_saturated:
        def mk0():
            rs = mk()
            for r in rs:
                r.arrival = 0.0
            return rs
        srv = serve.LayoutServer(iters=args.serve_iters, tick_iters=10, budget_bytes=80 * 2 ** 30, tile_warps=2,
                                 policy="srpt", config=cfg, tree_min_n=args.serve_tree_min_n)
        try:
            sat_served = srv.serve(mk0())
        finally:
            srv.close()
        sat_serial = serve.serial_baseline(mk0(), args.serve_iters, config=cfg, tree_min_n=args.serve_tree_min_n)
        sat = {"note": "every request present at time 0: layouts/s is the capacity of each arm",
               "served": sat_served, "serial_one_at_a_time": sat_serial,
               "speedup": sat_served["layouts_per_s"] / sat_serial["layouts_per_s"]}
        log_fn(f"[bench] serving at saturation: {sat_served['layouts_per_s']:.1f} vs "
               f"{sat_serial['layouts_per_s']:.1f} layouts/s")
    return {
        "workload": (f"{count} requests, Poisson arrivals at {args.serve_rate}/s, stochastic block models with n "
                     f"log-uniform in [1000, 300000], mean degree 6, 128-d embeddings, {args.serve_iters} "
                     f"iterations each, 80 GB admission budget"),
        "policy": ("continuous batching, shortest remaining work first with aging (20 ticks), 1,024-point tiles "
                   "(2 warps)"),
        "repulsion": (f"tree code (theta {args.tree_theta}) for the {n_tree} requests of at least "
                      f"{args.serve_tree_min_n} points, exact pass for the others, in both arms"
                      if args.serve_tree_min_n > 0 else "exact pass for every request"),
        "layouts_per_s": served["layouts_per_s"],
        "p50_s": served["p50_s"],
        "p99_s": served["p99_s"],
        "wall_s": served["wall_s"],
        "offered_per_s": args.serve_rate,
        # an offered rate above what the GPU completes keeps the queue busy for
        # the whole trace, so the completion rate is then the sustainable rate
        "max_sustainable_per_s": (served["layouts_per_s"] if served["layouts_per_s"] < 0.9 * args.serve_rate
                                  else None),
        "serial_one_at_a_time": serial,
        "saturated": sat,
    }


def hbm_peak():
    """Measured HBM copy bandwidth (GB/s) from MEASURED_PEAKS.json, else the fallback figure."""
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return float(json.load(f)["hbm_gbs"]), "measured (MEASURED_PEAKS.json hbm_gbs)"
    except Exception:
        return 6800.0, "fallback 6.8 TB/s"


def attraction_bytes(n, nnz, prec):
    """Algorithmic bytes of one attraction+update launch: row_ptr, col and P
    once; per point F^r, update and gains read, Y_next, update and gains
    written, and Y_i read (FP32: 8 B; BF16: the 4-B shadow for the forces
    plus the 8-B master for the update, and a 4-B shadow write).  Neighbour
    gathers of Y are L2 hits after the first read (the layout is 16.8 MB in
    FP32 at 2^21 points, 8.4 MB in BF16)."""
    if prec == 0:
        return 8 * (n + 1) + 8 * nnz + 7 * 8 * n
    return 8 * (n + 1) + 6 * nnz + 8 * 8 * n


def bench_rmat(args, pkg, log_fn=log):
    """Config 4, R-MAT 2^21 nodes / 2^24 edges.

    Timing: the attraction+update kernel (S3+S5) against the HBM roofline in
    both storage precisions (FP32; BF16 P and Y reads with FP32 arithmetic),
    over --rmat-steps iterations whose repulsion is the tree code (the
    attraction kernel is the same whichever repulsion runs, and tree
    iterations take milliseconds instead of the exact pass's 0.7 s); the
    exact all-pairs repulsion pass is timed separately over --rmat-exact-steps
    iterations.  Error: FP32, BF16 and tree-code arms against the exact FP64
    oracle on the 20K-node induced subgraph (BFS ball from the highest-degree
    node): gradient relative L2, KL and Z."""
    import torch
    import oracle

    t0 = time.perf_counter()
    scale = args.rmat_scale
    g, X = synth.rmat(scale, 1 << (scale + 3), seed=args.seed)
    log_fn(f"[bench] rmat: n={g.n} edges={g.m // 2} max degree {int(np.diff(g.row_ptr).max())} "
           f"({time.perf_counter() - t0:.1f}s)")
    peak, src = hbm_peak()
    flush = torch.empty(320 * 2 ** 20 // 4, dtype=torch.float32, device="cuda")
    out = {
        "workload": f"R-MAT scale {scale} ({1 << scale} nodes), 2^{scale + 3} distinct undirected edges, a=0.57 "
                    f"b=c=0.19, 64-d embedding of 64 recursion communities, perplexity 30",
        "l2": "flushed (320 MB write) before every step",
    }
    # ---- attraction roofline, both precisions (tree-code iterations)
    for prec, name in ((0, "fp32"), (1, "bf16")):
        lay = pkg.Layout(profile=1, precision=prec, repulsion=1, theta=args.tree_theta)
        tb = time.perf_counter()
        lay.build_P(g.row_ptr, g.col, X)
        build_ms = (time.perf_counter() - tb) * 1e3
        n, nnz = lay.sizes()
        lay.init_Y(synth.y_init(n, seed=args.seed))
        for _ in range(3):
            lay.step()
        lay.sync()
        lay.kernel_times(reset=True)
        with ClockSampler(int(os.environ.get("LOCAL_RANK", "0"))) as clk:
            for k in range(args.rmat_steps):
                with torch.cuda.stream(lay.stream):
                    flush.fill_(float(k))
                lay.step()
            lay.sync()
        kt = lay.kernel_times(reset=True)
        lay.close()
        att_ms = kt["attract_update"][0] / kt["attract_update"][1]
        hub_ms = kt["attract_hubs"][0] / max(kt["attract_hubs"][1], 1)
        att_bytes = attraction_bytes(n, nnz, prec)
        achieved = att_bytes / ((att_ms + hub_ms) * 1e-3) / 1e9
        out[name] = {
            "nnz_P": int(nnz),
            "build_ms": build_ms,
            "tree_repulsion_ms": (kt["tree_build"][0] / kt["tree_build"][1] + kt["repulsion"][0] / kt["repulsion"][1]),
            "attraction_roofline": {"bound": "hbm", "kernel": "attract_update (S3+S5)", "achieved": achieved,
                                    "peak": peak, "unit": "GB/s", "frac": achieved / peak, "peak_source": src,
                                    "bytes_per_launch": att_bytes, "ms_per_launch": att_ms + hub_ms,
                                    "launches_timed": int(kt["attract_update"][1]),
                                    "ms_split": {"rows_and_update": att_ms, "hub_row_chunks": hub_ms}},
            "clocks": clk.summary(),
        }
        log_fn(f"[bench] rmat {name}: attraction {att_ms + hub_ms:.3f} ms ({achieved:.0f} GB/s, "
               f"{achieved / peak:.3f} of peak)")
    # ---- the exact repulsion pass at this size (FP32)
    if args.rmat_exact_steps > 0:
        with pkg.Layout(profile=1) as lay:
            lay.build_P(g.row_ptr, g.col, X)
            lay.init_Y(synth.y_init(g.n, seed=args.seed))
            lay.step()
            lay.sync()
            lay.kernel_times(reset=True)
            for _ in range(args.rmat_exact_steps):
                lay.step()
            lay.sync()
            kt = lay.kernel_times(reset=True)
        rep_ms = kt["repulsion"][0] / kt["repulsion"][1]
        fl = FLOPS_PER_UNORDERED_PAIR * g.n * (g.n - 1) / 2.0
        out["fp32"]["exact_repulsion_ms"] = rep_ms
        out["fp32"]["exact_repulsion_tflops"] = fl / (rep_ms * 1e-3) / 1e12
        log_fn(f"[bench] rmat exact repulsion: {rep_ms:.1f} ms ({fl / (rep_ms * 1e-3) / 1e12:.1f} TFLOP/s)")
    # ---- error arms on the 20K-node induced subgraph against the FP64 oracle
    nodes, sub = synth.induced_bfs_ball(g, 20_000)
    Xs = X[nodes]
    Ys = synth.spread_layout(sub.labels, scale=25.0, seed=args.seed)
    orp, ocol, oP = oracle.build_P(sub.n, sub.row_ptr, sub.col, Xs, 30.0)
    oG, oZ = oracle.gradient(sub.n, orp, ocol, oP, Ys.astype(np.float64), 1.0)
    okl, _ = oracle.kl(sub.n, orp, ocol, oP, Ys.astype(np.float64))
    errs = {"oracle_subgraph_nodes": int(sub.n), "layout": "spread layout, block centres N(0, 25^2 I)"}
    for prec, rep, name in ((0, 0, "fp32"), (1, 0, "bf16"), (0, 1, f"fp32_tree_theta{args.tree_theta}")):
        with pkg.Layout(precision=prec, repulsion=rep, theta=args.tree_theta) as l2:
            l2.build_P(sub.row_ptr, sub.col, Xs)
            l2.init_Y(Ys)
            G, Z = l2.gradient(1.0)
            kl = l2.kl()
        errs[name] = {"grad_rel_l2": float(np.linalg.norm(G - oG) / np.linalg.norm(oG)),
                      "kl_rel": abs(kl - okl) / okl, "Z_rel": abs(Z - oZ) / oZ}
        log_fn(f"[bench] rmat error {name}: grad {errs[name]['grad_rel_l2']:.2e}, KL {errs[name]['kl_rel']:.2e}")
    out["vs_fp64_oracle_20k"] = errs
    return out


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--seed", type=int, default=0)
    ap.add_argument("--e2e-iters", type=int, default=1000)
    ap.add_argument("--cpu-seconds", type=float, default=10.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--ref-step-seconds", type=float, default=1.0)
    ap.add_argument("--no-batched", action="store_true")
    ap.add_argument("--batch-graphs", type=int, default=256)
    ap.add_argument("--batch-iters", type=int, default=20)
    ap.add_argument("--no-serving", action="store_true")
    ap.add_argument("--serve-requests", type=int, default=200)
    ap.add_argument("--serve-tree-min-n", type=int, default=20000,
                    help="requests of at least this many points use the tree code in both serving arms (0: none)")
    ap.add_argument("--serve-rate", type=float, default=20.0)
    ap.add_argument("--serve-iters", type=int, default=500)
    ap.add_argument("--serve-saturated", type=int, default=1, help="also serve the trace with every request at t=0")
    ap.add_argument("--no-tree", action="store_true", help="skip the tree-code repulsion section")
    ap.add_argument("--no-autotune", action="store_true", help="keep the default shape of the exact pass")
    ap.add_argument("--no-config0", action="store_true",
                    help="skip the 2,000-node, 1,000-iteration layout against the oracle's whole run")
    ap.add_argument("--tree-theta", type=float, default=0.5)
    ap.add_argument("--rw-walks", type=int, default=64)
    ap.add_argument("--rw-length", type=int, default=3)
    ap.add_argument("--no-rmat", action="store_true", help="skip the R-MAT 2^21 section (config 4)")
    ap.add_argument("--rmat-steps", type=int, default=20)
    ap.add_argument("--rmat-exact-steps", type=int, default=2)
    ap.add_argument("--rmat-scale", type=int, default=21)
    ap.add_argument("--only-rmat", action="store_true", help="run only the R-MAT section (profiling)")
    ap.add_argument("--only-tree", action="store_true", help="run only the tree-code section (profiling)")
    ap.add_argument("--only-batched", action="store_true", help="run only the batched section (profiling)")
    ap.add_argument("--no-scale", action="store_true",
                    help="skip the 3M- and 4M-node tree-code layouts (about a minute, most of it building the graphs)")
    ap.add_argument("--workload", choices=WORKLOADS, default=WORKLOAD,
                    help="zipf300k is the benchmark; the others are smaller cases for profiling")
    args = ap.parse_args()
    if args.warmup < 3:
        ap.error("--warmup must be >= 3")
    if args.impl == "reference":
        return run_reference(args)
    if args.only_rmat:
        import torch

        from paper_2310_11186_gb300 import build as pbuild
        import paper_2310_11186_gb300 as pkg

        torch.cuda.set_device(0)
        pbuild.build()
        print(json.dumps({"rmat": bench_rmat(args, pkg)}), flush=True)
        return 0
    if args.only_batched:
        import torch

        from paper_2310_11186_gb300 import build as pbuild
        import paper_2310_11186_gb300 as pkg

        torch.cuda.set_device(0)
        pbuild.build()
        print(json.dumps({"batched": bench_batched(args, pkg)}), flush=True)
        return 0
    if args.only_tree:
        import torch

        from paper_2310_11186_gb300 import build as pbuild
        import paper_2310_11186_gb300 as pkg

        torch.cuda.set_device(0)
        pbuild.build()
        g, X = synth.workload(args.workload, seed=args.seed)
        Y0 = synth.y_init(g.n, seed=args.seed)
        Yt = synth.spread_layout(g.labels, scale=30.0, seed=args.seed)
        print(json.dumps({"tree": bench_tree(args, pkg, g, X, Y0, Yt)}), flush=True)
        return 0
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
