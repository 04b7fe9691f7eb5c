#!/usr/bin/env python
"""Benchmark: time-to-1e-6 rel-KKT on the 100k x 250k general-form LP (2.5M nonzeros,
power-law columns, mixed bounds, planted optimum; lpgen.make_c2(seed=1)).

One step = one complete pass of the hot path on that LP through the C ABI: rhpdhg_create from
device-resident arrays (validation, transpose, Ruiz + Pock-Chambolle scaling, power iteration),
rhpdhg_solve to rel-KKT <= 1e-6 and rhpdhg_poll into device buffers, then rhpdhg_free.
``value`` is the whole-job throughput in LPs solved per second (1 / time-to-tolerance at one
GPU); the e2e figure repeats the step from pinned host buffers, with the host->device copy of
the problem and the device->host copy of (x, y) inside the timed region.

Multi-GPU: the LPs are independent, so each rank solves its own copy (weak scaling, no data-path
collective; a barrier and a max-over-ranks of the timings only).

``--impl reference`` times the FP64 CPU oracle (written from the paper; the only reference
implementation there is) on the host cores instead, on bounded samples of the same workload.
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

# The CPU baseline is the oracle on one core: keep numpy's BLAS and OpenMP pools to one thread
# (unless the caller chose otherwise) so that the reported core count is the one used.
for _v in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
    os.environ.setdefault(_v, "1")

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "time-to-1e-6 rel-KKT, iters/s, HBM GB/s vs peak; batched LPs/s, p50/p99"
UNIT = "LP/s (100k x 250k LP solved to 1e-6 rel-KKT)"
WORKLOAD = ("general-form LP 100k rows (70k =, 30k >=) x 250k cols, 2.5M nnz, power-law "
            "columns (alpha 2.1, max 5000), mixed bounds, planted optimum, seed 1")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--algorithm", type=int, default=1)
    ap.add_argument("--precision", type=int, default=1,
                    help="headline precision: 1 = FP32 iterates / FP64 restarts, 0 = FP64")
    ap.add_argument("--tol", type=float, default=1e-6)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-large", action="store_true",
                    help="skip the 120M-nonzero multicommodity-flow section")
    ap.add_argument("--serve-requests", type=int, default=60,
                    help="requests of the 50/s Poisson stream replayed through the serving loop "
                         "(0 = skip)")
    ap.add_argument("--serve-max-iters", type=int, default=1_000_000)
    return ap.parse_args()


# DRAM bytes (read + write) per launch of the mixed-precision ordinary-iteration kernels on the
# 100k x 250k LP, from one ncu capture (summarised under profiles/) of the kernel sources with
# this digest (their code with comments and whitespace removed).  Reported as roofline.traffic
# only while that code is unchanged.
KERNEL_SOURCES = ["paper_2407_16144_gb300/csrc/iterate_mx.cu", "paper_2407_16144_gb300/csrc/common.cuh",
                  "paper_2407_16144_gb300/csrc/iter_common.cuh", "paper_2407_16144_gb300/csrc/internal.h"]
PROFILED_TRAFFIC = {
    "digest": "ee820081184d1800",
    "column kernel (K^T y~ + primal step)": 27730688,
    "row kernel (K x~ + dual step)": 23919872,
}


def code_text(src: str) -> str:
    """C/C++/CUDA source with comments removed and whitespace runs collapsed (string literals
    kept as they are), so that a digest follows the code only."""
    import re
    tok = re.compile(r'"(?:\\.|[^"\\])*"|/\*.*?\*/|//[^\n]*', re.S)
    out = tok.sub(lambda m: m.group(0) if m.group(0).startswith('"') else " ", src)
    return " ".join(out.split())


def kernel_digest():
    import hashlib
    h = hashlib.sha256()
    for f in KERNEL_SOURCES:
        with open(os.path.join(os.path.dirname(os.path.abspath(__file__)), f)) as fh:
            h.update(code_text(fh.read()).encode())
    return h.hexdigest()[:16]


def load_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons during the timed region."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        sm, smax, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        with open(self.path) as f:
            for line in f:
                parts = [p.strip() for p in line.split(",")]
                if len(parts) < 8:
                    continue
                try:
                    sm.append(float(parts[0]))
                    smax = float(parts[1])
                except ValueError:
                    continue
                for nm, v in zip(names, parts[4:8]):
                    if v.lower() == "active":
                        reasons.add(nm)
        os.unlink(self.path)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": smax, "samples": len(sm),
                "reasons": sorted(reasons)}


def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def replica_max(dist, values, device):
    """Max over ranks of each timed total (replicas: the slowest rank bounds the job)."""
    if dist is None:
        return [float(v) for v in values]
    import torch
    t = torch.tensor([float(v) for v in values], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(v) for v in t.tolist()]


def replica_throughput(world, units_per_rank, max_ms):
    """Whole-job rate of `world` independent replicas that each ran `units_per_rank` units in
    at most `max_ms` milliseconds (weak scaling)."""
    return world * units_per_rank / (max_ms / 1000.0)


TUNE_KEYS = ("tuned", "tune_ns_rule", "tune_ns_best", "cta_warps_row", "cta_warps_col",
             "walk_row", "grid_row", "grid_col")


def fp64_flops(lp):
    """Algorithmic FP64 flops of one launch of the FP64 row kernel (K x~ and the dual step) and
    of the column kernel (K^T y~ and the primal step) of r2HPDHG: one FMA (2 flops) per nonzero,
    and the fused elementwise work per row (reflected blends of y and K x, the dual step and
    projection, the three restart-test sums: 23 flops) and per column (blends of x and K^T y,
    the primal step and clamp, two sums: 19 flops)."""
    return 2.0 * lp.nnz + 23.0 * lp.m, 2.0 * lp.nnz + 19.0 * lp.n


def problem_bytes(lp):
    return (8 * (lp.m + 1) + 12 * lp.nnz + 8 * (3 * lp.n) + 8 * lp.m)


def cpu_oracle_sample(lp, algorithm, tol, iters_to_tol, sample_iters=100):
    """Times the FP64 oracle on the host: set-up (scaling + power iteration) plus
    ``sample_iters`` iterations; the time to tolerance is extrapolated with ``iters_to_tol``."""
    from oracle import rhpdhg_oracle as O
    t0 = time.perf_counter()
    K = O.csr_matrix(lp)
    Kh, D, E = O.scale_problem(K, 10, 1.0)
    O.power_sigma_max(Kh, 100)
    setup = time.perf_counter() - t0
    r = O.solve(lp, O.OracleParams(algorithm=algorithm, eps_rel_kkt=tol,
                                   max_iters=sample_iters))
    per_iter = (r.solve_seconds - setup) / sample_iters
    per_iter = max(per_iter, 1e-9)
    t_tol = setup + iters_to_tol * per_iter
    return dict(setup_s=setup, s_per_iter=per_iter, time_to_tol_s=t_tol,
                value=1.0 / t_tol, wall_s=time.perf_counter() - t0)


def sgm10(times):
    import math
    return math.exp(sum(math.log(t + 10.0) for t in times) / len(times)) - 10.0


def run_serving(args, rhpdhg, lpgen):
    """Replays a prefix of the serving stream (Poisson arrivals at 50/s, m log-uniform in
    [100, 200k], n = 2.5 m, C1 structure, tolerance 1e-4 or 1e-6 each) through the serving loop in
    mixed precision (FP32 iterates and matrix values, FP64 restarts and checks; LPs with at most
    small_nnz nonzeros become batched slots, larger ones get their own handle and stream), and,
    for comparison, through the plain FP64 single-LP path one request at a time."""
    import threading
    import numpy as np
    nreq = args.serve_requests
    reqs = lpgen.make_batch_stream(4, count=nreq)
    lps = [lpgen.make_standard_planted(seed=r["seed"], m=r["m"], n=r["n"]) for r in reqs]
    small_nnz = 20_000
    cap = args.serve_max_iters
    limit_s = 120.0
    results = {}
    with rhpdhg.Server(150 << 30, small_nnz=small_nnz, max_slots=256, iters_per_step=64) as srv:
        tick = {}
        start = time.perf_counter()

        def producer():
            for i, (r, lp) in enumerate(zip(reqs, lps)):
                now = time.perf_counter() - start
                if r["arrival_s"] > now:
                    time.sleep(r["arrival_s"] - now)
                tick[i] = srv.submit(lp, eps_rel_kkt=r["tol"], precision=1, max_iters=cap,
                                     time_limit_s=limit_s)

        th = threading.Thread(target=producer)
        th.start()
        while len(results) < nreq:
            for i in list(tick.keys()):
                if i not in results:
                    out = srv.poll(tick[i])
                    if out is not None:
                        results[i] = out
            time.sleep(0.0005)
        th.join()
        makespan = time.perf_counter() - start
        st = srv.stats()
    lat = np.array([results[i][1] for i in range(nreq)])
    solved = sum(results[i][0].status == rhpdhg.STATUS_OPTIMAL for i in range(nreq))
    # the plain FP64 single-LP path: each request alone (create, solve, poll, free), its service
    # time measured; latencies from a FIFO replay of those service times against the same arrivals
    svc, solved_b = [], 0
    for r, lp in zip(reqs, lps):
        t0 = time.perf_counter()
        with rhpdhg.Solver(lp, eps_rel_kkt=r["tol"], precision=0, max_iters=cap,
                           time_limit_s=limit_s) as s:
            rr = s.run()
        svc.append(time.perf_counter() - t0)
        solved_b += rr.status == rhpdhg.STATUS_OPTIMAL
    fin, lat_b = 0.0, []
    for r, sv in zip(reqs, svc):
        st_ = max(fin, r["arrival_s"])
        fin = st_ + sv
        lat_b.append(fin - r["arrival_s"])
    lat_b = np.array(lat_b)
    return {
        "workload": f"first {nreq} requests of the stream: Poisson arrivals at 50/s, m log-uniform "
                    "in [100, 200k], n = 2.5 m, 5 nnz per column, planted optimum, tol 1e-4 or "
                    f"1e-6 (seed 4); at most {cap} iterations and {limit_s:.0f} s each",
        "solved_lps_per_s": solved / makespan, "makespan_s": makespan,
        "p50_latency_s": float(np.percentile(lat, 50)),
        "p99_latency_s": float(np.percentile(lat, 99)),
        "sgm10_latency_s": sgm10(list(lat)), "solved": int(solved), "requests": nreq,
        "policy": f"all requests FP32 iterates / FP64 restarts; nnz <= {small_nnz}: batched slots "
                  "(one CTA per LP, one launch for all slots); larger: own handle and stream",
        "admitted_batched": st["admitted_batched"], "admitted_single": st["admitted_single"],
        "peak_bytes_in_use": st["peak_bytes_in_use"],
        "plain_fp64_single_lp": {
            "how": "each request solved alone through the FP64 single-LP path (service time "
                   "measured); arrivals replayed through a simulated FIFO queue of those times",
            "solved_lps_per_s": solved_b / fin, "makespan_s": fin,
            "p50_latency_s": float(np.percentile(lat_b, 50)),
            "p99_latency_s": float(np.percentile(lat_b, 99)),
            "sgm10_latency_s": sgm10(list(lat_b)), "solved": int(solved_b)},
    }


def run_large(args, rhpdhg, lpgen, peak, peak_kind):
    """The 120M-nonzero multicommodity-flow LP to 1e-4 in three precisions (BF16 matrix values,
    FP32 values, FP64), plus one profiled solve of each low-precision mode for the per-kernel
    HBM roofline.  Every handle is created with the autotuner on (its launch-shape choice is
    reported; the profiled handles reuse it from the tuner's cache)."""
    lp = lpgen.make_multicommodity_flow()
    out = {"workload": "multicommodity flow: 20 commodities on 250k nodes / 2M arcs "
                       "(7M rows, 40M columns, 120M nonzeros), arc costs U[1,100], "
                       "capacities U[5,50], planted feasible flow (seed 2)",
           "tol": 1e-4}
    names = {2: "bf16 matrix, fp32 iterates, fp64 restarts", 1: "fp32 iterates, fp64 restarts",
             0: "fp64"}
    for prec in (2, 1, 0):
        t0 = time.perf_counter()
        s = rhpdhg.Solver(lp, algorithm=args.algorithm, precision=prec, eps_rel_kkt=1e-4,
                          time_limit_s=300.0, autotune=1)
        t1 = time.perf_counter()
        r = s.run()
        lay = s.layout()
        s.close()
        out[names[prec]] = {"status": r.status_name, "iters": r.iters, "solve_s": r.solve_seconds,
                            "create_s": t1 - t0, "iters_per_s": r.iters / r.solve_seconds,
                            "rel_kkt": r.rel_kkt, "primal_obj": r.primal_obj,
                            "continued_in_fp64": bool(r.escalated),
                            "autotune": {k: lay.get(k) for k in TUNE_KEYS}}
    out["roofline"] = {"bound": "hbm", "unit": "GB/s", "peak": peak, "peak_kind": peak_kind}
    for prec in (1, 2):
        s = rhpdhg.Solver(lp, algorithm=args.algorithm, precision=prec, eps_rel_kkt=1e-4,
                          profile=1, autotune=1)
        s.run()
        kt = s.kernel_times()
        s.close()
        ach_c = kt["bytes_col"] / (kt["ms_col"] / 1000.0) / 1e9
        ach_r = kt["bytes_row"] / (kt["ms_row"] / 1000.0) / 1e9
        out["roofline"][names[prec]] = {
            "column_kernel": {"achieved": ach_c, "frac": ach_c / peak,
                              "ms_per_launch": kt["ms_col"], "bytes_per_launch": kt["bytes_col"]},
            "row_kernel": {"achieved": ach_r, "frac": ach_r / peak,
                           "ms_per_launch": kt["ms_row"], "bytes_per_launch": kt["bytes_row"]}}
    return out


def run_reference(args):
    world, rank, _ = dist_setup()
    if rank != 0:
        return 0
    from oracle import rhpdhg_oracle as O
    from paper_2407_16144_gb300 import lpgen
    lp = lpgen.make_c2(1)
    # first warm-up step: one full solve, which fixes the oracle's own iteration count
    t0 = time.perf_counter()
    full = O.solve(lp, O.OracleParams(algorithm=args.algorithm, eps_rel_kkt=args.tol,
                                      max_iters=1_000_000))
    full_s = time.perf_counter() - t0
    iters = full.iters
    samples = []
    for i in range(max(args.warmup - 1, 0) + args.steps):
        s = cpu_oracle_sample(lp, args.algorithm, args.tol, iters)
        if i >= max(args.warmup - 1, 0):
            samples.append(s)
    t = statistics.mean(s["time_to_tol_s"] for s in samples)
    # ms_per_step is the measured wall time of a timed step (the bounded sample); value is the
    # time-to-tol rate extrapolated from it, as cpu_baseline.sample says
    step_s = statistics.mean(s["wall_s"] for s in samples)
    line = {
        "impl": "reference", "metric": METRIC, "value": 1.0 / t, "unit": UNIT, "n_gpus": 1,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000.0 * step_s,
        "timed_steps_wall_s": [round(s["wall_s"], 3) for s in samples],
        "value_basis": "1 / (set-up + iterations to 1e-6 x seconds per iteration), both measured "
                       "in each timed step; the iteration count from the warm-up's full solve",
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": WORKLOAD, "tol": args.tol, "algorithm": args.algorithm,
                   "precision": "fp64"},
        "time_to_tol_s": t, "iters": iters, "full_solve_s": full_s,
        "iters_per_s": 1.0 / statistics.mean(s["s_per_iter"] for s in samples),
        "cpu_baseline": {"value": 1.0 / t, "unit": UNIT, "cores": 1, "kind": "oracle",
                         "sample": f"one full oracle solve ({iters} iterations, {full_s:.1f} s) "
                                   f"fixes the iteration count; each step = set-up + 100 "
                                   f"iterations, time-to-tol extrapolated"},
        "e2e": {"value": 1.0 / t, "unit": UNIT, "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


def run_ours(args):
    import numpy as np
    import torch
    from paper_2407_16144_gb300 import _build, lpgen, rhpdhg

    world, rank, local = dist_setup()
    if not torch.cuda.is_available():
        raise RuntimeError("bench.py needs a CUDA GPU")
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    if rank == 0:
        _build.build()
    if dist is not None:
        dist.barrier()
    rhpdhg.load()
    lp = lpgen.make_c2(1)
    dev = lpgen.LP(**{f: (torch.as_tensor(getattr(lp, f), device="cuda")
                          if isinstance(getattr(lp, f), np.ndarray) else getattr(lp, f))
                      for f in ("m_eq", "m_ineq", "n", "row_ptr", "col_idx", "val", "c", "q",
                                "l", "u")})
    pinned = lpgen.LP(**{f: (torch.as_tensor(getattr(lp, f)).pin_memory().numpy()
                             if isinstance(getattr(lp, f), np.ndarray) else getattr(lp, f))
                         for f in ("m_eq", "m_ineq", "n", "row_ptr", "col_idx", "val", "c", "q",
                                   "l", "u")})
    stream = torch.cuda.current_stream()
    sh = stream.cuda_stream
    xo = torch.empty(lp.n, dtype=torch.float64, device="cuda")
    yo = torch.empty(lp.m, dtype=torch.float64, device="cuda")
    xh = torch.empty(lp.n, dtype=torch.float64).pin_memory().numpy()
    yh = torch.empty(lp.m, dtype=torch.float64).pin_memory().numpy()
    flush = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")   # > 129 MB L2
    params = dict(algorithm=args.algorithm, precision=args.precision, eps_rel_kkt=args.tol,
                  autotune=1)

    layouts = []

    def step_device():
        s = rhpdhg.Solver(dev, device=True, stream=sh, **params)
        s.solve(1)
        r = s.poll(x=xo, y=yo, out_memory=rhpdhg.MEM_DEVICE)
        nl = s.launch_count()
        layouts.append(s.layout())
        s.close()
        return r, nl

    def step_host():
        s = rhpdhg.Solver(pinned, stream=sh, **params)
        s.solve(1)
        r = s.poll(x=xh, y=yh)
        s.close()
        return r

    def timed(fn, k):
        out, ms = [], []
        for _ in range(k):
            flush.zero_()
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            o = fn()
            e1.record(stream)
            e1.synchronize()
            ms.append(e0.elapsed_time(e1))
            out.append(o)
        return out, ms

    for _ in range(args.warmup):
        step_device()
    if dist is not None:
        dist.barrier()
    torch.cuda.synchronize()
    clocks = ClockSampler(torch.cuda.current_device()) if rank == 0 else None
    if clocks:
        clocks.start()
    outs, ms = timed(step_device, args.steps)
    if clocks:
        clk = clocks.stop()
    torch.cuda.synchronize()
    if dist is not None:
        dist.barrier()
    total_ms = sum(ms)
    results = [o[0] for o in outs]
    launches = sum(o[1] for o in outs)
    iters = statistics.mean(r.iters for r in results)
    solve_s = statistics.mean(r.solve_seconds for r in results)
    ok = all(r.status == rhpdhg.STATUS_OPTIMAL for r in results)
    # e2e through host buffers
    e2e_outs, e2e_ms = timed(step_host, max(2, min(args.steps, 3)))
    # the other precision on the same workload (reported beside the headline), timed as the
    # same create + solve + poll + free step
    other = 1 - args.precision
    oparams = dict(params, precision=other)

    def step_other():
        so = rhpdhg.Solver(dev, device=True, stream=sh, **oparams)
        so.solve(1)
        r = so.poll(x=xo, y=yo, out_memory=rhpdhg.MEM_DEVICE)
        so.close()
        return r

    step_other()
    o_outs, o_ms = timed(step_other, 3)
    ro = o_outs[-1]
    # rate probes for the roofline denominators that MEASURED_PEAKS.json does not hold: the read
    # bandwidth of a 64 MiB buffer held in L2, and the FP64 FMA rate
    rc1, l2_gbs = rhpdhg.rhpdhg_probe_l2_read_bandwidth(64 << 20, sh)
    rc2, fp64_tflops = rhpdhg.rhpdhg_probe_fp64_fma_rate(sh)
    if rc1 != rhpdhg.OK or rc2 != rhpdhg.OK:
        raise RuntimeError("rate probe failed: " + rhpdhg.rhpdhg_last_error(None))
    read_gbs = {f"{b >> 20} MiB": rhpdhg.rhpdhg_probe_l2_read_bandwidth(b, sh)[1]
                for b in (16 << 20, 64 << 20, 1 << 30)}
    # kernel timing (CUDA events around each launch of the two iteration kernels), for the
    # headline precision and the other one
    def profiled(prm):
        s = rhpdhg.Solver(dev, device=True, stream=sh, profile=1, **prm)
        s.solve(1)
        r = s.poll(x=xo, y=yo, out_memory=rhpdhg.MEM_DEVICE)
        k = s.kernel_times()
        s.close()
        return r, k

    rp, kt = profiled(params)
    _, kt_other = profiled(oparams)
    total_ms, e2e_total = replica_max(dist, [total_ms, sum(e2e_ms)], "cuda")
    if rank != 0:
        return 0
    ms_step = total_ms / args.steps
    value = replica_throughput(world, args.steps, total_ms)
    e2e_value = replica_throughput(world, len(e2e_ms), e2e_total)
    peak, peak_kind = load_peaks()
    # dominant kernel by total time
    if kt["ms_col"] >= kt["ms_row"]:
        dom, dom_ms, dom_bytes = "column kernel (K^T y~ + primal step)", kt["ms_col"], kt["bytes_col"]
    else:
        dom, dom_ms, dom_bytes = "row kernel (K x~ + dual step)", kt["ms_row"], kt["bytes_row"]
    achieved = dom_bytes / (dom_ms / 1000.0) / 1e9
    # FP64 path: algorithmic FP64 flops per launch (one FMA per nonzero, the fused elementwise
    # work per row and per column) against the probed FP64 FMA rate
    kt64 = kt if args.precision == 0 else kt_other
    fl_row, fl_col = fp64_flops(lp)
    fp64_row = fl_row / (kt64["ms_row"] / 1000.0) / 1e12
    fp64_col = fl_col / (kt64["ms_col"] / 1000.0) / 1e12
    o_ms_step = statistics.mean(o_ms)
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_step,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
        "dtype": "f64" if args.precision == 0 else "f32+f64",
        "data": "synthetic",
        "config": {"workload": WORKLOAD, "tol": args.tol, "algorithm": args.algorithm,
                   "precision": "fp64" if args.precision == 0 else "fp32 iterates, fp64 restarts",
                   "parallelism": f"replicas x{world}",
                   "l2": "256 MB buffer written before every timed step (L2 flush)"},
        "time_to_tol_s": ms_step / 1000.0, "solve_only_s": solve_s, "iters": iters,
        "iters_per_s": iters / solve_s, "all_optimal": ok,
        "rel_kkt": max(results[-1].rel_p, results[-1].rel_d, results[-1].rel_gap),
        "other_precision": {"precision": "fp64" if other == 0 else "fp32 iterates, fp64 restarts",
                            "status": ro.status_name, "iters": ro.iters,
                            "value": 1000.0 / o_ms_step, "ms_per_step": o_ms_step,
                            "solve_s": ro.solve_seconds,
                            "iters_per_s": ro.iters / ro.solve_seconds,
                            "ms_per_launch_row": kt_other["ms_row"],
                            "ms_per_launch_col": kt_other["ms_col"]},
        "fp64_roofline": {"bound": "fp64 alu", "unit": "TFLOP/s",
                          "peak": fp64_tflops, "peak_kind": "probed FP64 FMA rate (this run)",
                          "flops_per_launch_row": fl_row, "flops_per_launch_col": fl_col,
                          "row_kernel": {"achieved": fp64_row, "frac": fp64_row / fp64_tflops},
                          "column_kernel": {"achieved": fp64_col,
                                            "frac": fp64_col / fp64_tflops}},
        "gpu_launches": int(launches),
        "autotune": {"first_create": {k: layouts[0][k] for k in TUNE_KEYS},
                     "timed_steps": {k: layouts[-1][k] for k in TUNE_KEYS},
                     "note": "the first warm-up create times the candidate geometries; later "
                             "creates of the same LP structure take the cached choice"},
        "e2e": {"value": e2e_value, "unit": UNIT,
                "h2d_bytes_per_step": problem_bytes(lp),
                "d2h_bytes_per_step": 8 * (lp.n + lp.m)},
        "roofline": {"bound": "hbm", "kernel": dom, "achieved": achieved, "peak": peak,
                     "peak_kind": f"{peak_kind} hbm_gbs", "unit": "GB/s",
                     "frac": achieved / peak,
                     "l2_peak": l2_gbs, "l2_peak_kind": "probed read bandwidth of a 64 MiB "
                                                       "L2-resident buffer (this run)",
                     "l2_frac": achieved / l2_gbs,
                     "read_bandwidth_by_buffer_size_gbs": read_gbs,
                     "traffic": (PROFILED_TRAFFIC.get(dom) if args.precision == 1 and
                                 kernel_digest() == PROFILED_TRAFFIC["digest"] else None),
                     "ms_per_launch_row": kt["ms_row"], "ms_per_launch_col": kt["ms_col"],
                     "bytes_per_launch_row": kt["bytes_row"],
                     "bytes_per_launch_col": kt["bytes_col"],
                     "profiled_iters": rp.iters},
        "clocks": clk,
    }
    if world == 1 and args.serve_requests > 0:
        line["serving"] = run_serving(args, rhpdhg, lpgen)
    if world == 1 and not args.no_large:
        line["large_lp"] = run_large(args, rhpdhg, lpgen, peak, f"{peak_kind} hbm_gbs")
    if world == 1 and not args.no_cpu_baseline:
        cb = cpu_oracle_sample(lp, args.algorithm, args.tol, iters)
        line["cpu_baseline"] = {
            "value": cb["value"], "unit": UNIT, "cores": 1, "kind": "oracle",
            "sample": f"oracle set-up ({cb['setup_s']:.1f} s) + 100 iterations "
                      f"({cb['s_per_iter'] * 1e3:.1f} ms each) on this LP; time-to-tol "
                      f"extrapolated to the {iters:.0f} iterations both paths take "
                      f"(FP64 iterate parity)"}
    print(json.dumps(line), flush=True)
    if dist is not None:
        dist.destroy_process_group()
    return 0


def main():
    args = parse()
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
