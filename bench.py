#!/usr/bin/env python
"""Benchmark of the motif-search hot path on one or more GB300s.

One step = momenti_hash_all + momenti_topk on one synthetic series of the
float32 plain-method workload: D=8, n=100,000, w=300, d=3, k=10,
delta=0.05, 8 GB memory limit, paper defaults K=8, L=200, r automatic
(random walk + 3 sinusoids + N(0, 0.1) noise, five motifs planted in 3
dims each).  The series is resident in HBM when a timed step starts; the
L2 is flushed (a 512 MB write) before every timed step, outside the timed
interval.  Each rank of a multi-GPU run searches its own series (weak
scaling, no collective on the data path).

value  = subsequence hashes (windows x dims x repetitions) pushed through
         the whole step per second, summed over ranks;
e2e    = the same through host buffers (pinned series copied in, motifs
         copied out, both inside the timed interval);
roofline: the dominant kernel timed live with CUDA events on its stream;
cpu_baseline: the CPU oracle (oracle/) on a bounded sample.

--impl reference times the CPU oracle (the reference arm of this build).
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

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

# DRAM bytes per launch (dram__bytes_read.sum + dram__bytes_write.sum) that
# ncu measured for a kernel on this workload at full size, with the SHA-256
# of the source file that kernel was built from: reported only while that
# file is unchanged (the capture and its command are summarised in profiles/)
NCU_TRAFFIC = {}


def measured_traffic(kernel):
    import hashlib
    if kernel not in NCU_TRAFFIC:
        return None
    path, sha, nbytes = NCU_TRAFFIC[kernel]
    try:
        with open(os.path.join(ROOT, path), "rb") as fh:
            if hashlib.sha256(fh.read()).hexdigest() != sha:
                return None
    except OSError:
        return None
    return nbytes


# dominant kernels and their algorithmic work per launch
DOMINANT = ("proj_hash_tc", "collide", "subbucket", "sort_*", "allpairs", "proj_hash_fp32",
            "verify_events")
# kernels whose roofline is reported beside the dominant one
SECONDARY = ("sort_*", "proj_hash_tc", "allpairs")
# the kernels of collision counting (step a7), reported together as "collision"
COLLISION = ("collide", "bucket_jobs", "subbucket", "subwarp")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="momenti", choices=["momenti", "reference"])
    ap.add_argument("--precision", default="f16x2", choices=["f16x2", "fp32"])
    ap.add_argument("--kernel", default="auto", help="kernel for the roofline object")
    ap.add_argument("--no-baseline", action="store_true", help="skip the CPU oracle leg")
    ap.add_argument("--no-fp32", action="store_true", help="skip the plain FP32 comparison")
    ap.add_argument("--batch-series", type=int, default=64,
                    help="series of the batching form timed beside the step (0: skip)")
    ap.add_argument("--n", type=int, default=0,
                    help="series length (0: the workload's; smaller only for profiler captures)")
    ap.add_argument("--workload", default="plain_fp32", choices=["plain_fp32", "precision_form"],
                    help="plain_fp32: D=8 n=1e5 w=300 (the default line); precision_form: "
                         "D=32 n=1e6 w=500 d=8 (minutes per step)")
    ap.add_argument("--r", type=float, default=0.0, help="quantisation width (0: Section 6.1 heuristic)")
    ap.add_argument("--large-form", type=float, default=0.0, metavar="SECONDS",
                    help="also run the large memory-bounded form at full size (D=64, n=1e7, "
                         "64 GB limit): hashing, then the anytime search for this many seconds")
    ap.add_argument("--no-rsweep", action="store_true",
                    help="skip the parameter legs (r, K, L, delta sweeps, tensoring, scalability)")
    return ap.parse_args()


def workload(rank: int, n: int = 0, name: str = "plain_fp32"):
    from paper_2502_14446_gb300 import synth
    if name == "precision_form":
        return synth.precision_form(seed=rank, n=n or 1_000_000)
    return synth.plain_fp32(seed=rank, n=n or 100_000)


def describe(wl) -> str:
    """The workload line of config: what it is, with its sizes."""
    mem = f", {wl.mem_limit >> 30} GB limit" if wl.mem_limit else ""
    prec = " (FP64 stats and re-verification)" if wl.name == "precision_form" else ""
    return (f"{wl.name}: D={wl.D} n={wl.n} w={wl.w} d={wl.d} k={wl.k} delta={wl.delta} "
            f"float32{mem}{prec}, K=8 L=200")


def combine(local_ms: float, units_per_step: int, steps: int, world: int, device=None) -> tuple:
    """Whole-job value over ranks: every rank pushes units_per_step through
    each of its steps; the job time is the slowest rank's.  Returns
    (value in units/s, max milliseconds)."""
    import torch
    import torch.distributed as dist
    total_ms = float(local_ms)
    if world > 1:
        t = torch.tensor([total_ms], dtype=torch.float64, device=device)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        total_ms = float(t.item())
    return world * units_per_step * steps / (total_ms / 1e3), total_ms


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        d = json.load(open(path))
        return {"hbm_gbs": d["hbm_gbs"], "tflops": d["bf16_tflops"],
                "tflops_sustained": d.get("bf16_tflops_sustained", d["bf16_tflops"]),
                "sm_max_mhz": d.get("sm_max_mhz", 2070.0), "src": "measured"}
    return {"hbm_gbs": 6800.0, "tflops": 1900.0, "tflops_sustained": 1700.0,
            "sm_max_mhz": 2070.0, "src": "fallback"}


class Clocks:
    """nvidia-smi sampling during the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, dev: int):
        self.dev = dev
        self.f = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        self.p = None

    def start(self):
        try:
            self.p = subprocess.Popen(["nvidia-smi", f"--id={self.dev}", f"--query-gpu={self.Q}",
                                       "--format=csv,noheader,nounits", "-lms", "200"],
                                      stdout=self.f, stderr=subprocess.DEVNULL)
        except (OSError, ValueError):
            self.p = None

    def stop(self):
        if self.p is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.p.terminate()
        try:
            self.p.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.p.kill()
        self.f.flush()
        text = open(self.f.name).read()
        os.unlink(self.f.name)
        return self.parse(text)

    @staticmethod
    def parse(text: str) -> dict:
        """Median SM clock, the maximum clock and the throttle reasons seen
        in nvidia-smi rows of the query Q (csv, no header, no units);
        malformed rows are skipped."""
        rows = [r.split(",") for r in text.strip().splitlines() if r.strip()]
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            try:
                clk, top = float(r[1]), float(r[2])
                flags = [v.strip() for v in r[5:9]]
            except (ValueError, IndexError):
                continue
            sm.append(clk)
            mx = top
            for nm, v in zip(names, flags):
                if v == "Active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx,
                "reasons": sorted(reasons), "samples": len(sm)}


def params_for(mom, wl, precision, r=0.0):
    return mom.default_params(w=wl.w, d=wl.d, k=wl.k, delta=wl.delta, mem_limit=wl.mem_limit,
                              K=8, L=200, precision=precision, r=r)


def sm_count(device=None) -> int:
    """Streaming multiprocessors of the GPU (152 on a GB300)."""
    import torch
    return torch.cuda.get_device_properties(device if device is not None else 0).multi_processor_count


def reps_processed(st, K, L):
    """(level, repetition) cells the traversal processed in one search:
    levels K down to the stopping level, where STOP held at (i, j) or the
    cost switch ended the search after its one-repetition probe."""
    if st["stop_i"] > 0:
        return (K - st["stop_i"]) * L + st["stop_j"]
    if st["switch_level"] > 0:
        return (K - st["switch_level"]) * L + 1
    return K * L


def roofline(kernel, k_ms, k_n, info, st, wl, steps, pk, sms=152):
    """Roofline object of one kernel from its live CUDA-event time over the
    timed steps: achieved = algorithmic work of the timed launches / their
    device time.  Algorithmic work per unit (per step, from the step's own
    counters):
      proj_hash_tc    2 w flop per useful projection (M D L K of them)
      proj_hash_fp32  the same, on FP32 CUDA cores
      verify_events   8 D w bytes per verified pair (both windows, all dims)
      allpairs        8 flop per pair and dim, the method's minimal count:
                      the sliding cross product of the diagonal recurrence
                      (two FMA, 4 flop) and the Pearson threshold test on
                      per-window factors (one FMA, one multiply, one
                      compare: 4); the kernel tests with one FMA (3 in
                      all), and runs groups with a passing dimension twice
      sort_*          20 bytes per index entry (window, dim, repetition):
                      its 8-byte key read, the sorted 12-byte (key, window)
                      written; every kernel of the index sort together
      collision       12 bytes per index entry per (level, repetition)
                      processed (8-byte key, 4-byte window of the sorted
                      order) and 16 D bytes per compared bucket pair (the
                      keys of both windows in every dim); the kernels of
                      COLLISION together
    """
    if not k_n or k_ms <= 0:
        return None
    M, D, L, K, w = info["M"], info["D"], info["L"], info["K"], wl.w
    secs = k_ms / 1e3
    sm_peak = sms * 128 * 2 * pk["sm_max_mhz"] * 1e6 / 1e12
    sm_src = f"{sms} SMs x 128 FP32 lanes x 2 flop x max SM clock"
    if kernel in ("proj_hash_tc", "proj_hash_fp32"):
        work = 2.0 * M * D * L * K * w * steps
        bound, unit = ("tensor", "TFLOP/s") if kernel == "proj_hash_tc" else ("alu", "TFLOP/s")
        achieved = work / secs / 1e12
        peak = pk["tflops_sustained"] if bound == "tensor" else sm_peak
        src = (pk["src"] + " sustained bf16 (fp16 same rate)") if bound == "tensor" else sm_src
    elif kernel == "verify_events":
        work = 8.0 * D * w * st["n_candidates"] * steps
        bound, unit = "hbm", "GB/s"
        achieved = work / secs / 1e9
        peak, src = pk["hbm_gbs"], pk["src"] + " copy bandwidth"
    elif kernel == "allpairs":
        excl = w // 2
        pairs = max(0, M - excl - 1) * max(0, M - excl) / 2.0
        work = 8.0 * D * pairs * steps
        bound, unit = "alu", "TFLOP/s"
        achieved = work / secs / 1e12
        peak, src = sm_peak, sm_src
    elif kernel == "collision":
        work = (12.0 * M * D * reps_processed(st, K, L) + 16.0 * D * st["n_pair_checks"]) * steps
        bound, unit = "hbm", "GB/s"
        achieved = work / secs / 1e9
        peak, src = pk["hbm_gbs"], pk["src"] + " copy bandwidth"
    elif kernel == "sort_*":
        work = 20.0 * M * D * L * steps
        bound, unit = "hbm", "GB/s"
        achieved = work / secs / 1e9
        peak, src = pk["hbm_gbs"], pk["src"] + " copy bandwidth"
    else:
        return {"kernel": kernel, "bound": None, "achieved": None, "peak": None, "unit": None,
                "frac": None, "traffic": None, "launches": k_n, "ms_per_launch": k_ms / k_n}
    return {"kernel": kernel, "bound": bound, "achieved": achieved, "peak": peak, "unit": unit,
            "frac": achieved / peak, "traffic": measured_traffic(kernel), "peak_src": src, "launches": k_n,
            "ms_per_launch": k_ms / k_n, "work_per_step": work / steps}


def run_momenti(args):
    import numpy as np
    import torch
    import torch.distributed as dist

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)

    from paper_2502_14446_gb300 import build_ext
    if rank == 0:
        build_ext.build()
    if world > 1:
        dist.barrier()
    from paper_2502_14446_gb300 import momenti as mom

    wl = workload(rank, args.n, args.workload)
    prec = mom.PREC_F16X2 if args.precision == "f16x2" else mom.PREC_FP32
    series = torch.from_numpy(wl.series).to(dev)
    flush = torch.empty(512 << 20, dtype=torch.uint8, device=dev)
    stream = torch.cuda.current_stream(dev)
    h = mom.Momenti(params_for(mom, wl, prec, args.r))
    sms = sm_count(dev)

    def step():
        h.hash_all(series, stream=stream.cuda_stream)
        return h.topk()

    for _ in range(args.warmup):
        motifs, st = step()
    torch.cuda.synchronize()
    info = h.info()

    # device time of each candidate kernel over one step: the dominant one is
    # timed live in the timed steps; the others' rooflines come from this step
    per_kernel = {}
    candidates = (DOMINANT + SECONDARY + COLLISION if args.kernel == "auto"
                  else SECONDARY + (args.kernel,))
    for kname in dict.fromkeys(candidates):
        mom.time_kernel(kname)
        _, st_k = step()
        ms, n = mom.kernel_time()
        per_kernel[kname] = (ms, n, st_k)
    mom.time_kernel(None)
    kernel = args.kernel
    if kernel == "auto":
        kernel = max(DOMINANT, key=lambda k: per_kernel[k][0])
    mom.time_kernel(kernel)

    clocks = Clocks(local)
    if world > 1:
        dist.barrier()
    torch.cuda.synchronize()
    launches0 = mom.launch_count()
    clocks.start()
    times = []
    for _ in range(args.steps):
        flush.fill_(1)
        ev0 = torch.cuda.Event(enable_timing=True)
        ev1 = torch.cuda.Event(enable_timing=True)
        ev0.record(stream)
        motifs, st = step()
        ev1.record(stream)
        ev1.synchronize()
        times.append(ev0.elapsed_time(ev1))
    torch.cuda.synchronize()
    clk = clocks.stop()
    launches = mom.launch_count() - launches0
    k_ms, k_n = mom.kernel_time()
    mom.time_kernel(None)
    units_step = info["M"] * info["D"] * info["L"]
    value, total_ms = combine(sum(times), units_step, args.steps, world, dev)
    if world > 1:
        dist.barrier()

    # ---- end to end through host buffers ----
    pinned = torch.from_numpy(wl.series).pin_memory().numpy()
    e2e_times = []
    for q in range(max(2, args.steps)):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        h.hash_all(pinned)
        m2, _ = h.topk()
        torch.cuda.synchronize()
        if q >= 1:
            e2e_times.append(time.perf_counter() - t0)
    e2e_s = statistics.mean(e2e_times)
    h_bytes = wl.series.nbytes
    d_bytes = wl.k * 48

    out = None
    if rank == 0:
        pk = peaks()
        roof = roofline(kernel, k_ms, k_n, info, st, wl, args.steps, pk, sms)
        others = {}
        for kname in SECONDARY:
            if kname == kernel:
                continue
            ms, n, st_k = per_kernel[kname]
            r2 = roofline(kname, ms, n, info, st_k, wl, 1, pk, sms)
            if r2 is not None:
                r2["timed"] = "one untimed step before the timed region"
                others[kname] = r2
        if all(k in per_kernel for k in COLLISION):
            ms = sum(per_kernel[k][0] for k in COLLISION)
            n = sum(per_kernel[k][1] for k in COLLISION)
            r2 = roofline("collision", ms, n, info, per_kernel["collide"][2], wl, 1, pk, sms)
            if r2 is not None:
                r2["timed"] = "one untimed step per kernel before the timed region"
                r2["kernels"] = list(COLLISION)
                r2["note"] = ("the unit counts a 16 D-byte key gather per compared bucket pair; "
                              "the kernels load each window's keys once per 32-window tile or "
                              "warp and compare them in registers, so achieved can exceed the "
                              "copy bandwidth")
                others["collision"] = r2
        plain = None
        if not args.no_fp32 and prec != mom.PREC_FP32:
            h32 = mom.Momenti(params_for(mom, wl, mom.PREC_FP32, args.r))
            h32.hash_all(series, stream=stream.cuda_stream)
            h32.topk()
            ts = []
            for _ in range(2):
                flush.fill_(1)
                e0 = torch.cuda.Event(enable_timing=True)
                e1 = torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                h32.hash_all(series, stream=stream.cuda_stream)
                _, st32 = h32.topk()
                e1.record(stream)
                e1.synchronize()
                ts.append(e0.elapsed_time(e1))
            plain = {"ms_per_step": statistics.mean(ts),
                     "value": units_step / (statistics.mean(ts) / 1e3),
                     "t_hash_ms": st32["t_hash_ms"]}
            h32.close()
        rsweep = tens = sweeps = scal = None
        if wl.name == "plain_fp32" and not args.no_rsweep:
            rsweep = r_sweep_leg(mom, wl, series, stream, flush, prec)
            tens = tensoring_leg(mom, wl, series, stream, flush, prec)
            sweeps = param_sweep_leg(mom, wl, series, stream, flush, prec)
            scal = scalability_leg(mom, dev, stream, flush, prec)
        batch = batch_leg(mom, args.batch_series, dev) if args.batch_series > 0 else None
        large = large_form_leg(mom, dev, stream, prec, args.large_form) if args.large_form > 0 else None
        base = None if args.no_baseline else cpu_baseline(wl)
        # float64 error of each result: the float32 traversal distance
        # against the float64 re-verification (stats), and the float64
        # distances returned
        out = {
            "metric": "time-to-top-k motifs (s) and subsequences hashed/s, BF16/batched vs plain FP32",
            "value": value, "unit": "subsequences/s", "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": total_ms / args.steps,
            "time_to_topk_s": total_ms / args.steps / 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f16x2+f32" if prec == mom.PREC_F16X2 else "f32",
            "data": "synthetic",
            "config": {"workload": describe(wl) + (f", r={args.r}" if args.r > 0 else ", r auto"),
                       "precision": args.precision, "L_used": info["L"], "K": info["K"],
                       "r": info["r"], "windows": info["M"], "l2": "flushed (512 MB write) before each step",
                       "parallelism": f"replicas x{world}"},
            "step": {"t_hash_ms": st["t_hash_ms"], "t_sort_ms": st["t_sort_ms"],
                     "t_traverse_ms": st["t_traverse_ms"], "t_fallback_ms": st["t_fallback_ms"],
                     "stop": [st["stop_i"], st["stop_j"]], "fallback": st["fallback"],
                     "switch_level": st["switch_level"],
                     "n_candidates": st["n_candidates"], "n_verified": st["n_verified"],
                     "n_rehashed": st["n_rehashed"], "precision_used": st["precision_used"],
                     "max_rel_err_fp32": st["max_rel_err_fp32"],
                     "hashed_per_s_hash_all": units_step / (st["t_hash_ms"] / 1e3),
                     "kernel_ms": {k: round(v[0], 3) for k, v in per_kernel.items()}},
            "motifs": [[m["a"], m["b"], round(m["dist_d"], 6), list(m["dims"])] for m in motifs],
            "plain_fp32": plain,
            "r_sweep": rsweep,
            "param_sweeps": sweeps,
            "scalability": scal,
            "tensoring": tens,
            "batch_form": batch,
            "large_form": large,
            "e2e": {"value": world * units_step / e2e_s, "unit": "subsequences/s",
                    "time_to_topk_s": e2e_s, "h2d_bytes_per_step": h_bytes,
                    "d2h_bytes_per_step": d_bytes},
            "roofline": roof,
            "rooflines_other": others,
            "cpu_baseline": base,
            "gpu_launches": int(launches),
            "clocks": clk,
        }
        print(json.dumps(out), flush=True)
    h.close()
    if world > 1:
        dist.barrier()
        dist.destroy_process_group()
    return out


def tensoring_leg(mom, wl, series, stream, flush, prec, m=14):
    """Tensoring (Section 6.1) against plain repetitions on this workload at
    the same L = m^2 (K = 8, r by the heuristic, library defaults
    otherwise): hash_all time (projections of K m instead of K L values per
    window and dim, then the key interleave), device memory held by the
    handle, time to top-k (mean of two steps after one warm-up, L2 flushed
    before each) and the motifs found."""
    import torch
    out = {"L": m * m}
    motifs = {}
    for name, flags in (("plain", 0), ("tensored", mom.FLAG_TENSORING)):
        p = params_for(mom, wl, prec)
        p.L = m * m
        p.flags = flags
        hh = mom.Momenti(p)
        hh.hash_all(series, stream=stream.cuda_stream)
        hh.topk()
        ts, th = [], []
        for _ in range(2):
            flush.fill_(1)
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            hh.hash_all(series, stream=stream.cuda_stream)
            mm, st = hh.topk()
            e1.record(stream)
            e1.synchronize()
            ts.append(e0.elapsed_time(e1))
            th.append(st["t_hash_ms"])
        hh.close()
        motifs[name] = [(x["a"], x["b"]) for x in mm]
        out[name] = {"t_hash_ms": statistics.mean(th), "t_sort_ms": st["t_sort_ms"],
                     "time_to_topk_ms": statistics.mean(ts), "device_bytes": st["device_bytes"],
                     "stop": [st["stop_i"], st["stop_j"]], "fallback": st["fallback"],
                     "n_verified": st["n_verified"], "r": st["r"]}
    out["same_motifs"] = motifs["plain"] == motifs["tensored"]
    return out


def timed_search(mom, params, series, stream, flush, reps=2):
    """hash_all + topk with ``params`` on a device series: one warm-up, then
    the mean of ``reps`` steps (L2 flushed before each, CUDA events on the
    stream); returns (ms, motifs, stats)."""
    import torch
    hh = mom.Momenti(params)
    hh.hash_all(series, stream=stream.cuda_stream)
    hh.topk()
    ts = []
    for _ in range(reps):
        flush.fill_(1)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        hh.hash_all(series, stream=stream.cuda_stream)
        m, st = hh.topk()
        e1.record(stream)
        e1.synchronize()
        ts.append(e0.elapsed_time(e1))
    hh.close()
    return statistics.mean(ts), m, st


def param_sweep_leg(mom, wl, series, stream, flush, prec):
    """The paper's parameter experiments (Section 7: impact of K, L and
    delta) on this workload, the other parameters at their defaults (K=8,
    L=200, the r heuristic, cost switch on).  K stops at 8: a composite key
    holds at most 8 hash values here.  Per setting: time to top-k, the
    stopping (i, j) or the exact path, distance computations, device memory
    and whether the motifs equal the stored exact top-k."""
    gold = None
    path = os.path.join(ROOT, "tests", "golden", "exact_plain_fp32_seed0.json")
    if wl.n == 100_000 and wl.seed == 0 and os.path.exists(path):
        gold = [(m[1], m[2]) for m in json.load(open(path))["motifs"]]
    out = {}
    for name, values in (("K", (2, 4, 6, 8)), ("L", (10, 50, 100, 200, 400)),
                         ("delta", (0.05, 0.1, 0.2, 0.4))):
        rows = []
        for v in values:
            p = params_for(mom, wl, prec)
            setattr(p, name, v)
            ms, m, st = timed_search(mom, p, series, stream, flush)
            rows.append({name: v, "time_to_topk_ms": ms, "stop": [st["stop_i"], st["stop_j"]],
                         "fallback": st["fallback"], "switch_level": st["switch_level"],
                         "n_verified": st["n_verified"], "device_bytes": st["device_bytes"],
                         "L_used": st["L"],
                         "matches_exact": None if gold is None else [(x["a"], x["b"]) for x in m] == gold})
        out[name] = rows
    return out


def large_form_leg(mom, dev, stream, prec, budget_s: float):
    """The large memory-bounded form at full size (synth.large_form: D=64,
    n=1e7, w=1000, d=16, k=10, delta=0.01, float32, 64 GB device-memory
    limit).  The memory planner picks L; hash_all is timed with CUDA events
    (second of two builds, series resident in HBM); then the anytime search
    (Section 4) advances one repetition at a time for budget_s seconds and
    reports where it stands: the cursor (i, j), how many candidates it
    holds and the smallest miss bound among them.  The exact fallback of
    this form (about 3e15 pair-dimension evaluations) is not run."""
    import torch
    from paper_2502_14446_gb300 import synth
    wl = synth.large_form(0)
    x = torch.from_numpy(wl.series).to(dev)
    desc = (f"large_form: D={wl.D} n={wl.n} w={wl.w} d={wl.d} k={wl.k} delta={wl.delta} float32, "
            f"{wl.mem_limit >> 30} GB limit, K=8, L planned")
    p = mom.default_params(w=wl.w, d=wl.d, k=wl.k, delta=wl.delta, precision=prec,
                           mem_limit=wl.mem_limit)
    h = mom.Momenti(p)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    for _ in range(2):
        torch.cuda.synchronize()
        e0.record(stream)
        h.hash_all(x, stream=stream.cuda_stream)
        e1.record(stream)
        e1.synchronize()
    hash_ms = e0.elapsed_time(e1)
    info = h.info()
    h.search_begin()
    t0 = time.perf_counter()
    steps, ended = 0, False
    while not ended and time.perf_counter() - t0 < budget_s:
        ended = h.search_step(1)
        steps += 1
    cur, (i, j, ended) = h.search_current()
    top = cur[wl.d]
    planted = {(a, b) for a, b, _ in wl.planted}
    out = {"workload": desc, "L_planned": info["L"], "K": info["K"], "r": info["r"],
           "windows": info["M"], "hash_all_ms": hash_ms,
           "hashed_per_s": info["M"] * 64 * info["L"] / (hash_ms / 1e3),
           "search_s": time.perf_counter() - t0, "repetitions_processed": steps,
           "cursor": [i, j, bool(ended)], "candidates": len(top),
           "planted_among_candidates": sum((m["a"], m["b"]) in planted for m in top),
           "smallest_miss_bound": min((m["fail_bound"] for m in top), default=None)}
    h.close()
    del x
    return out


def scalability_leg(mom, dev, stream, flush, prec, ns=(10_000, 30_000, 100_000, 300_000, 1_000_000)):
    """The synthetic scalability workload of Section 7 (synth.scalability:
    D=5 random walks, one sinusoidal motif of w=300 in 2 dims, d=2, k=1)
    at growing n: time to top-k, hashing time, how the search ended, and
    whether the planted pair is the returned motif."""
    import torch
    from paper_2502_14446_gb300 import synth
    rows = []
    for n in ns:
        wl = synth.scalability(0, n=n)
        x = torch.from_numpy(wl.series).to(dev)
        p = mom.default_params(w=wl.w, d=wl.d, k=wl.k, delta=wl.delta, precision=prec)
        ms, m, st = timed_search(mom, p, x, stream, flush, reps=1)
        a, b, _ = wl.planted[0]
        rows.append({"n": n, "time_to_topk_ms": ms, "t_hash_ms": st["t_hash_ms"],
                     "stop": [st["stop_i"], st["stop_j"]], "fallback": st["fallback"],
                     "n_verified": st["n_verified"],
                     "planted_found": bool(m) and (m[0]["a"], m[0]["b"]) == (a, b)})
        del x
    return {"workload": "scalability: D=5 random walks, sinusoidal motif w=300 in 2 dims, "
                        "noise 0.1, d=2, k=1, delta=0.05, float32", "runs": rows}


def r_sweep_leg(mom, wl, series, stream, flush, prec, rs=(0.0, 4.0, 8.0, 12.0, 16.0)):
    """The paper's quantisation-width experiment (Section 7, impact of r) on
    this workload: the Section 6.1 heuristic (r = 0) against fixed r, with
    the library's default search (cost switch on).  Per r: the stopping
    (i, j) or the exact path, the level at which the cost switch chose it,
    distance computations, time to top-k (mean of two steps after one
    warm-up, L2 flushed before each) and whether the motifs equal the
    exact top-k the oracle wrote (tests/golden, this workload at seed 0)."""
    import torch
    gold = None
    path = os.path.join(ROOT, "tests", "golden", "exact_plain_fp32_seed0.json")
    if wl.n == 100_000 and wl.seed == 0 and os.path.exists(path):
        gold = [(m[1], m[2]) for m in json.load(open(path))["motifs"]]
    out = []
    for r in rs:
        hh = mom.Momenti(params_for(mom, wl, prec, r))
        hh.hash_all(series, stream=stream.cuda_stream)
        hh.topk()
        ts = []
        for _ in range(2):
            flush.fill_(1)
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            hh.hash_all(series, stream=stream.cuda_stream)
            m, st = hh.topk()
            e1.record(stream)
            e1.synchronize()
            ts.append(e0.elapsed_time(e1))
        hh.close()
        out.append({"r": st["r"], "r_auto": r == 0.0, "stop": [st["stop_i"], st["stop_j"]],
                    "fallback": st["fallback"], "switch_level": st["switch_level"],
                    "n_verified": st["n_verified"], "time_to_topk_ms": statistics.mean(ts),
                    "t_traverse_ms": st["t_traverse_ms"], "t_fallback_ms": st["t_fallback_ms"],
                    "matches_exact": None if gold is None else [(x["a"], x["b"]) for x in m] == gold})
    return out


def batch_leg(mom, count: int, dev, threads: int = 8):
    """The batching form on its first ``count`` series (lengths log-uniform in
    [2,000, 200,000], D in 3..16, w in {50, 100, 200}, d = ceil(D/3), k=5,
    delta=0.05, float32, series resident in HBM): momenti_topk_batch with
    ``threads`` workers, against the same searches one at a time through
    the same entry point (one worker).  Throughput in subsequence hashes
    (windows x dims x repetitions) per second, whole batch."""
    import torch
    from paper_2502_14446_gb300 import synth
    wls = synth.batch_form(0, count=count)
    series = [torch.from_numpy(wl.series).to(dev) for wl in wls]
    params = [dict(w=wl.w, d=wl.d, k=wl.k, delta=wl.delta) for wl in wls]
    torch.cuda.synchronize()
    mom.topk_batch(params[:4], series[:4], threads=threads)          # warm-up
    out = {"series": count, "threads": threads,
           "workload": "batching form: n log-uniform [2e3, 2e5], D 3..16, w {50,100,200}, "
                       "d=ceil(D/3), k=5, delta=0.05, float32, 2 planted motifs each"}
    for name, T in (("batched", threads), ("one_at_a_time", 1)):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        res = mom.topk_batch(params, series, threads=T)
        torch.cuda.synchronize()
        dt = time.perf_counter() - t0
        units = sum(st["n_windows"] * wl.D * st["L"] for (m, st), wl in zip(res, wls))
        out[name] = {"seconds": dt, "value": units / dt, "unit": "subsequences/s",
                     "fallbacks": sum(st["fallback"] for m, st in res)}
    return out


def cpu_baseline(wl, budget_s: float = 20.0):
    """The CPU oracle (Algorithm 1 rendering, float64 numpy) on a bounded
    prefix of the same workload: the first 2,000 points of the series
    (1,200 for the 32-dimension precision form), all D dims, w, d, k, delta
    as the workload, K=8, L=200 hash functions drawn by the same
    generator."""
    from oracle import momenti_oracle as O
    from paper_2502_14446_gb300 import synth
    n = 1200 if wl.D > 16 else 2000
    T = wl.series[:, :n].astype("float64")
    A, U = synth.hash_draws(wl.D, 200, 8, wl.w, 0)
    t0 = time.perf_counter()
    r = O.estimate_r(T, wl.w, A)
    res = O.momenti(T, wl.w, wl.d, wl.k, wl.delta, A, U, r)
    dt = time.perf_counter() - t0
    M = n - wl.w + 1
    units = M * wl.D * 200
    return {"value": units / dt, "unit": "subsequences/s", "cores": os.cpu_count(),
            "kind": "oracle", "seconds": dt,
            "sample": f"first {n} points of the series (M={M} windows), all {wl.D} dims, "
                      f"L=200, K=8: Algorithm 1 rendering in float64 numpy "
                      f"(stop={res['stop']})"}


def run_reference(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    wl = workload(0)
    times = []
    base = None
    for q in range(args.warmup + args.steps):
        b = cpu_baseline(wl)
        if q >= args.warmup:
            times.append(b["seconds"])
            base = b
    mean = statistics.mean(times)
    units = base["value"] * base["seconds"]       # subsequences of one step's sample
    value = units / mean
    out = {"metric": "time-to-top-k motifs (s) and subsequences hashed/s, BF16/batched vs plain FP32",
           "value": value, "unit": "subsequences/s", "n_gpus": world, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": mean * 1e3, "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
           "impl": "reference",
           "config": {"workload": describe(wl) + ", r auto",
                      "sample": "each step times the oracle on a bounded prefix (cpu_baseline.sample) "
                                "and reports its throughput there; the per-window cost of the "
                                "search grows with n, so this throughput is above what the "
                                "oracle reaches on the whole series",
                      "parallelism": f"replicas x{world}"},
           "cpu_baseline": {"value": value, "unit": "subsequences/s", "cores": os.cpu_count(),
                            "kind": "oracle", "sample": base["sample"]},
           "e2e": {"value": value, "unit": "subsequences/s", "h2d_bytes_per_step": 0,
                   "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_momenti(args)


if __name__ == "__main__":
    main()
