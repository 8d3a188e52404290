#!/usr/bin/env python
"""Benchmark of the exact Tukey depth hot path on GB300.

One step = one td_depth call over the whole batch of queries of the
workload: p = 4, n = 1000 data points round(40 N(0,1)) clipped to [-127,127],
64 query points (32 data rows, the lower coordinate-wise median, 31 uniform
points of the bounding box) -- C(1000, 2) = 499,500 subset sweeps per query
(Algorithm 1 with Algorithm 2 as the inner count, exact under ties).  Every
subset is decided by counts over all points: by the tables that the subsets of
a fan share, by a pass of its own over the points, or by the exact steps.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Prints one JSON line.  `value` is subset sweeps/s with the inputs resident in
device memory (CUDA events on the launch stream, L2 flushed between steps by
writing a 512 MB buffer outside the timed events); `e2e` is the same metric
through td_depth with host buffers (host<->device copies inside); the plain
exact one-query-per-launch form is timed beside it; `cpu_baseline` is the CPU
oracle on a bounded sample.  `--impl reference` times the CPU oracle alone.
"""
import argparse
import hashlib
import json
import math
import os
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

WORKLOAD = "p=4 n=1000 m=64, round(40*N(0,1)) clipped to [-127,127], int32; C(1000,2) subsets/query"
METRIC = "subset sweeps/sec"
UNIT = "sweeps/s"
L2_FLUSH_BYTES = 512 << 20


def _args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--scaling", choices=["strong", "weak"], default="strong",
                    help="with several ranks: strong (default) -- every rank sweeps its shard of the "
                         "same workload and an all-reduce MIN merges the depths inside each step; "
                         "weak -- every rank solves a batch of its own")
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--plain-queries", type=int, default=8)
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-extra", action="store_true",
                    help="leave out the batched (W3) and stream (W5) objects of the default line")
    ap.add_argument("--workload", choices=["W2", "W3", "W4", "W5", "W6", "W7"], default="W2",
                    help="W2 (default) is the benchmark line; W3 (256 datasets, one batched call), "
                         "W4 (p=5 with ties), W5 (request stream with Poisson arrivals), W6 (p=2) "
                         "and W7 (the Section 5.2 shapes, Algorithm 1 against Algorithm 3) print "
                         "their own lines")
    ap.add_argument("--stream-seconds", type=float, default=20.0)
    ap.add_argument("--profile-case", choices=["rcom", "adia", "critical"], default=None,
                    help="run the small fixed case that the ncu captures under profiles/ use "
                         "(two td_depth calls on --profile-queries queries of --workload) and exit")
    ap.add_argument("--profile-queries", type=int, default=4)
    return ap.parse_args()


def _dist():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def _workload(rank, strong):
    from paper_1409_3901_gb300 import workloads as W
    # strong scaling: every rank holds the benchmark workload and sweeps its
    # own shard of each query's subset loop; weak scaling: rank r solves its
    # own batch (seed 1 + r), rank 0 the benchmark workload itself
    return W.w2(seed=1 if strong else 1 + rank)


def _golden_w2():
    """The stored oracle counts of the benchmark workload, if present."""
    path = os.path.join(ROOT, "tests", "golden", "W2.json")
    try:
        with open(path) as f:
            g = json.load(f)
        return g["checksum"], np.array(g["T"], dtype=np.int64)
    except Exception:
        return None, None


def _ops_per_sweep(nnz, p):
    """Algorithmic work of one sweep: projection 2p, key ~6, comparison sort
    ceil(log2 n') compare-exchanges at ~2 ops, O(1) walk: n'(2p+6+2ceil(log2 n'))."""
    return nnz * (2 * p + 6 + 2 * math.ceil(math.log2(max(nnz, 2))))


def _fan_ops(nnz, p):
    """Lane operations of the strip bounds for one query of p >= 3, with the
    fewest strips (8; 16 at p = 3): per fan and point the projection onto the
    quotient by the tail (three functionals of p - 2 terms), two ratios (5) and
    per strip a key (6), its range (2) and two counts; per subset and strip a
    key, a range cut in two (4) and four look-ups summed and compared (9).  The
    passes over the points that a few percent of the subsets take, and the
    prefix sums of the tables, are left out."""
    strips = 16 if p == 3 else 8
    fans = 1 if p == 3 else math.comb(nnz - 1, p - 3)
    return fans * nnz * (3 * (p - 2) + 5 + 10 * strips) + math.comb(nnz, p - 2) * 19 * strips


def _algorithmic_ops(d, sweeps_per_call):
    """Sum over queries of the sweep kernel's algorithmic lane operations,
    scaled to the sweeps the library reports (dependent subsets are skipped;
    None: not scaled)."""
    tot_ops, tot_sw = 0.0, 0.0
    for z in d.Zq:
        nnz = int(d.n - np.all(d.X == z, axis=1).sum())
        sw = math.comb(nnz, d.p - 2)
        tot_ops += _fan_ops(nnz, d.p) if d.p >= 3 else sw * _ops_per_sweep(nnz, d.p)
        tot_sw += sw
    if sweeps_per_call is None or tot_sw == 0:
        return tot_ops
    return tot_ops * (sweeps_per_call / tot_sw)


class _Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during a region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.Q,
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.f, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.f.close()
        rows = []
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) >= 9:
                rows.append(parts)
        os.unlink(self.path)
        if not rows:
            return None
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in rows for k in range(4) if r[5 + k].lower().startswith("active")})
        return {"sm_mhz": float(np.median(sm)) if sm else None,
                "sm_max_mhz": max(mx) if mx else None, "reasons": reasons, "samples": len(rows)}


def _peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as f:
            return json.load(f), "measured"
    except Exception:
        return {"sm_max_mhz": 2070.0}, "fallback"


KERNEL_SOURCES = ("td_kernels.cu", "td_internal.h", "td_exact.cuh", "td_fan.cuh", "td_adia.cuh", "td_critical.cuh",
                  "td_wide.cuh")


def kernel_sources_sha():
    """sha256[:16] over the sweep kernel's translation unit: td_kernels.cu and
    the headers it includes, in that order."""
    h = hashlib.sha256()
    for f in KERNEL_SOURCES:
        with open(os.path.join(ROOT, "paper_1409_3901_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def _traffic_for_current_kernel():
    """DRAM bytes per launch of the sweep kernel from the committed ncu summary,
    valid only while the kernel's sources are unchanged since the capture."""
    path = os.path.join(ROOT, "profiles", "td_k_filtered_w2.json")
    try:
        h = kernel_sources_sha()
        rec = json.load(open(path))
        if rec.get("kernel_source_sha") == h:
            return rec.get("dram_bytes_per_launch_full")
    except Exception:
        pass
    return None


def _batched_w3(tukey, W, dev, stream, flush, peak_tops, steps=1):
    """The batched workload (256 datasets, p in {3,4,5}, 4096 queries) as one
    td_depth_batched call with device-resident inputs, timed like `value`
    (CUDA events on the launch stream, L2 flushed before the call)."""
    import torch
    sets = W.w3()
    ctx = tukey.Context(dev.index, device_pointers=True, stream=stream.cuda_stream)
    batch = [(torch.from_numpy(d.X).to(dev), torch.from_numpy(d.Zq).to(dev)) for d in sets]
    ctx.depth_batched(batch)                           # warm-up (also captures the graph)
    ms, ms_sweep, sw = 0.0, 0.0, 0
    for _ in range(steps):
        flush.fill_(1)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        ctx.depth_batched(batch)
        e1.record(stream)
        torch.cuda.synchronize(dev)
        ms += e0.elapsed_time(e1)
        ms_sweep += ctx.last_stats.ms_sweep
        sw += ctx.last_stats.sweeps
    ops = sum(_algorithmic_ops(d, None) for d in sets) * steps
    nq = sum(d.m for d in sets)
    achieved = ops / (ms_sweep / 1e3) / 1e12
    return {"workload": "W3: 256 datasets, p in {3,4,5}, n log-uniform in [100,2000] capped at "
                        "C(n,p-2)*n <= 4e9, 16 queries each; one td_depth_batched call",
            "datasets": len(sets), "queries": nq, "steps": steps,
            "sweeps_per_s": sw / (ms / 1e3), "queries_per_s": nq * steps / (ms / 1e3),
            "ms_per_call": ms / steps, "kernel_ms": ms_sweep / steps, "sweeps_per_call": sw // steps,
            "roofline": {"bound": "alu", "achieved": achieved, "peak": peak_tops, "unit": "Tops/s",
                         "frac": achieved / peak_tops, "kernel": "td_k_filtered<3..5>"},
            "timing": "CUDA events on the launch stream around the call; L2 flushed before it"}


def _exact_path(st):
    """The exact path's hit rate of one call: of the points projected in passes
    for one subset (the subsets that shared tables decide have none) those the
    FP32 filter could not certify (the subset's own points among them), and the
    sweeps whose bounds did not reach the running minimum, so that
    their points were projected again at the fine level and the uncertain
    ones placed with exact integer arithmetic."""
    pts = st.exact_points + st.filtered_points
    return {"uncertain_point_fraction": st.exact_points / max(pts, 1),
            "rescanned_sweep_fraction": st.rescanned_sweeps / max(st.sweeps, 1),
            "resolved_sweep_fraction": st.resolved_buckets / max(st.sweeps, 1),
            "tight_sweep_fraction": st.tight_exceptions / max(st.sweeps, 1)}


def _small_w1(tukey, W, dev, stream, flush, reps=20):
    """The small case W1 (p = 3, n = 300, 16 queries, 300 subsets each): both
    forms on device-resident inputs (CUDA events on the launch stream, L2
    flushed before each call), and the latency of a one-query call through
    the host API (td_depth on host buffers, copies included, wall clock)."""
    import torch
    d = W.w1()
    Xd = torch.from_numpy(d.X).to(dev)
    Zd = torch.from_numpy(d.Zq).to(dev)
    res = {}
    outs = {}
    for name, mode in (("filtered", tukey.TD_MODE_FILTERED), ("plain_exact", tukey.TD_MODE_PLAIN_EXACT)):
        ctx = tukey.Context(dev.index, mode=mode, device_pointers=True, stream=stream.cuda_stream)
        out = torch.empty(d.m, dtype=torch.int32, device=dev)
        ctx.depth(Xd, Zd, out)
        ms, sw = [], 0
        for _ in range(reps):
            flush.fill_(1)
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            ctx.depth(Xd, Zd, out)
            e1.record(stream)
            torch.cuda.synchronize(dev)
            ms.append(e0.elapsed_time(e1))
            sw += ctx.last_stats.sweeps
        outs[name] = out.clone()
        host = tukey.Context(dev.index, mode=mode)
        host.depth(d.X, d.Zq[:1])
        lat = []
        for r in range(reps):
            z = d.Zq[r % d.m: r % d.m + 1]
            t0 = time.perf_counter()
            host.depth(d.X, z)
            lat.append(1e3 * (time.perf_counter() - t0))
        lat.sort()
        med = sorted(ms)[len(ms) // 2]
        res[name] = {"ms_per_call": med, "queries_per_s": d.m / (med / 1e3),
                     "sweeps_per_s": sw / reps / (med / 1e3),
                     "one_query_call_ms_p50": lat[len(lat) // 2], "one_query_call_ms_max": lat[-1]}
    res["same_results"] = bool(torch.equal(outs["filtered"], outs["plain_exact"]))
    res["workload"] = "W1: p=3, n=300 uniform ints in [-127,127], 16 queries (8 data rows, 8 uniform)"
    res["timing"] = ("ms_per_call: median of %d calls with device-resident inputs (CUDA events); "
                     "one_query_call: td_depth from host buffers for one query, wall clock" % reps)
    return res


def _tuning(tukey, W, dev, stream, flush, w2_default_ms, w3_default_ms):
    """The autotuner on the two batched forms: a context tuned by td_autotune
    for every (dimension, octave of n) the workload holds, timed like the
    untuned line (CUDA events on the launch stream, L2 flushed first)."""
    import torch

    def timed(ctx, fn, steps):
        fn()
        ms = 0.0
        for _ in range(steps):
            flush.fill_(1)
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            fn()
            e1.record(stream)
            torch.cuda.synchronize(dev)
            ms += e0.elapsed_time(e1)
        return ms / steps

    out = {}
    d2 = W.w2()
    c2 = tukey.Context(dev.index, device_pointers=True, stream=stream.cuda_stream)
    t0 = time.perf_counter()
    r2 = c2.autotune(4, d2.n)
    tune_s = time.perf_counter() - t0
    X2, Z2 = torch.from_numpy(d2.X).to(dev), torch.from_numpy(d2.Zq).to(dev)
    o2 = torch.empty(d2.m, dtype=torch.int32, device=dev)
    out["W2"] = {"default_ms": w2_default_ms, "tuned_ms": timed(c2, lambda: c2.depth(X2, Z2, o2), 5),
                 "choice": {"p4_oct%d" % math.ceil(math.log2(d2.n)): r2["best_spw"]}, "tune_seconds": tune_s,
                 "candidates_ms": r2["candidates"], "size_rule_ms": r2["ms_default"]}
    sets = W.w3()
    c3 = tukey.Context(dev.index, device_pointers=True, stream=stream.cuda_stream)
    choice = {}
    t0 = time.perf_counter()
    for p in sorted({d.p for d in sets}):
        for oc in sorted({math.ceil(math.log2(d.n)) for d in sets if d.p == p}):
            n = max(p + 2, min(2048, int(0.75 * 2 ** oc)))
            choice["p%d_oct%d" % (p, oc)] = c3.autotune(p, n)["best_spw"]
    tune_s = time.perf_counter() - t0
    batch = [(torch.from_numpy(d.X).to(dev), torch.from_numpy(d.Zq).to(dev)) for d in sets]
    out["W3"] = {"default_ms": w3_default_ms, "tuned_ms": timed(c3, lambda: c3.depth_batched(batch), 1),
                 "choice": choice, "tune_seconds": tune_s}
    out["note"] = ("td_autotune per (dimension, octave of n) on seeded synthetic data; best_spw 0 = the "
                   "size rule; times of one call like value / batched")
    return out


def _stream_w5(tukey, W, dev, seconds, count=64):
    """The request stream: the first `count` requests of the W5 stream (no
    cost filter: p = 5 requests reach n = 1000, C(1000,3) subsets a query),
    cycled, arriving Poisson at 70% of the back-to-back rate measured on the
    same requests; latency from arrival to completion, split by p."""
    import random
    from math import comb
    reqs = W.w5(count=count)
    ctx = tukey.Context(dev.index)
    s = ctx.stream(mem_budget_bytes=8 << 30)
    t0 = time.perf_counter()
    for tk in [s.submit(d.X, d.Zq) for d in reqs]:
        s.wait(tk)
    rate = len(reqs) / (time.perf_counter() - t0)
    lam = 0.7 * rate
    rnd = random.Random(5)
    lat, done_sweeps, refused = [], 0, 0
    t_start = time.perf_counter()
    next_t = t_start
    pending, k = [], 0
    while time.perf_counter() - t_start < seconds or pending:
        now = time.perf_counter()
        if now >= next_t and now - t_start < seconds:
            d = reqs[k % len(reqs)]
            k += 1
            tk = s.submit(d.X, d.Zq)
            if tk is not None:
                pending.append((tk, next_t, d))
            else:
                refused += 1
            next_t += rnd.expovariate(lam)
        still = []
        for tk, ta, d in pending:
            if s.poll(tk) is not None:
                lat.append((time.perf_counter() - ta, d.p))
                done_sweeps += comb(d.n, d.p - 2) * d.m
            else:
                still.append((tk, ta, d))
        pending = still
        time.sleep(0.0002)
    el = time.perf_counter() - t_start

    def pct(v):
        v = sorted(v)
        return {"p50_ms": 1e3 * v[len(v) // 2], "p99_ms": 1e3 * v[min(len(v) - 1, int(0.99 * len(v)))],
                "requests": len(v)} if v else None
    by_p = {str(p): pct([t for t, pp in lat if pp == p]) for p in (3, 4, 5, 6)}
    out = {"workload": "W5: the first %d requests of the stream (p in {3,4,5,6}, n in [50,1000], "
                       "p=6 n<=120, 1-64 queries), cycled, Poisson arrivals" % count,
           "arrival_rate_per_s": lam, "calibrated_rate_per_s": rate, "seconds": el,
           "throughput_requests_per_s": len(lat) / el, "throughput_sweeps_per_s": done_sweeps / el,
           "refused": refused, "dropped_from_sample": 0, "by_p": by_p}
    out.update(pct([t for t, _ in lat]))
    return out


def _cpu_baseline(d, seconds):
    """The CPU oracle, as it stands, on one host core: a bounded sample of the
    same workload (the first subset positions of query 0)."""
    import oracle
    oracle.build()
    z = d.Zq[0]
    t = time.perf_counter()
    oracle.depth_range(d.X, z, 0, 500)
    rate = 500 / max(time.perf_counter() - t, 1e-6)
    S = int(max(1000, min(rate * seconds, 2_000_000)))
    t = time.perf_counter()
    _, npos, ctr = oracle.depth_range(d.X, z, 0, S)
    dt = time.perf_counter() - t
    swept = ctr[0] - ctr[1]
    return {"value": swept / dt, "unit": UNIT, "cores": 1, "kind": "oracle",
            "sample": "query 0, subset positions [0, %d) of %d (%.1f s single-threaded)" % (S, npos, dt)}


def run_reference(a):
    ws, rank, _ = _dist()
    if rank != 0:
        return
    d = _workload(0, True)
    import oracle
    oracle.build()
    z = d.Zq[0]
    t = time.perf_counter()
    oracle.depth_range(d.X, z, 0, 300)
    rate = 300 / max(time.perf_counter() - t, 1e-6)
    # each step: a bounded sample sized so that warmup + steps end in ~2 minutes
    per_step = max(200, int(rate * min(8.0, 120.0 / max(a.steps + a.warmup, 1))))
    times, swept = [], 0
    for s in range(a.warmup + a.steps):
        q = d.Zq[s % d.m]
        t = time.perf_counter()
        _, npos, ctr = oracle.depth_range(d.X, q, 0, per_step)
        dt = time.perf_counter() - t
        if s >= a.warmup:
            times.append(dt)
            swept += ctr[0] - ctr[1]
    total = sum(times)
    value = swept / total
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws,
            "steps": a.steps, "warmup": a.warmup, "ms_per_step": 1e3 * total / len(times),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "i128",
            "data": "synthetic",
            "config": {"workload": WORKLOAD, "global_batch": d.m, "seq_len": None, "parallelism": "cpu1"},
            "cpu_baseline": {"kind": "oracle", "cores": 1, "value": value, "unit": UNIT,
                             "sample": "each step: subset positions [0, %d) of one query" % per_step},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def run_ours(a):
    import torch
    ws, rank, local = _dist()
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    from paper_1409_3901_gb300 import tukey

    strong = ws > 1 and a.scaling == "strong"
    d = _workload(rank, strong)
    stream = torch.cuda.current_stream(dev)
    shard = {"shard_index": rank, "shard_count": ws} if strong else {}
    ctx = tukey.Context(local, device_pointers=True, stream=stream.cuda_stream, **shard)
    Xd = torch.from_numpy(d.X).to(dev)
    Zd = torch.from_numpy(d.Zq).to(dev)
    out = torch.empty(d.m, dtype=torch.int32, device=dev)
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.int32, device=dev)

    def step():
        ctx.depth(Xd, Zd, out)
        if strong:
            # the exchange step of the sharded subset loop: MIN over the ranks
            dist.all_reduce(out, op=dist.ReduceOp.MIN)

    for _ in range(a.warmup):
        step()
    torch.cuda.synchronize(dev)
    if ws > 1:
        dist.barrier()
    clocks = _Clocks(local)
    clocks.start()
    evs = []
    sweeps = 0
    launches = 0
    ms_sweep = 0.0
    for _ in range(a.steps):
        flush.fill_(1)                           # L2 flush, outside the events
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        step()
        e1.record(stream)
        evs.append((e0, e1))
        st = ctx.last_stats
        sweeps += st.sweeps
        launches += st.kernel_launches
        ms_sweep += st.ms_sweep
    torch.cuda.synchronize(dev)
    clk = clocks.stop()
    ms_steps = [e0.elapsed_time(e1) for e0, e1 in evs]
    t_total = sum(ms_steps) / 1e3
    if ws > 1:
        tt = torch.tensor([t_total], device=dev, dtype=torch.float64)
        dist.all_reduce(tt, op=dist.ReduceOp.MAX)
        t_total = float(tt.item())
        sw = torch.tensor([sweeps], device=dev, dtype=torch.float64)
        dist.all_reduce(sw, op=dist.ReduceOp.SUM)
        sweeps_all = float(sw.item())
    else:
        sweeps_all = float(sweeps)
    value = sweeps_all / t_total
    queries_per_s = (1 if strong else ws) * d.m * a.steps / t_total
    check = None
    if strong:
        ck, want = _golden_w2()
        if want is not None and ck == d.checksum():
            check = bool(np.array_equal(out.cpu().numpy().astype(np.int64), want))

    # end to end through the public API with host buffers (copies inside;
    # with shards, the merged depths go through the MIN all-reduce)
    host = tukey.Context(local, stream=stream.cuda_stream, **shard)

    def e2e_step():
        o = host.depth(d.X, d.Zq)
        if strong:
            t_ = torch.from_numpy(o).to(dev)
            dist.all_reduce(t_, op=dist.ReduceOp.MIN)
            o = t_.cpu().numpy()
        return o

    e2e_step()
    e2e_steps = max(3, min(a.steps, 5))
    torch.cuda.synchronize(dev)
    if ws > 1:
        dist.barrier()
    t = time.perf_counter()
    e2e_sweeps = 0
    for _ in range(e2e_steps):
        o = e2e_step()
        e2e_sweeps += host.last_stats.sweeps
    e2e_t = time.perf_counter() - t
    if ws > 1:
        et = torch.tensor([e2e_t, float(e2e_sweeps)], device=dev, dtype=torch.float64)
        mx = et[:1].clone()
        dist.all_reduce(mx, op=dist.ReduceOp.MAX)
        dist.all_reduce(et, op=dist.ReduceOp.SUM)
        e2e_t, e2e_sweeps = float(mx.item()), float(et[1].item())
    e2e = {"value": e2e_sweeps / e2e_t, "unit": UNIT,
           "h2d_bytes_per_step": int(d.X.nbytes + d.Zq.nbytes), "d2h_bytes_per_step": int(o.nbytes)}
    if rank != 0 and ws > 1:
        dist.barrier()
        dist.destroy_process_group()
        return

    # the plain exact one-query-per-launch form on the same GPU
    plain = tukey.Context(local, mode=tukey.TD_MODE_PLAIN_EXACT, device_pointers=True,
                          stream=stream.cuda_stream)
    Zp = Zd[: a.plain_queries].contiguous()
    outp = torch.empty(Zp.shape[0], dtype=torch.int32, device=dev)
    plain.depth(Xd, Zp, outp)
    pm, psw = 0.0, 0
    for _ in range(2):
        flush.fill_(1)
        plain.depth(Xd, Zp, outp)
        pm += plain.last_stats.ms
        psw += plain.last_stats.sweeps
    plain_rate = psw / (pm / 1e3)
    same = bool(torch.equal(outp, out[: a.plain_queries]))

    # early-exit mode (reported apart from the full-sweep metric): the running
    # minimum starts at the data-direction bound and a query stops at V = 0
    early = tukey.Context(local, device_pointers=True, stream=stream.cuda_stream, early_exit=True)
    oute = torch.empty_like(out)
    early.depth(Xd, Zd, oute)
    em, esw, esk = 0.0, 0, 0
    e_steps = max(3, min(a.steps, 5))
    for _ in range(e_steps):
        flush.fill_(1)
        f0 = torch.cuda.Event(enable_timing=True)
        f1 = torch.cuda.Event(enable_timing=True)
        f0.record(stream)
        early.depth(Xd, Zd, oute)
        f1.record(stream)
        torch.cuda.synchronize(dev)
        em += f0.elapsed_time(f1)
        esw += early.last_stats.sweeps
        esk += early.last_stats.early_skipped
    # Algorithm 3 (ADIA) on the same queries, reported apart: its count is an
    # upper bound of T that the paper reports equal to T
    actx = tukey.Context(local, device_pointers=True, stream=stream.cuda_stream,
                         algorithm=tukey.TD_ALG_ADIA)
    outa = torch.empty_like(out)
    actx.depth(Xd, Zd, outa)
    am, asw, apops, aun, afb = 0.0, 0, 0, 0, 0
    for _ in range(e_steps):
        flush.fill_(1)
        f0 = torch.cuda.Event(enable_timing=True)
        f1 = torch.cuda.Event(enable_timing=True)
        f0.record(stream)
        actx.depth(Xd, Zd, outa)
        f1.record(stream)
        torch.cuda.synchronize(dev)
        am += f0.elapsed_time(f1)
        sa = actx.last_stats
        asw += sa.sweeps
        apops += sa.adia_pops
        aun += sa.adia_union_points
        afb += sa.adia_fallbacks
    adia_line = {"queries_per_s": d.m * e_steps / (am / 1e3), "ms_per_step": am / e_steps,
                 "step5_sweeps_per_step": asw // e_steps, "pops_per_step": apops // e_steps,
                 "mean_union_points": aun / e_steps / d.m, "fallbacks": afb,
                 "equal_to_exact": int((outa == out).sum().item()), "queries": d.m,
                 "note": "td_options.algorithm = TD_ALG_ADIA (Algorithm 3): search kernel, then the "
                         "filtered sweep over the subsets of the Step 5 union. Not the full-sweep metric."}
    early_line = {"queries_per_s": d.m * e_steps / (em / 1e3), "ms_per_step": em / e_steps,
                  "sweeps_per_step": esw // e_steps, "skipped_per_step": esk // e_steps,
                  "same_results": bool(torch.equal(oute, out)),
                  "note": "td_options.early_exit: data-direction upper bound (Algorithm 3 Step 2) "
                          "seeds each query's minimum; a query stops at V = 0. Not the full-sweep metric."}

    peaks, kind = _peaks()
    sm_max = float(peaks.get("sm_max_mhz", 2070.0))
    props = torch.cuda.get_device_properties(dev)
    peak_tops = props.multi_processor_count * 128 * sm_max * 1e6 / 1e12
    ops_per_call = _algorithmic_ops(d, sweeps / a.steps)
    if ms_sweep <= 0:
        raise SystemExit("the library reported no sweep-kernel time")
    achieved = ops_per_call * a.steps / (ms_sweep / 1e3) / 1e12
    roofline = {"bound": "alu", "achieved": achieved, "peak": peak_tops, "unit": "Tops/s",
                "frac": achieved / peak_tops, "traffic": _traffic_for_current_kernel(),
                "kernel": "td_k_filtered", "kernel_ms": ms_sweep / a.steps,
                "peak_basis": "%d SMs x 128 INT32/FP32 lanes x %.0f MHz (%s sm_max_mhz)"
                              % (props.multi_processor_count, sm_max, kind),
                "ops_basis": "strip bounds of whole fans (_fan_ops): per fan and point 3(p-2) + 5 + 10 "
                             "per strip, per subset 19 per strip, 8 strips; a sweep is one subset's "
                             "bound over all n' points, by these tables, by a pass over the points, "
                             "or exactly"}
    # the derived peak checked by measurement (after the timed region)
    from paper_1409_3901_gb300 import probe
    measured = {k: probe.issue_rate(k, local)[0] / 1e12 for k in probe.ISSUE_KINDS}
    measured["unit"] = "Tops/s"
    measured["note"] = ("td_issue_rate: independent chains over one full wave of blocks; "
                        "lane operations counted in the source (FMA = 1, f32x2 FMA = 2)")
    roofline["issue_rate_measured"] = measured
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": a.steps,
            "warmup": a.warmup, "ms_per_step": 1e3 * t_total / a.steps, "higher_is_better": True,
            "scaling": "strong" if strong else "weak", "vs_baseline": None, "dtype": "f32+i64/i128",
            "data": "synthetic",
            "config": {"workload": WORKLOAD, "global_batch": d.m * (1 if strong else ws), "seq_len": None,
                       "parallelism": ("subset-shards%d+allreduce-min" % ws) if strong else "dp%d" % ws,
                       "l2": "flushed between steps (512 MB write)"},
            "merged_depths_match_oracle": check,
            "queries_per_s": queries_per_s,
            "e2e": e2e, "gpu_launches": int(launches), "roofline": roofline,
            "plain_exact": {"value": plain_rate, "unit": UNIT, "queries": int(Zp.shape[0]),
                            "same_results": same, "speedup_filtered_over_plain": value / ws / plain_rate},
            "early_exit": early_line,
            "adia": adia_line,
            "stats_per_step": {k: v for k, v in ctx.last_stats.as_dict().items()},
            "exact_path": _exact_path(ctx.last_stats),
            "clocks": clk}
    if not a.no_extra:
        from paper_1409_3901_gb300 import workloads as W
        line["batched"] = _batched_w3(tukey, W, dev, stream, flush, peak_tops)
        line["tuning"] = _tuning(tukey, W, dev, stream, flush, 1e3 * t_total / a.steps,
                                 line["batched"]["ms_per_call"])
        line["stream"] = _stream_w5(tukey, W, dev, a.stream_seconds)
        line["small_w1"] = _small_w1(tukey, W, dev, stream, flush)
    if not a.no_cpu_baseline:
        line["cpu_baseline"] = _cpu_baseline(d, a.cpu_seconds)
    print(json.dumps(line), flush=True)
    if ws > 1:
        dist.barrier()
        dist.destroy_process_group()


def run_other(a):
    """Lines for the other workloads (one GPU, inputs from host memory)."""
    import torch
    from paper_1409_3901_gb300 import tukey, workloads as W
    torch.cuda.set_device(0)
    ctx = tukey.Context(0)
    if a.workload in ("W3", "W4", "W6"):
        sets = W.w3() if a.workload == "W3" else [W.WORKLOADS[a.workload]()]
        batch = [(d.X, d.Zq) for d in sets]
        for _ in range(max(1, a.warmup - 2)):
            ctx.depth_batched(batch)
        ms, msc, sw, ex, pts = [], [], 0, 0, 0
        for _ in range(a.steps):
            ctx.depth_batched(batch)
            st = ctx.last_stats
            ms.append(st.ms_sweep)
            msc.append(st.ms)
            sw += st.sweeps
            ex += st.exact_points
            pts += st.exact_points + st.filtered_points
        t = sum(ms) / 1e3
        nq = sum(d.m for d in sets)
        line = {"metric": METRIC, "value": sw / t, "unit": UNIT, "workload": a.workload,
                "datasets": len(sets), "queries": nq, "queries_per_s": nq * a.steps / t,
                "sweeps_per_call": sw // a.steps, "ms_per_call": 1e3 * t / a.steps,
                "exact_point_fraction": ex / max(pts, 1), "steps": a.steps,
                "ms_per_call_all_kernels": sum(msc) / a.steps,
                "queries_per_s_all_kernels": nq * a.steps / (sum(msc) / 1e3),
                "note": "sweep-kernel device time (td_stats.ms_sweep), one batched call per step; "
                        "*_all_kernels: set-up to finalize (td_stats.ms)"}
        if a.workload == "W4":
            line["critical_cross_check"] = _critical_cross_check(tukey, sets[0], ctx, a.steps)
        print(json.dumps(line), flush=True)
        return
    if a.workload == "W7":
        run_w7(a, tukey, W)
        return
    # W5: a stream of requests with Poisson arrivals, bounded sample
    import random
    from math import comb
    reqs = [d for d in W.w5(count=400) if comb(d.n, d.p - 2) * d.n <= 3e8][:120]
    s = ctx.stream(mem_budget_bytes=8 << 30)
    # calibration: back-to-back throughput over the whole sample
    t0 = time.perf_counter()
    tickets = [s.submit(d.X, d.Zq) for d in reqs]
    for tk in tickets:
        s.wait(tk)
    rate = len(reqs) / (time.perf_counter() - t0)
    lam = 0.7 * rate
    rnd = random.Random(5)
    lat, done_sweeps = [], 0
    t_start = time.perf_counter()
    next_t = t_start
    pending = []
    k = 0
    while time.perf_counter() - t_start < a.stream_seconds or pending:
        now = time.perf_counter()
        if now >= next_t and now - t_start < a.stream_seconds:
            d = reqs[k % len(reqs)]
            k += 1
            tk = s.submit(d.X, d.Zq)
            if tk is not None:
                pending.append((tk, next_t, d))
            next_t += rnd.expovariate(lam)
        still = []
        for tk, ta, d in pending:
            if s.poll(tk) is not None:
                lat.append(time.perf_counter() - ta)
                done_sweeps += comb(d.n, d.p - 2) * d.m
            else:
                still.append((tk, ta, d))
        pending = still
        time.sleep(0.0002)
    el = time.perf_counter() - t_start
    lat.sort()
    line = {"metric": "stream request latency", "workload": "W5", "unit": "ms",
            "p50": 1e3 * lat[len(lat) // 2], "p99": 1e3 * lat[min(len(lat) - 1, int(0.99 * len(lat)))],
            "requests": len(lat), "arrival_rate_per_s": lam, "calibrated_rate_per_s": rate,
            "throughput_requests_per_s": len(lat) / el, "throughput_sweeps_per_s": done_sweeps / el,
            "sample": "requests with C(n,p-2)*n <= 3e8 among the first 400 of the stream, cycled"}
    print(json.dumps(line), flush=True)


def _critical_cross_check(tukey, d, rcom, steps, count=64):
    """Proposition 1 with r = p-1 (TD_ALG_CRITICAL) on the first `count`
    queries: hyperplanes (p-1 subsets) per second, device time of the call,
    and agreement with Algorithm 1."""
    crit = tukey.Context(0, algorithm=tukey.TD_ALG_CRITICAL)
    Z = d.Zq[:count]
    want = rcom.depth(d.X, Z)
    crit.depth(d.X, Z)
    ms, hyp = 0.0, 0
    for _ in range(max(1, min(steps, 2))):
        got = crit.depth(d.X, Z)
        ms += crit.last_stats.ms
        hyp += crit.last_stats.sweeps
    reps = max(1, min(steps, 2))
    return {"queries": int(Z.shape[0]), "hyperplanes_per_s": hyp / (ms / 1e3), "ms_per_call": ms / reps,
            "hyperplanes_per_call": hyp // reps, "equal_to_algorithm_1": int((got == want).sum()),
            "note": "td_options.algorithm = TD_ALG_CRITICAL, one launch per query, exact int64"}


def run_w7(a, tukey, W):
    """The shapes of the paper's simulation (Section 5.2): Algorithm 1 (every
    subset, the exact count) against Algorithm 3 (ADIA), per (p, n) and per
    alpha, each cell one batched call over its 10 datasets; device time from
    the first to the last kernel of the call (td_stats.ms)."""
    sets = W.w7()
    rcom = tukey.Context(0)
    adia = tukey.Context(0, algorithm=tukey.TD_ALG_ADIA)

    def timed(ctx, batch):
        for _ in range(max(1, a.warmup - 2)):
            outs = ctx.depth_batched(batch)
        ms = 0.0
        for _ in range(a.steps):
            outs = ctx.depth_batched(batch)
            ms += ctx.last_stats.ms
        return ms / a.steps, outs, ctx.last_stats

    cells = []
    tot = {"rcom_ms": 0.0, "adia_ms": 0.0, "adia_shape_ms": 0.0, "queries": 0, "equal": 0}
    for p, n in W.W7_SHAPES:
        group = [d for d in sets if d.meta["p"] == p and d.meta["n"] == n]
        r_ms, r_out, r_st = timed(rcom, [(d.X, d.Zq) for d in group])
        nq = sum(d.m for d in group)
        tot["rcom_ms"] += r_ms
        tot["queries"] += nq
        s_ms, _, _ = timed(adia, [(d.X, d.Zq) for d in group])
        tot["adia_shape_ms"] += s_ms
        for ai, alpha in enumerate(W.W7_ALPHAS):
            batch = [(d.X, d.Zq[ai:ai + 1]) for d in group]
            a_ms, a_out, a_st = timed(adia, batch)
            exact = np.array([o[ai] for o in r_out])
            got = np.array([o[0] for o in a_out])
            eq = int((got == exact).sum())
            tot["adia_ms"] += a_ms
            tot["equal"] += eq
            cells.append({"p": p, "n": n, "alpha": alpha, "datasets": len(group),
                          "rcom_ms_per_query": r_ms / nq, "adia_ms_per_query": a_ms / len(group),
                          "adia_equal_to_exact": eq, "mean_exact_depth": float(exact.mean()),
                          "adia_pops": int(a_st.adia_pops), "adia_union_points": int(a_st.adia_union_points),
                          "adia_step5_sweeps": int(a_st.sweeps), "adia_fallbacks": int(a_st.adia_fallbacks)})
    line = {"metric": "query depths/s", "workload": "W7", "unit": "queries/s",
            "rcom_queries_per_s": tot["queries"] / (tot["rcom_ms"] / 1e3),
            "adia_queries_per_s": tot["queries"] / (tot["adia_ms"] / 1e3),
            "adia_queries_per_s_shape_batches": tot["queries"] / (tot["adia_shape_ms"] / 1e3),
            "queries": tot["queries"], "adia_equal_to_exact": tot["equal"], "steps": a.steps,
            "cells": cells,
            "note": "Algorithm 1 timed per (p, n) over its 40 queries, Algorithm 3 per (p, n, alpha) "
                    "over 10 queries (and per (p, n) over 40: *_shape_batches); td_stats.ms of one "
                    "batched call, averaged over the steps"}
    print(json.dumps(line), flush=True)


def run_profile_case(a):
    """A small, fixed case for ncu: td_depth twice on a few queries of a
    workload (the first call captures the CUDA graph, the second is the one to
    profile).  Launch order of one call:

    - rcom (Algorithm 1): set-up, tiles, td_k_filtered<2> .. <p>, finalize; at
      p = 4 `-k regex:td_k_filtered -s 5 -c 1` selects the second call's
      p = 4 sweep kernel, at p = 5 `-s 7`;
    - adia (Algorithm 3): the search kernels td_k_adia<3> .. <p> come before
      the sweep, so at p = 4 `-k regex:td_k_adia -s 3 -c 1` selects the second
      call's p = 4 search;
    - critical (Proposition 1, r = p - 1): one td_k_critical launch per query
      and call, so with one query `-k regex:td_k_critical -s 1 -c 1` selects
      the second call's.

    Every ncu command on a shared GPU takes `--clock-control none`."""
    from paper_1409_3901_gb300 import tukey, workloads as W
    workload = "W2" if a.workload in ("W3", "W5", "W7") else a.workload
    d = W.WORKLOADS[workload]()
    nq = a.profile_queries
    pick = [0, 40, 50, 63] if nq == 4 and d.m == 64 else list(range(0, d.m, max(1, d.m // nq)))[:nq]
    Z = d.Zq[pick]
    alg = {"rcom": tukey.TD_ALG_RCOM, "adia": tukey.TD_ALG_ADIA, "critical": tukey.TD_ALG_CRITICAL}[a.profile_case]
    ctx = tukey.Context(0, algorithm=alg)
    ctx.depth(d.X, Z)
    out = ctx.depth(d.X, Z)
    print(json.dumps({"profile_case": a.profile_case, "workload": workload, "queries": pick,
                      "out": out.tolist(), "stats": ctx.last_stats.as_dict()}), flush=True)


def main():
    a = _args()
    if a.profile_case:
        run_profile_case(a)
        return
    if a.warmup < 3:
        a.warmup = 3
    if a.impl == "reference":
        run_reference(a)
    elif a.workload != "W2":
        run_other(a)
    else:
        run_ours(a)


if __name__ == "__main__":
    main()
