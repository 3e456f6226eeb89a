#!/usr/bin/env python
"""Benchmark: exact lexicographic enumeration of one large factorization set.

Workload (single GPU): d = 6 generators drawn from seed 0 uniformly in
[50, 200] (distinct, sorted, gcd 1) and n the smallest element with
|Z(n)| >= 5e8 (found with the library's own device counting) -- about 12 GB
of int32 tuples per step.  One step is the whole path on the device: the
counting table, the memo build (elementwise batches of copy-and-increment),
and the rank-sliced enumeration writing every tuple to HBM.

Printed: one JSON line (rank 0).  `value` is factorizations/s with the
generators already on the device side, the memo depth and work-item size
chosen by the library's tuner in the warm-up (`config.k_choice` lists every
timed candidate); `e2e` is the same metric through fz_enumerate_host (plan,
enumeration and the device->host copy of every tuple into pinned host memory
inside the timed region; `e2e.pageable` and `e2e.pageable_staged` into a
plain numpy array); `roofline` is the enumeration kernel's written bytes per
launch over its CUDA-event time against the measured HBM copy bandwidth,
with the DRAM traffic of a committed ncu record; `cpu_baseline` is the
oracle (plain C recursion) on a bounded sample of the same workload on the
host cores; `secondary` holds bounded records of the other workloads: the
d = 5 memo build of all Z(0..1500), the 4096-instance batch (measured memo
policy, pipelined steps, against per-instance plans) and serving (grouped and
per-request launches and one request at a time, with a sweep of offered
rates).

`--impl reference` times that oracle alone, on the same workload and metric.
Under torchrun each rank runs its own replica of the workload (weak scaling,
no data exchange); times are the max over ranks.
"""
import argparse
import hashlib
import json
import re
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "Factorizations/s (exact, lex order) vs HBM roofline; served p50/p99 latency"
UNIT = "factorizations/s"
WORKLOAD = ("single large element: d=6 generators uniform in [50,200] (seed 0, distinct, "
            "sorted, gcd 1), n = smallest with |Z(n)| >= 5e8, int32 tuples, memo depth and "
            "work-item size chosen by fz_autotune_report (measured in the warm-up)")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--seed", type=int, default=0)
    ap.add_argument("--e2e-steps", type=int, default=2)
    ap.add_argument("--pg-timeout", type=float, default=300.0,
                    help="seconds a collective waits for a rank that has left (N > 1)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-autotune", action="store_true",
                    help="memo depth by the library's size rule instead of measuring")
    ap.add_argument("--no-secondary", action="store_true",
                    help="skip the batch / serve / memo records appended to the line")
    ap.add_argument("--no-graph", action="store_true",
                    help="launch every step's kernels directly instead of replaying a graph")
    ap.add_argument("--no-pipeline", action="store_true",
                    help="time steps one after another instead of overlapping each step's "
                         "count/memo build with the previous step's enumeration")
    ap.add_argument("--k", type=int, default=-1, help="memo depth (default: autotune)")
    ap.add_argument("--slice-rows", type=int, default=0)
    ap.add_argument("--cpu-seconds", type=float, default=15.0,
                    help="target duration of the bounded oracle sample")
    ap.add_argument("--target", type=int, default=0,
                    help="|Z(n)| target of the workload (default 5e8; smaller values give "
                         "the small profiling case)")
    ap.add_argument("--workload", choices=["single", "batch", "serve", "memo", "table1"],
                    default="single",
                    help="single: one large element (default line); batch: 4096 instances "
                         "in one launch vs per-instance launches; serve: Poisson request "
                         "stream over 64 resident sets; memo: dynamic build of all "
                         "Z(0..1500); table1: the paper's Table 1 instances")
    ap.add_argument("--serve-seconds", type=float, default=10.0)
    ap.add_argument("--batch-count", type=int, default=4096)
    ap.add_argument("--batch-pi-steps", type=int, default=5,
                    help="steps of the per-instance comparison (0: skip it)")
    ap.add_argument("--batch-d", type=int, default=0,
                    help="batch workload: keep only the instances with this many generators")
    return ap.parse_args()


# ---------------------------------------------------------------- workload
def resolve_instance(count_upto, seed, target=0):
    from paper_2407_20474_gb300 import workloads
    g = workloads.config2_generators(seed)
    n = workloads.find_n(count_upto, g, target or workloads.CONFIG2_TARGET, 4096)
    return g, n


# ---------------------------------------------------------- clock sampling
class ClockSampler:
    """nvidia-smi clocks / throttle reasons sampled in the background."""
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index=0, period_ms=50):
        self.path = tempfile.mktemp(suffix=".csv")
        self.proc = None
        try:
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(gpu_index), "--query-gpu=" + self.FIELDS,
                 "--format=csv,noheader,nounits", "-lms", str(period_ms)],
                stdout=self.fh, stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None
        self.t0 = self.t1 = None

    def mark_start(self):
        self.t0 = time.time()

    def mark_end(self):
        self.t1 = time.time()

    def stop(self):
        if self.proc is None:
            return None
        time.sleep(0.15)
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.fh.close()
        sms, maxes, reasons = [], [], set()
        with open(self.path) as f:
            for line in f:
                p = [x.strip() for x in line.split(",")]
                if len(p) < 9:
                    continue
                try:
                    sm = float(p[1])
                    mx = float(p[2])
                except ValueError:
                    continue
                sms.append(sm)
                maxes.append(mx)
                names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown",
                         "sw_power_cap"]
                for name, flag in zip(names, p[5:9]):
                    if flag.lower() == "active":
                        reasons.add(name)
        os.unlink(self.path)
        if not sms:
            return None
        return {"sm_mhz": statistics.median(sms), "sm_max_mhz": max(maxes),
                "reasons": sorted(reasons), "samples": len(sms)}


# ------------------------------------------------------------ distributed
def dist_setup(args):
    """One process per GPU from the torchrun environment.  A collective
    that waits on a rank that has left ends with an error after
    args.pg_timeout seconds (or as soon as the peer's connection closes)
    instead of hanging."""
    import datetime
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    pg = None
    if world > 1:
        import torch.distributed as dist
        backend = "nccl" if args.impl == "ours" else "gloo"
        if backend == "nccl":
            import torch
            torch.cuda.set_device(local)
        dist.init_process_group(backend=backend,
                                timeout=datetime.timedelta(seconds=float(args.pg_timeout)))
        pg = dist
    return world, rank, local, pg


def barrier(pg, torch=None):
    if pg is not None:
        if torch is not None:
            pg.barrier(device_ids=[torch.cuda.current_device()])
        else:
            pg.barrier()


def max_over_ranks(pg, value, torch=None):
    if pg is None:
        return value
    if torch is not None:
        t = torch.tensor([value], dtype=torch.float64, device="cuda")
    else:
        import torch as _t
        t = _t.tensor([value], dtype=_t.float64)
    pg.all_reduce(t, op=pg.ReduceOp.MAX)
    return float(t.item())


# ------------------------------------------------------------ cpu baseline
def cpu_baseline(g, n, seconds, count_table=None):
    """The oracle (plain C recursion, unchanged) on a bounded sample of the
    same workload: the subtrees of every s-th value of a_1, walked on all host
    cores; s is chosen so the run lasts about `seconds`."""
    import numpy as np
    import oracle
    T = count_table if count_table is not None else oracle.count_table(g, n)
    vals = np.arange(n // g[0], -1, -1, dtype=np.int64)
    sizes = np.asarray(T[1][n - g[0] * vals], dtype=np.float64)
    total = float(sizes.sum())
    threads = os.cpu_count() or 1
    # calibration on a small strided sample
    stride = 64
    t0 = time.perf_counter()
    rows, _, used = oracle.sample_a1(g, n, vals[::stride], threads=threads)
    dt = max(time.perf_counter() - t0, 1e-6)
    rate = rows / dt
    want_rows = rate * seconds
    stride = max(1, int(round(total / max(want_rows, 1.0))))
    sample = vals[::stride]
    t0 = time.perf_counter()
    rows, digest, used = oracle.sample_a1(g, n, sample, threads=threads)
    dt = time.perf_counter() - t0
    return {"value": rows / dt, "unit": UNIT, "cores": used, "kind": "oracle",
            "sample": "rows of Z(n) whose a_1 is every %d-th value (%d of %d values, "
                      "%d rows = %.2f%% of |Z|), plain recursion on %d threads, %.1f s"
                      % (stride, sample.size, vals.size, rows, 100.0 * rows / total,
                         used, dt),
            "rows": rows, "seconds": dt}


# --------------------------------------------------------------- our impl
def kernel_traffic(d):
    """dram bytes per launch of the enumeration kernel from the committed ncu
    summary, if it was taken on the current kernel source; else None."""
    path = os.path.join(ROOT, "profiles", "enum_kernel_traffic.json")
    if not os.path.exists(path):
        return None
    try:
        rec = json.load(open(path))
    except ValueError:
        return None
    csrc = os.path.join(ROOT, "paper_2407_20474_gb300", "csrc")
    src = ""
    for name in ("fz_enum.cu", "fz_enum.cuh", "fz_flat.cu", "fz_walk.cuh"):
        path = os.path.join(csrc, name)
        if os.path.exists(path):
            src += open(path).read()
    if rec.get("code_sha256") != code_hash(src):
        return None
    return rec.get("bytes_per_full_launch")


def code_hash(src):
    """sha256 of CUDA source with comments, blank lines and trailing spaces
    removed: edits to comments do not invalidate a profile of the code."""
    src = re.sub(r"/\*.*?\*/", "", src, flags=re.S)
    src = re.sub(r"//[^\n]*", "", src)
    lines = [l.rstrip() for l in src.splitlines()]
    return hashlib.sha256("\n".join(l for l in lines if l).encode()).hexdigest()


def enum_kernel_name(plan):
    """Name of the enumeration kernel the plan launches (without a memo the rank
    walk's, widths 4 to 7, when there are more than 3 prefixes a row)."""
    d, k = plan.d, plan.k
    if k == 0 and 3 <= d <= 9:
        flat = "fz_enum_flat_kernel<%d, %d, 1>" % (d, d - 2)
        return flat + (" or fz_enum_rank_kernel<%d>" % d if 4 <= d <= 7 else "")
    if plan.run_order:
        # the flat walk's widths and prefix lengths; else the run copy
        if 3 <= d <= 9 and 1 <= d - k - 1 <= 3:
            return "fz_enum_flat_kernel<%d, %d, 0>" % (d, d - k - 1)
        return "fz_enum_runs_kernel<%d, %d, %d>" % (d, d - k - 1, k)
    return "fz_enum_kernel<%d>" % d


def run_ours(args):
    import torch
    import __graft_entry__
    world, rank, local, pg = dist_setup(args)
    __graft_entry__.build()
    import paper_2407_20474_gb300 as fz
    torch.cuda.set_device(local)
    dev = torch.cuda.current_device()
    g, n = resolve_instance(lambda gg, nm: fz.fz_count_upto(gg, nm), args.seed, args.target)
    d = len(g)
    # memo depth k and work-item size: measured (fz_autotune_report times
    # every depth whose memo fits, at three work-item sizes, and the plan
    # below picks up the fastest) unless given on the command line
    k_choice = None
    if args.k == -1 and not args.no_autotune:
        t0 = time.perf_counter()
        (k_best, sl_best, ms_best), cands = fz.fz_autotune_report(g, n)
        k_choice = {"by": "fz_autotune_report: rebuild + enumeration of the whole set per "
                          "candidate, mean of 2 passes (measured in the warm-up)",
                    "k": k_best, "slice_rows": sl_best, "est_ms": ms_best,
                    "seconds": time.perf_counter() - t0,
                    "candidates": [{kk: (round(vv, 4) if isinstance(vv, float) else vv)
                                    for kk, vv in c.items()} for c in cands]}
    elif args.k == -1:
        k_choice = {"by": "size rule (choose_k: deepest k <= 4 whose memo stays small)"}
    else:
        k_choice = {"by": "command line"}
    plan = fz.Plan(g, n, k=args.k, slice_rows=args.slice_rows)
    count = plan.count
    out = torch.empty(count * d, dtype=torch.int32, device="cuda")
    stream = torch.cuda.current_stream()

    def step(ev=None):
        plan.rebuild()
        if ev is not None:
            ev[0].record(stream)
        plan.enumerate(out)
        if ev is not None:
            ev[1].record(stream)

    for _ in range(max(args.warmup, 0)):
        step()
    plan.sync()
    torch.cuda.synchronize()

    # the step (count tables, memo build, enumeration: about 16 dependent
    # launches) captured once as a CUDA graph and replayed
    graph = None
    if not args.no_graph:
        try:
            side = torch.cuda.Stream()
            side.wait_stream(stream)
            cg = torch.cuda.CUDAGraph()
            with torch.cuda.stream(side):
                plan.rebuild(stream=side)
                plan.enumerate(out, stream=side)
                side.synchronize()
                before = fz.fz_kernel_launches()
                with torch.cuda.graph(cg, stream=side):
                    plan.rebuild(stream=side)
                    plan.enumerate(out, stream=side)
                kernels_per_step = fz.fz_kernel_launches() - before
            torch.cuda.synchronize()
            plan.sync()
            graph = cg
        except Exception as e:
            graph = None
            graph_error = str(e)[:200]

    K = max(args.steps, 1)
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
           for _ in range(K)]
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    sampler = ClockSampler(dev) if rank == 0 else None
    if sampler:
        time.sleep(0.3)
    launches0 = fz.fz_kernel_launches()
    barrier(pg, torch)
    torch.cuda.synchronize()
    if sampler:
        sampler.mark_start()
    start.record(stream)
    if graph is not None:
        for i in range(K):
            graph.replay()
    else:
        for i in range(K):
            step(evs[i])
    end.record(stream)
    torch.cuda.synchronize()
    if sampler:
        sampler.mark_end()
    barrier(pg, torch)
    launches = fz.fz_kernel_launches() - launches0
    if graph is not None:
        launches = kernels_per_step * K  # graph replays launch the captured kernels
    plan.sync()
    ms = start.elapsed_time(end)
    ms_serial = ms
    pipelined = False
    enum_cap = depth = None
    trial_ms = {}
    if not args.no_pipeline:
        # Pipelined steps: `depth` plans of the same element take turns; the
        # count tables and memo builds of the next steps (latency-bound, 16
        # SMs each, one stream per plan) run while the current step's
        # enumeration (bandwidth-bound) runs on its own stream.  The
        # enumeration is capped at 4, 3 or 2 blocks per SM (larger rings at
        # lower caps) so the builds fit beside it.  The cap and the depth (2
        # or 3) are chosen in the warm-up.  Every step still does its whole
        # path.
        plans = [plan] + [fz.Plan(g, n, k=plan.k, slice_rows=args.slice_rows)
                          for _ in range(2)]
        s_bs = [torch.cuda.Stream() for _ in plans]
        s_e = torch.cuda.Stream()
        built = [torch.cuda.Event() for _ in plans]
        done = [torch.cuda.Event() for _ in plans]
        depth = 2

        def pipelined_steps(count_steps, kernel_evs=None):
            st0 = torch.cuda.Event(enable_timing=True)
            st1 = torch.cuda.Event(enable_timing=True)
            st0.record(s_e)
            for sb in s_bs:
                sb.wait_event(st0)
            for i in range(count_steps):
                j = i % depth
                if i >= depth:
                    s_bs[j].wait_event(done[j])
                plans[j].rebuild(stream=s_bs[j])
                built[j].record(s_bs[j])
                s_e.wait_event(built[j])
                if kernel_evs:  # enumeration launch time, on its own stream
                    kernel_evs[i][0].record(s_e)
                plans[j].enumerate(out, stream=s_e)
                if kernel_evs:
                    kernel_evs[i][1].record(s_e)
                done[j].record(s_e)
            st1.record(s_e)
            torch.cuda.synchronize()
            return st0.elapsed_time(st1)

        for dep in (2, 3):
            for cap in (4, 3, 2):
                depth = dep
                for p_ in plans:
                    p_.set_enum_ctas_per_sm(cap)
                pipelined_steps(dep + 1)
                c = max(args.warmup, 3) + dep
                trial_ms[(dep, cap)] = pipelined_steps(c) / c
        depth, enum_cap = min(trial_ms, key=trial_ms.get)
        for p_ in plans:
            p_.set_enum_ctas_per_sm(enum_cap)
        pipelined_steps(depth + 1)
        for p_ in plans:
            p_.sync()
        l0 = fz.fz_kernel_launches()
        barrier(pg, torch)
        if sampler:
            sampler.mark_start()
        pipe_evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
                    for _ in range(K)]
        ms_pipe = pipelined_steps(K, pipe_evs)
        if sampler:
            sampler.mark_end()
        barrier(pg, torch)
        launches = fz.fz_kernel_launches() - l0
        for p_ in plans:
            p_.sync()
        for p_ in plans[1:]:
            p_.close()
        plan.set_enum_ctas_per_sm(0)
        ms = ms_pipe
        pipelined = True
    ms = max_over_ranks(pg, ms, torch)
    if pipelined:
        # the enumeration launches of the timed (pipelined) steps
        enum_ms = statistics.mean(a.elapsed_time(b) for a, b in pipe_evs)
    elif graph is not None:
        # enumeration-kernel time measured on separate (non-graph) steps
        for i in range(min(K, 20)):
            step(evs[i])
        torch.cuda.synchronize()
        enum_ms = statistics.mean(a.elapsed_time(b) for a, b in evs[:min(K, 20)])
    else:
        enum_ms = statistics.mean(a.elapsed_time(b) for a, b in evs)
    clocks = sampler.stop() if sampler else None

    value = world * K * count / (ms / 1e3)
    bytes_per_launch = count * d * 4
    # plain device writes of the same bytes, reported beside the copy peak:
    # distinct words with 16-byte stores (fz_write_probe: the practical
    # write-only ceiling for data like ours), and one constant value
    # (fill_), which this GPU's memory system writes faster
    wbuf = out[:(out.numel() // 2) * 2].view(torch.int64)

    def write_gbs(fn):
        fn()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(3):
            fn()
        e1.record()
        torch.cuda.synchronize()
        return 3 * wbuf.numel() * 8 / (e0.elapsed_time(e1) / 1e3) / 1e9

    write_peak = write_gbs(lambda: fz.fz_write_probe(out, stream=stream))
    fill_const = write_gbs(lambda: wbuf.fill_(-1))
    achieved = bytes_per_launch / (enum_ms / 1e3) / 1e9
    peaks = {}
    pp = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(pp):
        peaks = json.load(open(pp))
    peak = peaks.get("hbm_gbs")
    peak_src = "measured" if peak else "fallback"
    if not peak:
        peak = 6800.0

    # end to end through the public host-buffer call
    e2e = None
    if not args.no_e2e:
        host = torch.empty(count * d, dtype=torch.int32, pin_memory=True)
        fz.fz_enumerate_host(g, n, host)   # warm-up (allocations, page-in)
        torch.cuda.synchronize()
        E = max(args.e2e_steps, 1)
        barrier(pg, torch)
        t0 = time.perf_counter()
        for _ in range(E):
            fz.fz_enumerate_host(g, n, host)
        torch.cuda.synchronize()
        t = time.perf_counter() - t0
        t = max_over_ranks(pg, t, torch)
        e2e = {"value": world * E * count / t, "unit": UNIT, "h2d_bytes_per_step": 4 * d,
               "d2h_bytes_per_step": count * d * 4,
               "note": "fz_enumerate_host: plan (count + memo), enumeration and D2H of "
                       "every tuple into pinned host memory, %d steps" % E}
        del host
        # the same call into pageable memory (a plain numpy array): written
        # by the kernel where the device reaches pageable memory through the
        # host's page tables, else through the page-locked staging ring; the
        # ring alone is timed beside it (128 MB chunks)
        import numpy as np
        page = np.empty(count * d, dtype=np.int32)
        page.fill(0)                     # touch every page once, outside the timing
        for label, chunk in (("pageable", 0),
                             ("pageable_staged", (128 << 20) // (4 * d))):
            fz.fz_enumerate_host(g, n, page, chunk_rows=chunk)  # warm-up
            barrier(pg, torch)
            t0 = time.perf_counter()
            for _ in range(E):
                fz.fz_enumerate_host(g, n, page, chunk_rows=chunk)
            t = time.perf_counter() - t0
            t = max_over_ranks(pg, t, torch)
            e2e[label] = {"value": world * E * count / t, "unit": UNIT,
                          "d2h_GBps": E * count * d * 4 / t / 1e9,
                          "note": ("fz_enumerate_host into a pageable numpy array (default "
                                   "path)" if chunk == 0 else
                                   "fz_enumerate_host_chunks into a pageable numpy array: "
                                   "128 MB chunks enumerated into page-locked staging buffers "
                                   "and copied by host threads while the next are made")}
        e2e["pinned_d2h_GBps"] = e2e["value"] / world * d * 4 / 1e9
        del page

    # the secondary workloads, bounded (about a minute together): batch,
    # serving (with a sweep of offered rates) and the d = 5 memo build
    secondary = None
    if rank == 0 and world == 1 and not args.no_secondary:
        secondary = {}
        for name, fn in (
                ("memo", lambda: measure_memo(torch, fz, 20, 3)),
                ("batch", lambda: measure_batch(torch, fz, 10, 3, 4096, 0, pi_steps=1)),
                ("serve", lambda: measure_serve(torch, fz, seconds=3.0,
                                                sweep_rates=(8000, 32000, 128000),
                                                sweep_requests=4000))):
            t0 = time.perf_counter()
            try:
                secondary[name] = fn()
            except Exception as e:  # reported, never hides the main line
                secondary[name] = {"error": repr(e)[:300]}
            secondary[name]["wall_s"] = time.perf_counter() - t0
        torch.cuda.synchronize()

    base = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        base = cpu_baseline(g, n, args.cpu_seconds)
        base = {k: v for k, v in base.items() if k not in ("rows", "seconds")}

    if rank == 0:
        rec = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": K,
            "warmup": args.warmup, "ms_per_step": ms / K, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "int32", "data": "synthetic",
            "config": {"workload": WORKLOAD, "g": list(g), "n": n, "count": count,
                       "k": plan.k, "k_choice": k_choice, "top": plan.top,
                       "memo_rows": plan.memo_rows,
                       "slice_rows": plan.slice_rows, "bytes_per_step": bytes_per_launch,
                       "parallelism": "replicas (one instance per GPU)",
                       "cuda_graph": graph is not None,
                       "pipelined": pipelined,
                       "pipeline_enum_ctas_per_sm": enum_cap if pipelined else None,
                       "pipeline_depth": depth if pipelined else None,
                       "pipeline_trials_ms_per_step": (
                           {"depth%d_cap%d" % k_: round(v_, 4) for k_, v_ in trial_ms.items()}
                           if pipelined else None),
                       "ms_per_step_serial": ms_serial / K,
                       "l2": "output %.1f GB per step >> 129 MB L2; count table and memo "
                             "rebuilt every step" % (bytes_per_launch / 1e9)},
            "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                         "frac": achieved / peak, "traffic": kernel_traffic(d),
                         "kernel": enum_kernel_name(plan),
                         "kernel_ms": enum_ms, "peak_source": peak_src,
                         "write_peak_gbs": write_peak,
                         "write_peak_kind": "fz_write_probe into the output buffer "
                                            "(distinct words, 16-byte stores)",
                         "frac_of_write_peak": achieved / write_peak,
                         "constant_fill_gbs": fill_const,
                         "algorithmic_bytes_per_launch": bytes_per_launch},
            "cpu_baseline": base,
            "e2e": e2e,
            "clocks": clocks,
            "gpu_launches": launches,
        }
        if secondary is not None:
            rec["secondary"] = secondary
        print(json.dumps(rec))
    plan.close()
    if pg is not None:
        pg.destroy_process_group()


# --------------------------------------------------------- reference arm
def run_reference(args):
    world, rank, local, pg = dist_setup(args)
    if rank != 0:
        if pg is not None:
            pg.destroy_process_group()
        return
    import oracle
    from oracle import build as ob
    ob.build_oracle()
    g, n = resolve_instance(oracle.count_upto, args.seed, args.target)
    T = oracle.count_table(g, n)
    count = int(T[0][n])
    K = max(args.steps, 1)
    W = max(args.warmup, 0)
    # each step: a bounded sample of the workload; keep the whole run short
    per_step = max(0.5, min(args.cpu_seconds, 120.0 / (K + W)))
    res = []
    for i in range(W + K):
        r = cpu_baseline(g, n, per_step, count_table=T)
        if i >= W:
            res.append(r)
    rows = sum(r["rows"] for r in res)
    secs = sum(r["seconds"] for r in res)
    value = rows / secs
    rec = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
        "steps": K, "warmup": W, "ms_per_step": 1e3 * secs / K, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "int32", "data": "synthetic",
        "config": {"workload": WORKLOAD, "g": list(g), "n": n, "count": count},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": res[-1]["cores"],
                         "kind": "oracle", "sample": res[-1]["sample"]},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                "d2h_bytes_per_step": 0},
    }
    print(json.dumps(rec))
    if pg is not None:
        pg.destroy_process_group()


# ---------------------------------------------------------- other workloads
def _gpu_env():
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2407_20474_gb300 as fz
    torch.cuda.set_device(0)
    return torch, fz


def _event_time(torch, fn, steps, warmup):
    for _ in range(warmup):
        fn()
    torch.cuda.synchronize()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    for _ in range(steps):
        fn()
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b) / steps


def measure_batch(torch, fz, steps, warmup, count=4096, only_d=0, pi_steps=5, autotune=True,
                  pipeline=True):
    """The batch: ``count`` instances (d 3..8, generators in [2,300], |Z|
    log-uniform in [1e2,1e6]) in one persistent launch -- the step (batched
    counting tables, memos and enumeration) replayed as a captured CUDA
    graph -- against the same instances launched one plan at a time.
    Returns a record (dict)."""
    from paper_2407_20474_gb300 import workloads
    t_setup = time.perf_counter()
    insts = workloads.config4_instances(2, count)
    if only_d:
        insts = [x for x in insts if len(x.g) == only_d]
    inst = [(x.g, workloads.find_n(fz.fz_count_upto, x.g, x.target, 64)) for x in insts]
    tune = None
    if autotune:
        # memo depth policy and layout per tuple width, measured on samples
        t0 = time.perf_counter()
        cands, chosen = fz.fz_batch_autotune(inst)
        tune = {"by": "fz_batch_autotune: rebuild + enumeration of the instances of each "
                      "width (up to 1024) under each candidate (measured)",
                "seconds": time.perf_counter() - t0,
                "chosen": {str(d): {"cap_rows": c, "run_order": r}
                           for d, (c, r) in chosen.items()},
                "candidates": [{k: (round(v, 4) if isinstance(v, float) else v)
                                for k, v in c.items()} for c in cands]}
    b = fz.Batch(inst)
    out = torch.empty(int(b.total_words) + 16, dtype=torch.int32, device="cuda")
    side = torch.cuda.Stream()
    graph_ok = True
    graph_err = None
    try:
        cg = torch.cuda.CUDAGraph()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            b.rebuild(stream=side)
            b.enumerate(out, stream=side)
            side.synchronize()
            with torch.cuda.graph(cg, stream=side):
                b.rebuild(stream=side)
                b.enumerate(out, stream=side)
        torch.cuda.synchronize()
        step = cg.replay
    except Exception as e:  # capture unsupported: plain launches
        graph_ok = False
        graph_err = str(e)[:200]

        def step():
            b.rebuild()
            b.enumerate(out)
    ms = _event_time(torch, step, max(steps, 1), max(warmup, 1))
    b.sync()
    # the two halves of the step, each timed alone (plain launches)
    ms_rebuild = _event_time(torch, b.rebuild, max(steps, 1), 1)
    ms_enum = _event_time(torch, lambda: b.enumerate(out), max(steps, 1), 1)
    b.sync()
    ms_serial = ms
    pipe = None
    if pipeline:
        # Pipelined steps, as for the single large set: two batches of the
        # same instances take turns; one's rebuild (tables and memos, latency-bound) runs on
        # its own stream while the other's enumeration runs on another, the
        # enumeration capped at 4, 3 or 2 blocks per SM (chosen in the
        # warm-up) so the rebuild's blocks fit beside it.  Every step still
        # rebuilds all tables and memos and enumerates every instance.
        bs = [b, fz.Batch(inst)]
        s_bs = [torch.cuda.Stream() for _ in bs]
        s_e = torch.cuda.Stream()
        built = [torch.cuda.Event() for _ in bs]
        done = [torch.cuda.Event() for _ in bs]

        def pipelined(count):
            st0 = torch.cuda.Event(enable_timing=True)
            st1 = torch.cuda.Event(enable_timing=True)
            st0.record(s_e)
            for sb in s_bs:
                sb.wait_event(st0)
            for i in range(count):
                j = i % 2
                if i >= 2:
                    s_bs[j].wait_event(done[j])
                bs[j].rebuild(stream=s_bs[j])
                built[j].record(s_bs[j])
                s_e.wait_event(built[j])
                bs[j].enumerate(out, stream=s_e)
                done[j].record(s_e)
            st1.record(s_e)
            torch.cuda.synchronize()
            return st0.elapsed_time(st1) / count

        trials = {}
        for cap in (4, 3, 2):
            for x in bs:
                x.set_enum_ctas_per_sm(cap)
            pipelined(3)
            trials[cap] = pipelined(max(warmup, 3) + 2)
        cap = min(trials, key=trials.get)
        for x in bs:
            x.set_enum_ctas_per_sm(cap)
        pipelined(3)
        ms_pipe = pipelined(max(steps, 1))
        for x in bs:
            x.sync()
            x.set_enum_ctas_per_sm(0)
        bs[1].close()
        pipe = {"ms_per_step": ms_pipe, "enum_ctas_per_sm": cap,
                "trials_ms_per_step": {str(k): round(v, 4) for k, v in trials.items()}}
        if ms_pipe < ms:
            ms = ms_pipe
    bytes_out = sum(int(r) * len(g) * 4 for (g, _), r in zip(inst, b.rows))
    # per-instance launches of the same instances
    ms_pi = None
    if pi_steps > 0:
        plans = [fz.Plan(gg, n) for gg, n in inst]
        offs = [int(x) for x in b.word_offsets]

        def per_instance():
            for i, p in enumerate(plans):
                if p.count:
                    p.rebuild()
                    p.enumerate(out[offs[i]:], capacity_rows=p.count)
        ms_pi = _event_time(torch, per_instance, pi_steps, 1)
        for p in plans:
            p.close()
    peak = _hbm_peak()
    rec = {"workload": "batched: %d instances, d uniform 3..8, generators uniform [2,300] "
                       "(distinct, gcd 1), |Z| log-uniform [1e2,1e6], seed 2%s"
                       % (len(inst), (", only d = %d" % only_d) if only_d else ""),
           "instances": len(inst), "total_rows": int(b.total_rows), "bytes_out": bytes_out,
           "ms_per_step": ms, "value": b.total_rows / (ms / 1e3), "unit": UNIT,
           "memos": b.memos, "run_order_instances": b.run_order,
           "run_order_memos": b.run_memos, "work_items": b.work_items,
           "cuda_graph": graph_ok, "ms_per_step_serial": ms_serial, "pipelined": pipe,
           "rebuild_ms": ms_rebuild, "enumerate_ms": ms_enum,
           "per_instance_ms_per_step": ms_pi,
           "per_instance_value": b.total_rows / (ms_pi / 1e3) if ms_pi else None,
           "speedup_vs_per_instance": ms_pi / ms if ms_pi else None,
           "roofline_enumeration": {
               "bound": "hbm", "kernel": "fz_flat_batch_kernel",
               "achieved": bytes_out / (ms_enum / 1e3) / 1e9, "peak": peak[0],
               "unit": "GB/s", "frac": bytes_out / (ms_enum / 1e3) / 1e9 / peak[0],
               "peak_source": peak[1]},
           "memo_policy": tune if tune else "hand-set rule (cap 4x rows at d >= 6, 1x below)",
           "setup_s": time.perf_counter() - t_setup}
    if graph_err:
        rec["graph_error"] = graph_err
    b.close()
    return rec


def run_batch_workload(args):
    torch, fz = _gpu_env()
    r = measure_batch(torch, fz, args.steps, args.warmup, args.batch_count, args.batch_d,
                      pi_steps=args.batch_pi_steps, autotune=not args.no_autotune,
                      pipeline=not args.no_pipeline)
    rec = {"metric": "Factorizations/s, batched (%d instances, one persistent launch)"
                     % r["instances"],
           "value": r["value"], "unit": UNIT, "n_gpus": 1, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": r["ms_per_step"], "higher_is_better": True,
           "dtype": "int32", "data": "synthetic",
           "config": {k: v for k, v in r.items() if k not in ("value", "unit", "ms_per_step")}}
    print(json.dumps(rec))


def _hbm_peak():
    pp = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(pp):
        v = json.load(open(pp)).get("hbm_gbs")
        if v:
            return float(v), "measured"
    return 6800.0, "fallback"


def measure_serve(torch, fz, seconds=10.0, sweep_rates=(), sweep_requests=4000,
                  serial=True):
    """Serving: an open-loop Poisson stream (2000 req/s) of queries over 64
    resident generator sets (d 4..7, generators in [5,500]), |Z| log-uniform
    in [1e3,1e7]; continuous batching against one-request-at-a-time serving.
    ``sweep_rates`` replays the same query mix at higher offered rates,
    ``sweep_requests`` requests each, in both modes, to find the sustainable
    rate.
    Returns a record (dict)."""
    import numpy as np
    from paper_2407_20474_gb300 import workloads
    t_setup = time.perf_counter()
    base = workloads.config5_stream(3, duration_s=seconds)
    sets = base.sets
    # per set: counts up to the element of the largest target, then each
    # request's n = the smallest element reaching its target
    n_max, set_counts = [], []
    for g in sets:
        nm = workloads.find_n(fz.fz_count_upto, g, int(base.targets.max()), 1024)
        set_counts.append(fz.fz_count_upto(g, nm).astype(np.float64))
        n_max.append(nm)

    def n_for(set_index, targets):
        return np.array([int(np.argmax(set_counts[s_i] >= t))
                         for s_i, t in zip(set_index, targets)], dtype=np.int64)

    def replay(srv, ids, arrivals, set_index, ns):
        # the library's native replay: submissions at the arrival times
        # and the drain run on native threads, so the client's interpreter
        # does not bound the measured rate
        import numpy as np
        m = len(ns)
        sid = np.asarray([ids[i] for i in set_index], dtype=np.int32)
        lat, rows, span = srv.replay(sid, np.asarray(ns, dtype=np.int32),
                                     np.asarray(arrivals, dtype=np.float64))
        offered_span = float(arrivals[-1]) if m else 0.0
        return {"p50_ms": 1e3 * float(np.percentile(lat, 50)),
                "p99_ms": 1e3 * float(np.percentile(lat, 99)),
                "mean_ms": 1e3 * float(lat.mean()),
                "throughput": float(rows.sum() / span) if span > 0 else 0.0,
                "requests": int(m), "rows": float(rows.sum()),
                "offered_req_per_s": m / offered_span if offered_span > 0 else 0.0,
                "achieved_req_per_s": m / span if span > 0 else 0.0}

    def server(max_in_flight, streams, per_request):
        srv = fz.Server(max_in_flight=max_in_flight, streams=streams, per_request=per_request)
        ids = [srv.register(g, nm) for g, nm in zip(sets, n_max)]
        return srv, ids

    # continuous: the requests admitted together form one launch (default);
    # continuous_per_request: the same admission, one launch per request;
    # serial: one request on the device at a time
    modes = {"continuous": (64, 8, False), "continuous_per_request": (64, 8, True)}
    if serial:
        modes["serial_one_at_a_time"] = (1, 1, True)
    res = {}
    servers = {k: server(*v) for k, v in modes.items()}
    t_setup = time.perf_counter() - t_setup
    st = workloads.config5_stream(3, duration_s=seconds)
    ns = n_for(st.set_index, st.targets)
    for name, (srv, ids) in servers.items():
        replay(srv, ids, st.arrivals_s[:64], st.set_index[:64], ns[:64])  # warm-up
        res[name] = replay(srv, ids, st.arrivals_s, st.set_index, ns)
    sweep = {}
    for rate in sweep_rates:
        sw = workloads.config5_stream(3, rate=float(rate),
                                      duration_s=1.2 * sweep_requests / float(rate) + 0.01)
        m = min(sweep_requests, len(sw.arrivals_s))
        # targets above the largest the sets were sized for are clipped to it
        tg = np.minimum(sw.targets[:m], base.targets.max())
        nsw = n_for(sw.set_index[:m], tg)
        for name, (srv, ids) in servers.items():
            sweep.setdefault(name, []).append(
                dict(rate=float(rate),
                     **replay(srv, ids, sw.arrivals_s[:m], sw.set_index[:m], nsw)))
    for srv, _ in servers.values():
        srv.close()
    rec = {"workload": "served: Poisson %.0f req/s for %.1f s over 64 resident sets (d 4..7, "
                       "generators [5,500], gcd 1), |Z| log-uniform [1e3,1e7], seed 3"
                       % (st.rate, st.duration_s),
           "value": res["continuous"]["throughput"], "unit": UNIT,
           "p50_ms": res["continuous"]["p50_ms"], "p99_ms": res["continuous"]["p99_ms"],
           "setup_s": t_setup}
    rec.update(res)
    if sweep:
        sat = {}
        for name, pts in sweep.items():
            # sustainable: the request rate keeps up with the offered rate
            # (>= 95 %) and p99 stays within 10x of its value at 2000 req/s
            ok = [p for p in pts if p["achieved_req_per_s"] >= 0.95 * p["offered_req_per_s"]
                  and p["p99_ms"] <= 10.0 * res[name]["p99_ms"]]
            best = max(ok, key=lambda p: p["rate"]) if ok else None
            sat[name] = {"sustainable_rate": best["rate"] if best else None,
                         "throughput_at_sustainable": best["throughput"] if best else None,
                         "max_throughput": max(p["throughput"] for p in pts),
                         "points": pts}
        rec["saturation"] = sat
    return rec


def run_serve_workload(args):
    torch, fz = _gpu_env()
    r = measure_serve(torch, fz, args.serve_seconds,
                      sweep_rates=(4000, 8000, 16000, 32000, 64000, 128000, 256000),
                      sweep_requests=8000)
    rec = {"metric": "Served factorizations/s with p50/p99 latency (Poisson 2000 req/s)",
           "value": r["value"], "unit": UNIT, "n_gpus": 1, "higher_is_better": True,
           "dtype": "int32", "data": "synthetic",
           "p50_ms": r["p50_ms"], "p99_ms": r["p99_ms"],
           "config": {k: v for k, v in r.items() if k not in ("value", "unit")}}
    print(json.dumps(rec))


def measure_memo(torch, fz, steps, warmup):
    """The memo build: dynamic FactorizationsUpToElement build of all Z(0..1500) for
    d = 5 generators in [3,40] (seed 1): the full CSR, built level by level from
    run-order tables.  Timed on the device as the rebuild of a plan whose
    memo is that CSR (k = d, top = N + 1: count table, offsets, levels,
    no allocation), CUDA events over the steps; the one-shot
    host call fz_build_memo_into (which allocates its work buffers and
    synchronises) is timed beside it.  Returns a record (dict)."""
    from paper_2407_20474_gb300 import workloads
    g = workloads.config3_generators(1)
    N = workloads.CONFIG3_N
    rows = fz.fz_memo_rows(g, N + 1)
    with fz.Plan(g, N, k=len(g), top=N + 1) as plan:
        assert plan.memo_rows == rows
        ms = _event_time(torch, plan.rebuild, max(steps, 1), max(warmup, 1))
        plan.sync()
    off = torch.zeros(N + 2, dtype=torch.int64, device="cuda")
    buf = torch.empty(rows * len(g) + 16, dtype=torch.int32, device="cuda")
    ts = []
    for i in range(max(warmup, 1) + max(min(steps, 20), 1)):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        fz.fz_build_memo_into(g, N + 1, off, buf, rows)
        torch.cuda.synchronize()
        if i >= max(warmup, 1):
            ts.append(time.perf_counter() - t0)
    t_host = statistics.median(ts)
    nbatch = -(-(N + 1) // min(g))
    return {"workload": "d=5 generators %s (seed 1), N=%d" % (list(g), N),
            "value": rows / (ms / 1e3), "unit": "rows/s", "ms_per_step": ms,
            "rows": rows, "bytes_written": rows * len(g) * 4,
            "write_GBps": rows * len(g) * 4 / (ms / 1e3) / 1e9,
            "elementwise_batches": nbatch, "levels": len(g) - 1,
            "bound": "output write and table reads through L2 (built by levels)",
            "host_call_ms": 1e3 * t_host,
            "note": "value: device time of a plan rebuild (CUDA events); "
                    "host_call_ms: fz_build_memo_into incl. its allocations"}


def run_memo_workload(args):
    torch, fz = _gpu_env()
    r = measure_memo(torch, fz, args.steps, args.warmup)
    rec = {"metric": "Memo rows/s, dynamic build of all Z(0..N) (FactorizationsUpToElement)",
           "value": r["value"], "unit": "rows/s", "n_gpus": 1, "higher_is_better": True,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": r["ms_per_step"],
           "dtype": "int32", "data": "synthetic",
           "config": {k: v for k, v in r.items() if k not in ("value", "unit", "ms_per_step")}}
    print(json.dumps(rec))


def run_table1_workload(args):
    """The paper's Table 1 instances Z(n, first d of (13,37,38,40..45)) with
    the paper's memo depth, timed end to end on the device (count table +
    memo + enumeration, output resident), beside the paper's runtimes."""
    torch, fz = _gpu_env()
    from paper_2407_20474_gb300 import workloads
    rows_out = []
    table = [(3, 1, 100000, 2733), (3, 1, 200000, 7904), (3, 1, 300000, 16241),
             (4, 2, 5000, 400), (4, 2, 10000, 420), (4, 2, 15000, 679),
             (5, 2, 1000, 485), (5, 2, 3000, 1047), (5, 2, 5000, 2101), (5, 2, 10000, 7600),
             (5, 3, 1000, 502), (5, 3, 3000, 702), (5, 3, 5000, 953),
             (6, 3, 1000, 601), (6, 3, 3000, 1751), (6, 3, 5000, 6298),
             (6, 4, 1000, 1155), (6, 4, 2000, 4079), (6, 4, 3000, 10640),
             (7, 4, 1000, 1153), (7, 4, 1500, 2299), (7, 4, 2000, 5416),
             (8, 4, 1000, 1659), (8, 4, 1500, 5736), (8, 4, 2000, 25165),
             (9, 4, 500, 1326), (9, 4, 1000, 8202), (9, 4, 1500, 52694),
             (9, 5, 500, 1129), (9, 5, 1000, 6018), (9, 5, 1500, 47513)]
    # memo population per (d, memo_dim) group, up to the group's largest
    # element: the device build in each launch schedule (wall clock of the
    # synchronising call, median of 3) beside the paper's CPU and GPU columns
    # and the single-threaded CPU build of the oracle (cpu_baseline leg)
    import oracle
    paper_memo = {(3, 1): (313, 9764), (4, 2): (2920, 27188), (5, 2): (1674, 30028),
                  (5, 3): (7952, 26683), (6, 3): (7586, 27999), (6, 4): (43686, 24625),
                  (7, 4): (44906, 24383), (8, 4): (47843, 25655), (9, 4): (49239, 29815),
                  (9, 5): (21401, 18208)}
    memo_rows = []
    for (d, k), (paper_cpu_us, paper_gpu_us) in paper_memo.items():
        top = max(n for dd, kk, n, _ in table if (dd, kk) == (d, k)) + 1
        tail = workloads.TABLE1_GENERATORS[:d][d - k:]
        rows = fz.fz_memo_rows(tail, top)
        off = torch.zeros(top + 1, dtype=torch.int64, device="cuda")
        buf = torch.empty(max(rows, 1) * k, dtype=torch.int32, device="cuda")
        rec = {"d": d, "memo_dim": k, "top": top, "rows": rows,
               "paper_cpu_memo_us": paper_cpu_us, "paper_gpu_memo_us": paper_gpu_us}
        for name, sched in (("batched", fz.FZ_MEMO_BATCHED), ("per_batch", fz.FZ_MEMO_PER_BATCH),
                            ("per_copy", fz.FZ_MEMO_PER_COPY)):
            ts = []
            for _ in range(4):
                t0 = time.perf_counter()
                fz.fz_build_memo_schedule(tail, top, sched, off, buf, rows)
                ts.append(time.perf_counter() - t0)
            rec["gpu_memo_us_" + name] = 1e6 * statistics.median(ts[1:])
        ts = []
        for _ in range(3):
            t0 = time.perf_counter()
            oracle.lex_lists_c(tail, top)
            ts.append(time.perf_counter() - t0)
        rec["cpu_memo_us_oracle_1thread"] = 1e6 * statistics.median(ts)
        memo_rows.append(rec)
        del off, buf
    for d, k, n, paper_ms in table:
        g = workloads.TABLE1_GENERATORS[:d]
        with fz.Plan(g, n, k=k) as p:
            out = torch.empty(max(p.count, 1) * d, dtype=torch.int32, device="cuda")

            def step():
                p.rebuild()
                p.enumerate(out)
            ms = _event_time(torch, step, 5, 2)
            p.sync()
            rows_out.append({"d": d, "memo_dim": k, "n": n, "count": p.count, "ms": ms,
                             "fact_per_s": p.count / (ms / 1e3),
                             "paper_ms": paper_ms, "paper_fact_per_s": p.count / (paper_ms / 1e3)})
    total = sum(r["count"] for r in rows_out)
    ms = sum(r["ms"] for r in rows_out)
    rec = {"metric": "Factorizations/s on the paper's Table 1 instances (paper's memo depth)",
           "value": total / (ms / 1e3), "unit": UNIT, "n_gpus": 1, "higher_is_better": True,
           "dtype": "int32", "data": "synthetic",
           "config": {"workload": "Table 1: Z(n, first d of (13,37,38,40..45))", "rows": rows_out,
                      "memo_population": memo_rows,
                      "note": "paper: RTX 3080 + Ryzen 3900X, host-buffered output; here "
                              "output resident in HBM"}}
    print(json.dumps(rec))


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
    elif args.workload == "batch":
        run_batch_workload(args)
    elif args.workload == "serve":
        run_serve_workload(args)
    elif args.workload == "memo":
        run_memo_workload(args)
    elif args.workload == "table1":
        run_table1_workload(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
