#!/usr/bin/env python
"""Throughput of the exact component-matrix path on one GB300.

Workload (default): power-law bursty temporal network, n = 500,000 nodes,
m = 10^8 events (configuration-model degrees with exponent 2.5, Pareto(1.5,
60 s) inter-event gaps per link, times rounded down to seconds, so timestamp
groups hold thousands of events), seeded and synthetic; the component matrix is
31.3 GB.  One step is one pass of the whole exact path over that batch, inputs
resident in HBM: validation + schedule (tn_plan_create), S <- I
(tn_init_matrix), the column-slab event stream (tn_plan_apply), out-sizes +
largest out-component (tn_out_sizes).  The metric is bit-updates/s = n * m /
step time (also reported as events/s).  The plan options come from the
autotuner (tn_autotune) on a prefix of the events.

Prints one JSON line (rank 0).  `--impl reference` times the CPU oracle (the
only reference this project has) on a bounded sample of the same workload:
every event over a seeded subset of source columns, one column slab per host
thread, extrapolated linearly to all n columns (columns are independent).
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "events/s and bit-updates/s (n·m/time) at 1 GB300; achieved HBM GB/s vs peak"
ONLINE_METRIC = "events/s through the online state (batches that split timestamp groups)"
# ncu summaries under profiles/ and the sources whose hash they record (a summary
# taken on other sources gives no traffic figure)
STREAM_SOURCES = ["paper_2307_04890_gb300/csrc/tn_apply.cu", "paper_2307_04890_gb300/csrc/tn_internal.cuh",
                  "paper_2307_04890_gb300/csrc/tn_plan.cu"]
PROFILE_SUMMARIES = {"activity": ("stream_kernel_activity_n1e5_m1e7.txt", STREAM_SOURCES),
                     "bursty-scaled": ("stream_kernel_bursty_scaled_40000x503808_m2e6_traffic.txt", STREAM_SOURCES),
                     "online": ("grow_kernel_online_n1e5_to_102048.txt",
                                ["paper_2307_04890_gb300/csrc/tn_online.cu",
                                 "paper_2307_04890_gb300/csrc/tn_internal.cuh"])}

WORKLOADS = {
    "activity": dict(desc="activity-driven n=100000 m=10000000 (power-law activity 2.1, a_min 1e-3, us ticks)",
                     kind="activity", n=100_000, m=10_000_000, seed=2),
    "bursty-scaled": dict(desc="profiling case of the bursty launch: the first 2000000 events of the bursty "
                               "n=500000 stream with node ids folded mod 40000, 503808 source columns (each node "
                               "12.6 times), 64-word slabs: 123 CTAs as in the full launch, a 2.5 GB matrix",
                          kind="scaled", n=40_000, m=2_000_000, seed=3, ncols=123 * 64 * 64, slab=64),
    "uniform-small": dict(desc="uniform pairs n=1000 m=20000, t uniform in [0,1e4)", kind="uniform",
                          n=1000, m=20_000, seed=1, t_range=10_000),
    "er-small": dict(desc="ER G(n, 2/n) with Poisson link activity, n=10000 m=10000000 (the paper's largest "
                          "synthetic n; autotuned: the resident-slab form)", kind="er", n=10_000, m=10_000_000,
                     seed=7),
    "bursty": dict(desc="power-law bursty n=500000 m=100000000 (degree exponent 2.5, Pareto(1.5, 60 s) gaps, "
                        "integer seconds: large tie groups)", kind="bursty", n=500_000, m=100_000_000, seed=3),
    "hashed": dict(desc="hashed estimate n=1000000 m=100000000 activity-driven, k=16384, R=8, 65536 sampled sources",
                   kind="hashed", n=1_000_000, m=100_000_000, seed=4, k=16384, R=8, nsrc=65536),
    "er-sweep": dict(desc="sweep: ER G(n, 2/n) with Poisson link activity, n in {100..10000}, m = 1e4..1e9; "
                          "hashed estimate with n_s = 0.3 n, K = 5 against exact sizes", kind="sweep", n=0, m=0, seed=6),
    "online": dict(desc="online: the activity-driven n=100000 m=10000000 stream pushed in 16 batches cut at seeded "
                        "points, 7 of them inside timestamp groups, plus node growth 100000 -> 102048",
                   kind="online", n=100_000, m=10_000_000, seed=2, batches=16, grow_to=102_048),
    "serving": dict(desc="serving: Poisson arrivals 200 req/s, n log-uniform [1e3,1e5], m log-uniform [1e4,1e7], "
                         "uniform endpoints, 4 incremental batches per job", kind="serving", n=0, m=0, seed=5),
}


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", choices=sorted(WORKLOADS), default="bursty")
    ap.add_argument("--window", type=int, default=0, help="events per scheduling window (0 = library default)")
    ap.add_argument("--slab", type=int, default=0, help="row words per CTA (0 = library default)")
    ap.add_argument("--resident", type=int, default=0,
                    help="resident-slab form with this many row words per CTA (1 or 2; 0 = column slabs)")
    ap.add_argument("--cpu-seconds", type=float, default=12.0, help="target CPU time of the oracle sample")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--autotune", choices=["auto", "on", "off"], default="auto",
                    help="pick plan options with tn_autotune before timing (auto: on for bursty and er-small)")
    ap.add_argument("--tune-sample", type=int, default=2_000_000, help="events the autotuner times")
    ap.add_argument("--sweep-max-m", type=float, default=1e9, help="er-sweep: largest number of events")
    ap.add_argument("--jobs", type=int, default=2000, help="serving: number of jobs")
    ap.add_argument("--distinct-jobs", type=int, default=200, help="serving: distinct event sets the jobs cycle")
    ap.add_argument("--rate", type=float, default=200.0, help="serving: mean arrivals per second")
    ap.add_argument("--batch-gap-ms", type=float, default=20.0, help="serving: time between a job's batches")
    ap.add_argument("--max-active", type=int, default=64, help="serving: jobs resident at once")
    ap.add_argument("--workers", type=int, default=32, help="serving: host worker threads of the server")
    return ap.parse_args()


def make_events(w, rank=0):
    from paper_2307_04890_gb300 import synth
    seed = replica_seed(w, rank)
    if w["kind"] in ("activity", "hashed", "online"):
        return synth.activity_driven(w["n"], w["m"], seed=seed)
    if w["kind"] == "bursty":
        return synth.powerlaw_bursty(w["n"], w["m"], seed=seed)
    if w["kind"] == "er":
        return synth.er_poisson(w["n"], w["m"], seed=seed)
    return synth.uniform_events(w["n"], w["m"], t_range=w["t_range"], seed=seed)


def column_range(n, rank, world):
    """Source columns [c0, c1) of one rank when the exact matrix is split over
    ranks: columns never interact (Section 3.1), so each rank streams every
    event over its own contiguous block of sources."""
    return rank * n // world, (rank + 1) * n // world


def gather_sizes(local, local_argmax, n, rank, world, dist):
    """All-gather of every rank's out-sizes (its columns, in order) into the n
    sizes of the whole matrix, and the largest out-component: each rank's own
    largest (its lowest column among equal sizes, from tn_out_sizes) is
    gathered beside the sizes and the winner is the largest size, lowest
    node id on ties.  `local` is an int32 tensor on the rank's device (gloo:
    CPU, NCCL: CUDA), `local_argmax` an int; returns (sizes, argmax)."""
    import torch
    if world == 1 or dist is None:
        return local, int(local_argmax)
    counts = [column_range(n, r, world)[1] - column_range(n, r, world)[0] for r in range(world)]
    buf = torch.zeros(max(counts) + 2, dtype=local.dtype, device=local.device)
    buf[: local.numel()] = local
    buf[-2] = local[local_argmax]
    buf[-1] = column_range(n, rank, world)[0] + local_argmax
    parts = [torch.empty_like(buf) for _ in range(world)]
    dist.all_gather(parts, buf)
    full = torch.cat([parts[r][: counts[r]] for r in range(world)])
    best = [(int(p[-2]), -int(p[-1])) for p in (q.cpu() for q in parts)]
    size, neg_id = max(best)  # largest size, then the lowest id
    return full, -neg_id


def gather_blocks(local, total, rank, world, dist):
    """All-gather of contiguous per-rank blocks (rank r holds entries
    column_range(total, r, world)) into the whole array, in rank order."""
    import torch
    if world == 1 or dist is None:
        return local
    counts = [column_range(total, r, world)[1] - column_range(total, r, world)[0] for r in range(world)]
    buf = torch.zeros(max(counts), dtype=local.dtype, device=local.device)
    buf[: local.numel()] = local
    parts = [torch.empty_like(buf) for _ in range(world)]
    dist.all_gather(parts, buf)
    return torch.cat([parts[r][: counts[r]] for r in range(world)])


def replica_owner(j, world):
    """Rank that builds hash replica j when the hashed workload is split over
    ranks: the R proxy networks are independent (Section 4.2), dealt round-robin."""
    return j % world


def share_proxies(P, R, world, dist):
    """Every rank receives every proxy matrix from the rank that built it (one
    broadcast per replica): the fusion of Section 4.2 intersects all R replicas
    for every source, so this is the split's one exchange step."""
    if world == 1 or dist is None:
        return
    for j in range(R):
        dist.broadcast(P[j], src=replica_owner(j, world))


def replica_seed(w, rank):
    """Rank r runs an independent replica of the workload (weak scaling), seeded apart."""
    return w["seed"] + 1000 * rank


def job_max_ms(ms, dist, device):
    """The job's time is its slowest rank's: all-reduce MAX over ranks (no-op alone)."""
    if dist is None:
        return ms
    import torch
    tt = torch.tensor([ms], dtype=torch.float64, device=device)
    dist.all_reduce(tt, op=dist.ReduceOp.MAX)
    return float(tt.item())


def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def code_only(text):
    """C++/CUDA source without comments and blank space: what the compiler sees
    of it (an edit to a comment does not change the kernel a profile measured)."""
    import re
    text = re.sub(r"/\*.*?\*/", " ", text, flags=re.S)
    text = re.sub(r"//[^\n]*", " ", text)
    return " ".join(text.split())


def kernel_source_sha(sources):
    h = hashlib.sha256()
    for rel in sources:
        with open(os.path.join(ROOT, rel), encoding="utf-8") as f:
            h.update(code_only(f.read()).encode())
    return h.hexdigest()[:16]


def profiled_traffic(workload_key, slab_words=None):
    """DRAM bytes per launch of the workload's dominant kernel from the committed
    ncu summary, if it was taken on the current kernel sources, this workload
    and (when the summary names one) the same slab width."""
    try:
        fields = {}
        name, sources = PROFILE_SUMMARIES[workload_key]
        with open(os.path.join(ROOT, "profiles", name)) as f:
            for line in f:
                if ":" in line and not line.startswith("#"):
                    k, v = line.split(":", 1)
                    fields[k.strip()] = v.strip()
        if fields.get("kernel_source_sha256_16") != kernel_source_sha(sources):
            return None
        if fields.get("workload") != workload_key:
            return None
        if slab_words is not None and "slab_words" in fields and int(fields["slab_words"]) != int(slab_words):
            return None
        return float(fields["dram_bytes_per_launch"])
    except Exception:
        return None


class ClockSampler:
    """nvidia-smi clock / throttle-reason samples during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.proc = None
        import tempfile
        self.path = os.path.join(tempfile.gettempdir(), f"tn_bench_clocks_{os.getpid()}.csv")
        self.gpu = gpu_index

    def __enter__(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-i", str(self.gpu), "-lms", "200"], stdout=self.f,
                                         stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *exc):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
            self.f.close()

    def summary(self):
        if not self.proc:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        with open(self.path) as f:
            for line in f:
                parts = [p.strip() for p in line.split(",")]
                if len(parts) < 9:
                    continue
                try:
                    sm.append(float(parts[1]))
                    mx.append(float(parts[2]))
                except ValueError:
                    continue
                for name, val in zip(names, parts[5:9]):
                    if val.lower().startswith("active"):
                        reasons.add(name)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def cpu_model():
    """The host CPU's model name (lscpu, else /proc/cpuinfo, else the machine)."""
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.strip().lower().startswith("model name"):
                return line.split(":", 1)[1].strip()
    except Exception:
        pass
    try:
        with open("/proc/cpuinfo") as f:
            for line in f:
                if line.lower().startswith("model name"):
                    return line.split(":", 1)[1].strip()
    except Exception:
        pass
    import platform
    return platform.processor() or platform.machine()


def group_prefix(t, ms):
    """Events [0, ms) extended to the end of the timestamp group of event ms - 1."""
    if ms >= len(t):
        return len(t)
    return int(np.searchsorted(t, t[ms - 1], side="right"))


def cpu_oracle_columns(u, v, t, n, target_s, seed, threads=None):
    """The unchanged oracle on disjoint seeded subsets of source columns, one
    subset per host thread (columns of the component matrix are independent,
    and the oracle's C routine runs without the GIL).  All events are streamed
    when one 64-column slab per thread fits the time budget, else a prefix that
    ends at a timestamp-group boundary.  Returns (columns, events, wall seconds,
    threads); the n-column run on the same threads would take wall * n / columns."""
    import oracle
    from concurrent.futures import ThreadPoolExecutor
    oracle.build_oracle()
    threads = max(1, threads or os.cpu_count() or 1)
    m = len(u)
    rng = np.random.default_rng(seed)
    probe = group_prefix(t, min(m, 1_000_000))
    cols0 = np.sort(rng.choice(n, min(n, 64), replace=False)).astype(np.uint32)
    t0 = time.perf_counter()
    oracle.component_matrix(u[:probe], v[:probe], t[:probe], n, src=cols0)
    per_event = (time.perf_counter() - t0) / max(probe, 1)
    if per_event * m <= target_s:
        ms, words = m, max(1, int(target_s / max(per_event * m, 1e-9)))
    else:
        ms, words = group_prefix(t, max(probe, int(target_s / max(per_event, 1e-12)))), 1
    cols_per = max(1, min(64 * words, n // threads))
    total = min(n, cols_per * threads)
    perm = rng.permutation(n)[:total].astype(np.uint32)
    chunks = [np.sort(perm[i:i + cols_per]) for i in range(0, total, cols_per)]
    uu, vv, tt = u[:ms], v[:ms], t[:ms]
    t0 = time.perf_counter()
    with ThreadPoolExecutor(len(chunks)) as ex:
        list(ex.map(lambda c: oracle.component_matrix(uu, vv, tt, n, src=c), chunks))
    wall = time.perf_counter() - t0
    return total, ms, wall, len(chunks)


def cpu_baseline_line(u, v, t, n, target_s, seed):
    cols, ms, wall, threads = cpu_oracle_columns(u, v, t, n, target_s, seed)
    value = cols * ms / wall
    sample = (f"{'all' if ms == len(u) else 'first'} {ms} of {len(u)} events over {cols} seeded source columns "
              f"({threads} threads, one column slab each), {wall:.1f} s wall; extrapolated linearly to all "
              f"{n} columns")
    return {"value": value, "unit": "bit-updates/s", "cores": threads, "kind": "oracle", "sample": sample,
            "extrapolated": cols < n, "nproc": os.cpu_count(), "cpu_model": cpu_model()}


def run_reference_serving(args, w, world):
    """The oracle on whole jobs of the serving stream, in arrival order, until
    about --cpu-seconds of CPU time: events/s of the sample."""
    import oracle
    from concurrent.futures import ThreadPoolExecutor
    from paper_2307_04890_gb300 import synth
    oracle.build_oracle()
    specs = synth.serving_jobs(args.jobs, rate=args.rate, seed=w["seed"])
    threads = os.cpu_count() or 1
    # whole jobs of the stream in arrival order (n * m <= 2e11 each), one job per host
    # thread at a time, until about --cpu-seconds of wall time
    picked = [sp for sp in specs if sp["n"] * sp["m"] <= 2e11]
    done_events, jobs_done = 0, 0
    t0 = time.perf_counter()

    def one(spec):
        u, v, t = synth.job_events(spec)
        s0 = time.perf_counter()
        oracle.column_counts(oracle.component_matrix(u, v, t, spec["n"]), spec["n"])
        return len(u), time.perf_counter() - s0

    spent = 0.0
    with ThreadPoolExecutor(threads) as ex:
        for i in range(0, len(picked), threads):
            if time.perf_counter() - t0 >= args.cpu_seconds:
                break
            s0 = time.perf_counter()
            for m_, _ in ex.map(one, picked[i:i + threads]):
                done_events += m_
                jobs_done += 1
            spent += time.perf_counter() - s0
    value = done_events / max(spent, 1e-9)
    sample = (f"{jobs_done} whole jobs of the stream (n*m <= 2e11), {threads} threads, one job each at a time, "
              f"{spent:.1f} s wall (event generation included)")
    line = {"impl": "reference", "metric": METRIC + " (serving)", "value": value, "unit": "events/s",
            "n_gpus": world, "steps": jobs_done, "warmup": 0, "ms_per_step": spent * 1e3 / max(jobs_done, 1),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u64", "data": "synthetic",
            "config": {"workload": w["desc"], "jobs": jobs_done},
            "cpu_baseline": {"value": value, "unit": "events/s", "cores": threads, "kind": "oracle", "sample": sample,
                             "nproc": os.cpu_count(), "cpu_model": cpu_model()},
            "e2e": {"value": value, "unit": "events/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def run_reference_hashed(args, w, world):
    """The oracle's hashing path on a prefix of the events: hash tables, super-
    events and the R proxy component matrices (events/s of the prefix)."""
    import oracle
    oracle.build_oracle()
    u, v, t = make_events(w)
    n, k, R = w["n"], w["k"], w["R"]
    t0 = time.perf_counter()
    H = oracle.hash_nodes(0, R, k, n)
    hash_s = time.perf_counter() - t0
    from concurrent.futures import ThreadPoolExecutor
    threads = min(R, os.cpu_count() or 1)  # one proxy network per host thread (they are independent)

    def proxies(ms_):
        with ThreadPoolExecutor(threads) as ex:
            list(ex.map(lambda j: oracle.proxy_matrices(u[:ms_], v[:ms_], t[:ms_], H[j:j + 1], k), range(R)))

    probe = group_prefix(t, 200_000)
    t0 = time.perf_counter()
    proxies(probe)
    per_event = (time.perf_counter() - t0) / probe
    ms = group_prefix(t, int(min(len(u), max(probe, args.cpu_seconds / max(per_event, 1e-12)))))
    t0 = time.perf_counter()
    proxies(ms)
    spent = time.perf_counter() - t0
    value = ms / spent
    sample = (f"hash tables ({hash_s:.1f} s, untimed) then the {R} proxy matrices over the first {ms} events, "
              f"{threads} threads (one proxy network each)")
    line = {"impl": "reference", "metric": METRIC + " (hashed estimate)", "value": value, "unit": "events/s",
            "n_gpus": world, "steps": 1, "warmup": 0, "ms_per_step": spent * 1e3, "higher_is_better": True,
            "scaling": "strong", "vs_baseline": None, "dtype": "u64", "data": "synthetic",
            "config": {"workload": w["desc"], "n": n, "m": w["m"], "k": k, "R": R},
            "cpu_baseline": {"value": value, "unit": "events/s", "cores": threads, "kind": "oracle", "sample": sample,
                             "nproc": os.cpu_count(), "cpu_model": cpu_model()},
            "e2e": {"value": value, "unit": "events/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def run_reference(args, w, rank, world):
    if rank != 0:
        return
    if w["kind"] == "serving":
        run_reference_serving(args, w, world)
        return
    if w["kind"] == "hashed":
        run_reference_hashed(args, w, world)
        return
    u, v, t = make_events(w)
    n = w["n"]
    rates, walls = [], []
    per_step = max(1.0, args.cpu_seconds / max(1, args.steps + args.warmup) * 2)
    for i in range(args.warmup + args.steps):
        cols, ms, wall, threads = cpu_oracle_columns(u, v, t, n, per_step, seed=w["seed"] + i)
        if i >= args.warmup:
            rates.append(cols * ms / wall)  # bit-updates/s, extrapolated to all columns
            walls.append(wall)
    value = statistics.mean(rates)
    mean = statistics.mean(walls)
    metric, unit = METRIC, "bit-updates/s"
    if w["kind"] == "online":  # the online arm reports events/s (of the extrapolated n-column run)
        value, metric, unit = value / n, ONLINE_METRIC, "events/s"
    sample = (f"per step: {'all' if ms == len(u) else 'first'} {ms} of {w['m']} events over {cols} seeded source "
              f"columns ({threads} threads, one column slab each); extrapolated linearly to all {n} columns")
    line = {"impl": "reference", "metric": metric, "value": value, "unit": unit, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": mean * 1e3, "higher_is_better": True,
            "scaling": "weak" if w["kind"] == "online" else "strong", "vs_baseline": None, "dtype": "u64",
            "data": "synthetic", "config": {"workload": w["desc"], "n": n, "m": w["m"]},
            "events_per_s": statistics.mean(rates) / n,
            "cpu_baseline": {"value": value, "unit": unit, "cores": threads, "kind": "oracle", "sample": sample,
                             "extrapolated": cols < n, "nproc": os.cpu_count(), "cpu_model": cpu_model()},
            "e2e": {"value": value, "unit": unit, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def run_scaled(args, w, rank, world, local_rank):
    """The bursty launch at a size an ncu --set full capture can replay: the
    same 123 CTAs of 64-word slabs and global-memory windows, on a 2.5 GB
    matrix (node ids folded, source ids repeated).  One step = init + stream."""
    import torch
    import paper_2307_04890_gb300 as tn
    from paper_2307_04890_gb300 import synth
    from paper_2307_04890_gb300.build import build_library

    build_library()
    tn.load_library()
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    n, m, ncols = w["n"], w["m"], w["ncols"]
    u, v, t = synth.powerlaw_bursty(500_000, 100_000_000, seed=w["seed"])
    u, v, t = (u[:m] % n).astype(np.uint32), (v[:m] % n).astype(np.uint32), t[:m]
    du = torch.from_numpy(u.view(np.int32)).to(dev)
    dv = torch.from_numpy(v.view(np.int32)).to(dev)
    dt = torch.from_numpy(t).to(dev)
    src = torch.from_numpy((np.arange(ncols) % n).astype(np.int32)).to(dev)
    plan = tn.Plan(du, dv, dt, n, slab_words=w["slab"])
    S = torch.empty((n, tn.tn_row_words(ncols)), dtype=torch.int64, device=dev)
    ev = lambda: torch.cuda.Event(enable_timing=True)
    for _ in range(args.warmup):
        plan.apply(S, ncols=ncols, src=src, init=True)
    times = []
    for _ in range(args.steps):
        e0, e1 = ev(), ev()
        e0.record()
        plan.apply(S, ncols=ncols, src=src, init=True)
        e1.record()
        torch.cuda.synchronize()
        times.append(e0.elapsed_time(e1))
    assert plan.status() == 0
    ms = statistics.mean(times)
    alg = 8 * plan.stats()["ops"] + n * tn.tn_row_words(ncols) * 8  # schedule in, matrix out
    traffic = profiled_traffic("bursty-scaled", w["slab"])  # DRAM bytes of the launch (ncu)
    peak, _ = measured_peaks()
    if rank == 0:
        print(json.dumps({"metric": "bit-updates/s of the scaled bursty launch (profiling case)",
                          "value": ncols * m / (ms * 1e-3), "unit": "bit-updates/s", "n_gpus": 1,
                          "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
                          "scaling": "weak", "vs_baseline": None, "dtype": "u64", "data": "synthetic",
                          "config": {"workload": w["desc"], "plan": plan.stats()},
                          "roofline": {"bound": "hbm", "achieved": (traffic or alg) / (ms * 1e-3) / 1e9, "peak": peak,
                                       "unit": "GB/s", "frac": (traffic or alg) / (ms * 1e-3) / 1e9 / peak,
                                       "traffic": traffic, "algorithmic_bytes_per_launch": alg}}), flush=True)


def run_serving(args, w, rank, world, local_rank):
    """Continuous admission of a Poisson stream of jobs through tn_server_*.
    Job j opens at its arrival time and its 4 batches (split at timestamp
    quartiles) are pushed at arrival + b * batch gap, so later batches reach a
    job whose matrix is already on the device.  Latency = open -> out-sizes
    on the host (and last push -> results); throughput = all events (and
    n * m bit-updates) of all jobs / wall time from the first open to the last
    result.  The jobs cycle through --distinct-jobs event sets (host memory).
    Beside it: the same distinct jobs one after another through the plain
    one-shot path (tn_out_component_sizes_host), identical results required."""
    import torch
    import paper_2307_04890_gb300 as tn
    from paper_2307_04890_gb300 import synth
    from paper_2307_04890_gb300.build import build_library

    build_library()
    tn.load_library()
    torch.cuda.set_device(local_rank)
    specs = synth.serving_jobs(args.jobs, rate=args.rate, seed=w["seed"] + 1000 * rank)
    distinct = min(args.distinct_jobs, len(specs))
    pinned = []  # the events wait in pinned host memory, as a serving front end would hold them

    def pin(a, view):
        p_ = torch.from_numpy(a.view(view)).pin_memory()
        pinned.append(p_)
        return p_.numpy().view(a.dtype)

    events = []
    for spec in specs[:distinct]:
        u, v, t = synth.job_events(spec)
        bounds = synth.split_batches(t, 4)
        events.append((spec["n"], pin(u, np.int32), pin(v, np.int32), pin(t, np.int64), bounds))
    jobs = [(spec, events[i % distinct]) for i, spec in enumerate(specs)]
    gap = args.batch_gap_ms * 1e-3

    def serve(job_list, rate_scale=1.0):
        srv = tn.Server(max_active=args.max_active, workers=args.workers)
        by_id = {spec["job"]: (spec, ev_) for spec, ev_ in job_list}
        actions = []
        for spec, (n, u, v, t, bounds) in job_list:
            for b in range(len(bounds)):
                actions.append((spec["arrival"] * rate_scale + b * gap, spec["job"], b))
        actions.sort()
        recs = []
        t0 = time.perf_counter()
        for when, jid, b in actions:
            delay = t0 + when - time.perf_counter()
            if delay > 0.002:
                recs += srv.poll(wait_ms=0)
                time.sleep(max(0.0, t0 + when - time.perf_counter()))
            spec, (n, u, v, t, bounds) = by_id[jid]
            a, e = bounds[b]
            if b == 0:
                srv.open(jid, n, max(e_ - a_ for a_, e_ in bounds))
            srv.push(jid, u[a:e], v[a:e], t[a:e], last=b + 1 == len(bounds))
        while len(recs) < len(job_list):
            recs += srv.poll(wait_ms=100)
        wall = time.perf_counter() - t0
        st = srv.stats()
        results = dict(srv.results)
        srv.close()
        return recs, wall, st, results

    # warm-up: the first jobs once, unmeasured
    warm = [(dict(s_, job=i, arrival=0.0), e_) for i, (s_, e_) in enumerate(jobs[: max(3, args.warmup)])]
    serve(warm)
    with ClockSampler(torch.cuda.current_device()) as clocks:
        recs, wall, st, results = serve(jobs)
    bad = [r for r in recs if r["status"] != 0]
    ms = lambda a, b: np.array([(r[b] - r[a]) / 1e6 for r in recs])
    lat, res_lat = ms("t_submit_ns", "t_done_ns"), ms("t_last_push_ns", "t_done_ns")
    host_last, gpu_tail = ms("t_last_push_ns", "t_enqueued_ns"), ms("t_enqueued_ns", "t_done_ns")
    by_open = sorted(recs, key=lambda r: r["t_submit_ns"])
    queue = np.array([(r["t_admit_ns"] - r["t_submit_ns"]) / 1e6 for r in by_open])
    q = max(1, len(queue) // 4)
    n_events = sum(len(e[1]) for _, e in jobs)
    bit_updates = sum(e[0] * len(e[1]) for _, e in jobs)
    pct = lambda x: {"p50": float(np.percentile(x, 50)), "p99": float(np.percentile(x, 99)),
                     "mean": float(x.mean()), "max": float(x.max())}

    # the plain single-network path on the distinct jobs, one after another
    plain_events = plain_bits = 0
    identical = True
    t0 = time.perf_counter()
    for i, (n, u, v, t, bounds) in enumerate(events):
        sizes, am = tn.tn_out_component_sizes_host(u, v, t, n)
        plain_events += len(u)
        plain_bits += n * len(u)
        identical = identical and np.array_equal(sizes, results[i][0]) and am == results[i][1]
    plain_wall = time.perf_counter() - t0

    result = {"metric": METRIC + " (serving)", "value": n_events / wall, "unit": "events/s", "n_gpus": world,
              "steps": len(jobs), "warmup": len(warm), "ms_per_step": wall * 1e3 / len(jobs),
              "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u64", "data": "synthetic",
              "config": {"workload": w["desc"], "jobs": len(jobs), "distinct_event_sets": distinct,
                         "host_events": "pinned",
                         "rate_per_s": args.rate, "batch_gap_ms": args.batch_gap_ms,
                         "max_active": args.max_active, "workers": args.workers,
                         "cuda_device_max_connections": os.environ.get("CUDA_DEVICE_MAX_CONNECTIONS"),
                         "l2": "per-job matrices up to 1.25 GB; jobs overlap"},
              "bit_updates_per_s": bit_updates / wall,
              "offered_events_per_s": n_events / max(specs[-1]["arrival"], 1e-9),
              "latency_ms": pct(lat), "result_latency_ms": pct(res_lat),
              "breakdown_ms": {"last_push_to_enqueued": pct(host_last), "enqueued_to_results": pct(gpu_tail)},
              "queue_delay_ms": {"first_quarter_median": float(np.median(queue[:q])),
                                 "last_quarter_median": float(np.median(queue[-q:]))},
              "plain_one_after_another": {"jobs": len(events), "events_per_s": plain_events / plain_wall,
                                          "bit_updates_per_s": plain_bits / plain_wall,
                                          "identical_results": bool(identical)},
              "server": st,
              "host_ms": {"admit_per_job": st["admit_ns"] / 1e6 / max(st["admitted"], 1),
                          "copy_in_per_batch": st["copy_ns"] / 1e6 / max(st["batches"], 1),
                          "schedule_per_batch": st["schedule_ns"] / 1e6 / max(st["batches"], 1),
                          "results_per_job": st["result_ns"] / 1e6 / max(st["completed"], 1),
                          "retire_per_job": st["retire_ns"] / 1e6 / max(st["completed"], 1),
                          "worker_busy_fraction": (st["admit_ns"] + st["copy_ns"] + st["schedule_ns"] +
                                                   st["result_ns"] + st["retire_ns"]) / 1e9 /
                                                  (wall * args.workers)},
              "failed_jobs": len(bad), "clocks": clocks.summary(),
              "e2e": {"value": n_events / wall, "unit": "events/s",
                      "h2d_bytes_per_step": n_events * 16 / len(jobs),
                      "d2h_bytes_per_step": sum(e[0] * 4 + 4 for _, e in jobs) / len(jobs)}}
    if rank == 0:
        print(json.dumps(result), flush=True)


def run_hashed(args, w, rank, world, local_rank):
    """Network hashing end to end (Section 4): hash tables and super-events, the
    R proxy schedules and the schedule of the sampled exact columns, the R
    proxy matrices and the exact sampled columns in ONE persistent launch
    (a job list over slab widths chosen so that the launch is one wave), the fused
    estimate for the sampled sources, their exact out-sizes and the error
    against them.  Beside the step: the same work in separate launches, the
    proxies replayed as a CUDA graph against one launch per proxy (identical
    matrices throughout), and the error on an unsaturated prefix of the stream
    (every node of the full stream reaches every node, so the error there is 0)."""
    import torch
    import paper_2307_04890_gb300 as tn
    from paper_2307_04890_gb300.build import build_library

    build_library()
    tn.load_library()
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    n, m, k, R, nsrc = w["n"], w["m"], w["k"], w["R"], w["nsrc"]
    # one job over all ranks: the same events and sampled sources everywhere;
    # rank r builds the replicas it owns and the exact columns of its share of
    # the sources, receives the other replicas' matrices, and fuses its share
    u, v, t = make_events(w)
    rng = np.random.default_rng(w["seed"])
    src_np = np.sort(rng.choice(n, nsrc, replace=False)).astype(np.uint32)
    mine = [j for j in range(R) if replica_owner(j, world) == rank]
    s0, s1 = column_range(nsrc, rank, world)
    ns = s1 - s0
    du = torch.from_numpy(u.view(np.int32)).to(dev)
    dv = torch.from_numpy(v.view(np.int32)).to(dev)
    dt = torch.from_numpy(t).to(dev)
    src_all = torch.from_numpy(src_np.view(np.int32)).to(dev)
    src = src_all[s0:s1]
    P = torch.empty((R, k, tn.tn_row_words(k)), dtype=torch.int64, device=dev)
    Sx = torch.empty((n, tn.tn_row_words(ns)), dtype=torch.int64, device=dev)
    stream = torch.cuda.current_stream(dev)
    seed = 0  # replica j hashes with splitmix64(seed ^ j): seeds 0..R-1
    ev = lambda: torch.cuda.Event(enable_timing=True)
    # no options: slab widths are chosen for the whole launch, and rows are tracked
    popts, xopts = {}, {}
    timing = {"combined_ms": [], "estimate_ms": []}

    def step(record):
        H, pu, pv = tn.tn_hash_proxy(du, dv, n, k, R, seed)                              # a5
        plans = [tn.Plan(pu[j].contiguous(), pv[j].contiguous(), dt, k, **popts) for j in mine]  # a1 (proxies)
        plan_x = tn.Plan(du, dv, dt, n, **xopts)                                          # a1 (exact sample)
        e = [ev() for _ in range(3)]
        e[0].record(stream)
        tn.tn_plan_apply_batch(plans + [plan_x], [P[j] for j in mine] + [Sx],             # a2 + a3 + a6, and
                               ncols=[k] * len(mine) + [ns], init=True,                   # a8's exact columns
                               srcs=[None] * len(mine) + [src])
        e[1].record(stream)
        share_proxies(P, R, world, dist)                                                  # (N > 1)
        est = tn.tn_hash_estimate(P, R, k, H, n, src=src)                                 # a7
        e[2].record(stream)
        exact, _, _ = tn.tn_out_sizes(Sx, n, ns)
        est = gather_blocks(est, nsrc, rank, world, dist)                                 # (N > 1)
        exact = gather_blocks(exact, nsrc, rank, world, dist)
        err = tn.tn_error_stats(est, exact, n)                                            # a8 (synchronises)
        if record:
            timing["combined_ms"].append(e[0].elapsed_time(e[1]))
            timing["estimate_ms"].append(e[1].elapsed_time(e[2]))
        for p in plans:
            p.destroy()
        plan_x.destroy()
        return err, H, pu, pv

    for _ in range(args.warmup):
        step(False)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    launches0 = tn.tn_kernel_launches()
    start, end = ev(), ev()
    with ClockSampler(torch.cuda.current_device()) as clocks:
        torch.cuda.synchronize()
        start.record(stream)
        for _ in range(args.steps):
            err, H, pu, pv = step(True)
        end.record(stream)
        torch.cuda.synchronize()
    launches = tn.tn_kernel_launches() - launches0
    ms_total = job_max_ms(start.elapsed_time(end), dist, dev)
    ms_step = ms_total / args.steps

    # beside the step, on one GPU: the same work in separate launches, the graph
    # replay against single launches, and the error on unsaturated prefixes
    proxies_alone_ms = exact_alone_ms = graph_ms = single_ms = None
    separate_identical = identical = None
    sopts = {}
    keys = ("mean_abs", "max_abs", "mean_rel", "max_rel", "w1")
    prefixes = []
    if world == 1:
        # the same work in separate launches (each with the widths chosen for it alone),
        # and the proxies as a graph vs one launch each
        P_ref, Sx_ref = P.clone(), Sx.clone()
        plans = [tn.Plan(pu[j].contiguous(), pv[j].contiguous(), dt, k, **sopts) for j in range(R)]
        plan_x = tn.Plan(du, dv, dt, n, **xopts)
        e0, e1, e2 = ev(), ev(), ev()
        e0.record(stream)
        tn.tn_plan_apply_batch(plans, [P[j] for j in range(R)], init=True)
        e1.record(stream)
        plan_x.apply(Sx, ncols=nsrc, src=src, init=True)
        e2.record(stream)
        torch.cuda.synchronize()
        proxies_alone_ms, exact_alone_ms = e0.elapsed_time(e1), e1.elapsed_time(e2)
        separate_identical = bool(torch.equal(P, P_ref) and torch.equal(Sx, Sx_ref))
        g = tn.BatchGraph(plans, [P[j] for j in range(R)])
        g.launch()
        torch.cuda.synchronize()
        e0.record(stream)
        g.launch()
        e1.record(stream)
        torch.cuda.synchronize()
        graph_ms = e0.elapsed_time(e1)
        P2 = torch.empty_like(P)
        e0.record(stream)
        for j in range(R):
            plans[j].apply(P2[j], init=True)
        e1.record(stream)
        torch.cuda.synchronize()
        single_ms = e0.elapsed_time(e1)
        identical = bool(torch.equal(P, P_ref) and torch.equal(P2, P_ref))
        g.destroy()
        for p in plans:
            p.destroy()
        plan_x.destroy()
        del P2, P_ref, Sx_ref

        # error on unsaturated prefixes of the stream (to a group boundary)
        for want in (10_000, 100_000, 1_000_000):
            mp = group_prefix(t, want)
            Hp, pup, pvp = tn.tn_hash_proxy(du[:mp], dv[:mp], n, k, R, seed)
            plans_p = [tn.Plan(pup[j].contiguous(), pvp[j].contiguous(), dt[:mp], k, **popts) for j in range(R)]
            plan_xp = tn.Plan(du[:mp], dv[:mp], dt[:mp], n, **xopts)
            tn.tn_plan_apply_batch(plans_p + [plan_xp], [P[j] for j in range(R)] + [Sx], ncols=[k] * R + [nsrc],
                                   init=True, srcs=[None] * R + [src])
            est_p = tn.tn_hash_estimate(P, R, k, Hp, n, src=src)
            exact_p, _, _ = tn.tn_out_sizes(Sx, n, nsrc)
            err_p = tn.tn_error_stats(est_p, exact_p, n)
            prefixes.append(dict({key: err_p[key] for key in keys}, events=mp,
                                 mean_exact=float(exact_p.float().mean().item()),
                                 mean_estimate=float(est_p.float().mean().item())))
            for p in plans_p + [plan_xp]:
                p.destroy()

    combined_ms = statistics.mean(timing["combined_ms"])
    wx = tn.tn_row_words(nsrc)
    # this rank's launch: its replicas and its share of the sampled columns
    # what the launch cannot do without: every schedule in (8 bytes per op, about an
    # op per event) and every matrix out once (updates that change nothing move no row)
    alg_exact = 8 * m + n * tn.tn_row_words(ns) * 8
    alg_proxy = len(mine) * (8 * m + k * tn.tn_row_words(k) * 8)
    peak, peak_kind = measured_peaks()
    bit_updates = (R * k + nsrc) * m  # the whole job
    result = {"metric": METRIC + " (hashed estimate)", "value": m / (ms_step * 1e-3), "unit": "events/s",
              "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_step,
              "higher_is_better": True, "scaling": "strong", "vs_baseline": None, "dtype": "u64",
              "data": "synthetic",
              "config": {"workload": w["desc"], "n": n, "m": m, "k": k, "R": R, "sampled_sources": nsrc,
                         "plan_options": {"proxies": popts, "exact_sampled": xopts},
                         "parallelism": (f"{world} GPUs: replicas dealt round-robin and broadcast to every rank, "
                                         "sampled sources split, estimates and sizes all-gathered")
                                        if world > 1 else "single GPU",
                         "l2": "inputs larger than L2 (events 1.6 GB, sampled matrix %.1f GB)" % (n * wx * 8 / 1e9)},
              "bit_updates_per_s": bit_updates / (ms_step * 1e-3),
              "kernels_ms": {"proxies_and_exact_columns_one_launch": combined_ms,
                             "estimate": statistics.mean(timing["estimate_ms"]),
                             "proxies_alone": proxies_alone_ms, "exact_columns_alone": exact_alone_ms},
              "roofline": {"bound": "hbm", "kernel": "stream_kernel (%d proxies + %d exact columns, one launch)"
                                                     % (len(mine), ns),
                           "achieved": (alg_exact + alg_proxy) / (combined_ms * 1e-3) / 1e9, "peak": peak,
                           "peak_source": f"{peak_kind} MEASURED_PEAKS hbm_gbs", "unit": "GB/s",
                           "frac": (alg_exact + alg_proxy) / (combined_ms * 1e-3) / 1e9 / peak, "traffic": None,
                           "achieved_is": "schedules in once + matrices out once / kernel time",
                           "algorithmic_bytes_per_launch": alg_exact + alg_proxy,
                           "note": "the proxies' 32 MB matrices are served largely from L2"},
              "error": {key: err[key] for key in keys},
              "error_prefixes": prefixes,
              "combined_vs_separate": {"combined_ms": combined_ms,
                                       "separate_ms": proxies_alone_ms + exact_alone_ms,
                                       "separate_shapes": {"proxies": sopts, "exact_sampled": xopts},
                                       "identical": separate_identical},
              "batched_vs_single": {"graph_replay_ms": graph_ms, "single_launches_ms": single_ms,
                                    "identical": identical},
              "gpu_launches": launches, "clocks": clocks.summary()}
    if rank == 0:
        print(json.dumps(result), flush=True)
    if dist:
        dist.destroy_process_group()


def run_online(args, w, rank, world, local_rank):
    """The online state (tn_online_*): one step pushes the whole stream in
    batches cut at arbitrary points, flushes and takes the out-sizes.  Beside
    it: the same step with every batch copied from pinned host memory (e2e),
    and the one-shot step over the same events (schedule + init + apply +
    sizes), which must give the same matrix.  Node growth is timed on its own:
    the reallocating growth of the final matrix to more nodes (an HBM copy)."""
    import torch
    import paper_2307_04890_gb300 as tn
    from paper_2307_04890_gb300.build import build_library

    build_library()
    tn.load_library()
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)
    n, m, B = w["n"], w["m"], w["batches"]
    u, v, t = make_events(w, rank)
    du = torch.from_numpy(u.view(np.int32)).to(dev)
    dv = torch.from_numpy(v.view(np.int32)).to(dev)
    dt = torch.from_numpy(t).to(dev)
    hu = torch.from_numpy(u.view(np.int32)).pin_memory()
    hv = torch.from_numpy(v.view(np.int32)).pin_memory()
    ht = torch.from_numpy(t).pin_memory()
    rng = np.random.default_rng(replica_seed(w, rank))
    # half of the cuts inside timestamp groups (between two events of equal t), half anywhere
    inside = np.flatnonzero(t[1:] == t[:-1]) + 1
    picks = rng.choice(inside, min(len(inside), (B - 1) // 2), replace=False) if len(inside) else np.array([], int)
    rest = rng.choice(np.setdiff1d(np.arange(1, m), picks), B - 1 - len(picks), replace=False)
    cuts = np.r_[0, np.sort(np.r_[picks, rest]), m].astype(np.int64)
    split = int(sum(1 for c in cuts[1:-1] if t[c - 1] == t[c]))
    stream = torch.cuda.current_stream(dev)
    ev = lambda: torch.cuda.Event(enable_timing=True)

    def online_step():
        on = tn.Online(n)
        for a, b in zip(cuts[:-1], cuts[1:]):
            on.push(du[a:b], dv[a:b], dt[a:b])
        on.flush()
        out, _, am = tn.tn_out_sizes(on.matrix(), n, n, argmax=True)
        return on, out, am

    def online_e2e_step():
        on = tn.Online(n)
        for a, b in zip(cuts[:-1], cuts[1:]):
            on.push(hu[a:b].to(dev, non_blocking=True), hv[a:b].to(dev, non_blocking=True),
                    ht[a:b].to(dev, non_blocking=True))
        on.flush()
        out, _, am = tn.tn_out_sizes(on.matrix(), n, n, argmax=True)
        return on, out.cpu(), am.cpu()

    def one_shot_step():
        plan = tn.Plan(du, dv, dt, n)
        S = plan.apply(None, init=True)
        out, _, am = tn.tn_out_sizes(S, n, n, argmax=True)
        plan.destroy()
        return S, out, am

    def release(r):
        if isinstance(r[0], tn.Online):
            r[0].close()

    def timed(fn):
        for _ in range(args.warmup):
            r = fn()
            torch.cuda.synchronize()
            release(r)
        if dist:
            dist.barrier()
        e0, e1 = ev(), ev()
        torch.cuda.synchronize()
        e0.record(stream)
        for i in range(args.steps):
            r = fn()
            if i < args.steps - 1:
                release(r)
        e1.record(stream)
        torch.cuda.synchronize()
        return job_max_ms(e0.elapsed_time(e1), dist, dev) / args.steps, r

    launches0 = tn.tn_kernel_launches()
    with ClockSampler(torch.cuda.current_device()) as clocks:
        online_ms, (on, out_on, am_on) = timed(online_step)
    launches = (tn.tn_kernel_launches() - launches0) // args.steps
    e2e_ms, (on_e2e, out_e2e, _) = timed(online_e2e_step)
    e2e_ok = bool(torch.equal(out_e2e, out_on.cpu()))
    on_e2e.close()
    shot_ms, (S_ref, out_ref, am_ref) = timed(one_shot_step)
    identical = bool(torch.equal(on.matrix(), S_ref) and torch.equal(out_on, out_ref) and
                     int(am_on.item()) == int(am_ref.item()))
    del S_ref
    # node growth into a new buffer (the row stride grows), timed alone
    n2 = w["grow_to"]
    S0 = on.matrix()
    G = torch.empty((n2, tn.tn_row_words(n2)), dtype=torch.int64, device=dev)
    for _ in range(3):
        tn.tn_grow_matrix(S0, n, n2, out=G)
    reps = 10
    e0, e1 = ev(), ev()
    torch.cuda.synchronize()
    e0.record(stream)
    for _ in range(reps):
        tn.tn_grow_matrix(S0, n, n2, out=G)
    e1.record(stream)
    torch.cuda.synchronize()
    grow_ms = e0.elapsed_time(e1) / reps
    grow_bytes = n * tn.tn_row_words(n) * 8 + n2 * tn.tn_row_words(n2) * 8
    grown_ok = bool(torch.equal(G[:n, : tn.tn_row_words(n)], S0) and
                    int(tn.tn_out_sizes(G, n2, n2)[0][n:].sum().item()) == n2 - n)
    on.close()
    peak, peak_kind = measured_peaks()
    result = {"metric": ONLINE_METRIC, "value": world * m / (online_ms * 1e-3), "unit": "events/s",
              "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "ms_per_step": online_ms,
              "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "u64", "data": "synthetic",
              "config": {"workload": w["desc"], "n": n, "m": m, "batches": B, "cuts_inside_a_group": split,
                         "parallelism": f"replicas x{world}" if world > 1 else "single GPU",
                         "l2": "inputs larger than L2 (S 1.25 GB, events 160 MB)"},
              "e2e": {"value": world * m / (e2e_ms * 1e-3), "unit": "events/s", "h2d_bytes_per_step": m * 16,
                      "d2h_bytes_per_step": n * 4 + 4, "ms_per_step": e2e_ms, "identical": e2e_ok},
              "one_shot_ms": shot_ms, "online_over_one_shot": online_ms / shot_ms,
              "identical_to_one_shot": identical,
              "roofline": {"bound": "hbm", "kernel": "grow_kernel (growth %d -> %d nodes into a new buffer)" % (n, n2),
                           "achieved": grow_bytes / (grow_ms * 1e-3) / 1e9, "peak": peak,
                           "peak_source": f"{peak_kind} MEASURED_PEAKS hbm_gbs", "unit": "GB/s",
                           "frac": grow_bytes / (grow_ms * 1e-3) / 1e9 / peak,
                           "traffic": profiled_traffic("online"),
                           "algorithmic_bytes_per_launch": grow_bytes, "kernel_ms": grow_ms, "correct": grown_ok},
              "gpu_launches": launches, "clocks": clocks.summary()}
    if rank == 0:
        print(json.dumps(result), flush=True)
    if dist:
        dist.destroy_process_group()


def run_sweep(args, w, rank, world, local_rank):
    """The synthetic experiments of Sections 3.5 and 4.4: ER G(n, 2/n) with an
    independent Poisson process per link, n in {100 .. 10^4}, m = 10^4 .. 10^9.
    For every (n, m): exact out-sizes (component matrix) and hashed estimates
    (n_s = 0.3 n super-nodes, K = 5 replicas, all n sources), their
    Earth-Mover (W1) distance on raw sizes and on sizes divided by n, the
    relative error, the GPU time of each (schedule + apply + sizes / hash +
    proxies + fusion; events already on the device) and the memory of the
    matrices.  Event counts above 10^8 are generated and applied in chunks of
    10^8 that end at timestamp-group boundaries: each chunk continues the same
    matrices (the method is one pass over the stream, Section 3.5)."""
    import torch
    import paper_2307_04890_gb300 as tn
    from paper_2307_04890_gb300 import synth
    from paper_2307_04890_gb300.build import build_library

    build_library()
    tn.load_library()
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    K = 5
    chunk = 100_000_000
    ev = lambda: torch.cuda.Event(enable_timing=True)
    points = []
    mmax = int(args.sweep_max_m)
    keys = ("window_events", "slab_words", "smem_rows", "wave_ctas", "resident_words")
    tuned = {}
    for n in (100, 200, 500, 1000, 2000, 5000, 10000):
        # launch shapes from the autotuner, once per n, on the first 2e6 events of the
        # same kind of network (exact matrix; the K proxies of n_s = 0.3 n nodes)
        k = max(1, int(0.3 * n))
        us, vs, ts = synth.er_poisson(n, 2_000_000, seed=w["seed"] + 1000 * rank + n)
        dus, dvs = (torch.from_numpy(a.view(np.int32)).to(dev) for a in (us, vs))
        dts = torch.from_numpy(ts).to(dev)
        ex = tn.tn_autotune(dus, dvs, dts, n, sample_events=2_000_000)
        _, pus, pvs = tn.tn_hash_proxy(dus, dvs, n, k, K, w["seed"])
        px = tn.tn_autotune(pus[0].contiguous(), pvs[0].contiguous(), dts, k, replicas=K, sample_events=2_000_000)
        tuned[n] = tuple({key: r[key] if r["best_ms"] <= 1.05 * r["open_ms"] else 0 for key in keys} for r in (ex, px))
        del dus, dvs, dts, pus, pvs
        m = 10_000
        while m <= mmax:
            seed = w["seed"] + 1000 * rank + n
            chunks = [synth.er_poisson(n, m, seed=seed)] if m <= chunk else \
                synth.er_poisson_stream(n, m, chunk=chunk, seed=seed)
            k = max(1, int(0.3 * n))
            S = torch.empty((n, tn.tn_row_words(n)), dtype=torch.int64, device=dev)
            P = torch.empty((K, k, tn.tn_row_words(k)), dtype=torch.int64, device=dev)
            exact_ms = hashed_ms = 0.0
            first = True
            for u, v, t in chunks:
                du = torch.from_numpy(u.view(np.int32)).to(dev)
                dv = torch.from_numpy(v.view(np.int32)).to(dev)
                dt = torch.from_numpy(t).to(dev)
                e = [ev() for _ in range(4)]
                torch.cuda.synchronize()
                e[0].record()
                plan = tn.Plan(du, dv, dt, n, **tuned[n][0])
                plan.apply(S, init=first)
                e[1].record()
                e[2].record()
                H, pu, pv = tn.tn_hash_proxy(du, dv, n, k, K, w["seed"])
                plans = [tn.Plan(pu[j].contiguous(), pv[j].contiguous(), dt, k, **tuned[n][1])
                         for j in range(K)]
                tn.tn_plan_apply_batch(plans, [P[j] for j in range(K)], init=first)
                e[3].record()
                torch.cuda.synchronize()
                exact_ms += e[0].elapsed_time(e[1])
                hashed_ms += e[2].elapsed_time(e[3])
                for p_ in plans:
                    p_.destroy()
                plan.destroy()
                del du, dv, dt, pu, pv
                first = False
            e = [ev() for _ in range(4)]
            e[0].record()
            exact, _, _ = tn.tn_out_sizes(S, n, n)
            e[1].record()
            e[2].record()
            est = tn.tn_hash_estimate(P, K, k, H, n)
            e[3].record()
            torch.cuda.synchronize()
            exact_ms += e[0].elapsed_time(e[1])
            hashed_ms += e[2].elapsed_time(e[3])
            err = tn.tn_error_stats(est, exact, n)
            ex = exact.cpu().numpy().view(np.uint32)
            points.append({"n": n, "m": m, "emd_w1": err["w1"], "emd_w1_over_n": err["w1"] / n,
                           "mean_rel_error": err["mean_rel"], "max_rel_error": err["max_rel"],
                           "mean_exact_size": float(ex.mean()),
                           "mean_estimate": float(est.cpu().numpy().view(np.uint32).mean()),
                           "exact_ms": exact_ms, "hashed_ms": hashed_ms,
                           "relative_time": hashed_ms / max(exact_ms, 1e-9),
                           "relative_memory": K * k * ((k + 63) // 64) / (n * ((n + 63) // 64))})
            print(json.dumps(points[-1]), file=sys.stderr, flush=True)
            del S, P, H
            m *= 10
    result = {"metric": "hashed estimate accuracy and cost against the exact matrix (ER sweep)",
              "value": float(np.mean([q["emd_w1_over_n"] for q in points])), "unit": "mean W1 / n over the sweep",
              "n_gpus": world, "steps": len(points), "warmup": 0,
              "ms_per_step": float(np.mean([q["exact_ms"] + q["hashed_ms"] for q in points])),
              "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": "u64",
              "data": "synthetic", "config": {"workload": w["desc"], "n_s": "0.3 n", "K": K, "chunk_events": chunk,
                                             "plan_options": {str(n): {"exact": o[0], "proxies": o[1]}
                                                              for n, o in tuned.items()}},
              "sweep": points}
    if rank == 0:
        print(json.dumps(result), flush=True)


def main():
    args = parse_args()
    w = WORKLOADS[args.workload]
    if w["kind"] == "serving":
        # jobs run on two streams each: with the default 8 hardware work queues a
        # job's short scheduling kernels wait behind other jobs' long updates that
        # share their queue; 32 is the most a context has (read at its creation)
        os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if w["kind"] == "serving" and args.impl == "ours":
        run_serving(args, w, rank, world, local_rank)
        return
    if w["kind"] == "hashed" and args.impl == "ours":
        run_hashed(args, w, rank, world, local_rank)
        return
    if w["kind"] == "online" and args.impl == "ours":
        run_online(args, w, rank, world, local_rank)
        return
    if w["kind"] == "scaled":
        if args.impl == "ours":
            run_scaled(args, w, rank, world, local_rank)
        elif rank == 0:
            print(json.dumps({"impl": "reference", "unavailable": "a profiling case of the GPU launch, not a "
                              "workload; its reference is the bursty workload's"}), flush=True)
        return
    if w["kind"] == "sweep":
        if args.impl == "ours":
            run_sweep(args, w, rank, world, local_rank)
        elif rank == 0:
            print(json.dumps({"impl": "reference", "unavailable": "the sweep compares two GPU paths; its oracle "
                              "counterpart is the parity suite"}), flush=True)
        return
    if args.impl == "reference":
        run_reference(args, w, rank, world)
        return

    import torch
    import paper_2307_04890_gb300 as tn
    from paper_2307_04890_gb300.build import build_library

    build_library()
    tn.load_library()
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=dev)

    n, m = w["n"], w["m"]
    u, v, t = make_events(w)  # every rank streams the same events (column split, below)
    du = torch.from_numpy(u.view(np.int32)).to(dev)
    dv = torch.from_numpy(v.view(np.int32)).to(dev)
    dt = torch.from_numpy(t).to(dev)
    # N > 1: rank r owns source columns [c0, c1) and the sizes are all-gathered
    c0, c1 = column_range(n, rank, world)
    ncols = c1 - c0
    src = None if world == 1 else torch.arange(c0, c1, dtype=torch.int32, device=dev)
    W = tn.tn_row_words(ncols)
    S = torch.empty((n, W), dtype=torch.int64, device=dev)
    stream = torch.cuda.current_stream(dev)

    k1_events = []
    opts = dict(window_events=args.window, slab_words=args.slab, smem_rows=0, resident_words=args.resident)
    tuned = None
    if args.autotune == "on" or (args.autotune == "auto" and w["kind"] in ("bursty", "er")):
        tuned = tn.tn_autotune(du, dv, dt, n, sample_events=args.tune_sample, ncols=ncols)
        opts = {key: tuned[key] if tuned["best_ms"] <= 1.05 * tuned["open_ms"] else 0  # (5 %: the timings' noise)
                for key in ("window_events", "slab_words", "smem_rows", "wave_ctas", "resident_words")}

    def step(record):
        plan = tn.Plan(du, dv, dt, n, **opts)                                            # a1
        if src is None:
            tn.tn_init_matrix(S, n)                                                      # a2
        else:
            tn.tn_init_matrix(S, n, ncols=ncols, src=src)
        if record:
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
        plan.apply(S, ncols=ncols, src=src)                                              # a3
        if record:
            e1.record(stream)
            k1_events.append((e0, e1))
        out, _, am = tn.tn_out_sizes(S, n, ncols, argmax=True)                           # a4
        out, am = gather_sizes(out, int(am.item()), n, rank, world, dist)                # (N > 1)
        stats = plan.stats()
        plan.destroy()
        return out, am, stats

    for _ in range(args.warmup):
        step(False)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    launches0 = tn.tn_kernel_launches()
    start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    with ClockSampler(torch.cuda.current_device()) as clocks:
        torch.cuda.synchronize()
        start.record(stream)
        for _ in range(args.steps):
            out, am, stats = step(True)
        end.record(stream)
        torch.cuda.synchronize()
    if dist:
        dist.barrier()
    launches = tn.tn_kernel_launches() - launches0
    ms_total = job_max_ms(start.elapsed_time(end), dist, dev)
    ms_step = ms_total / args.steps
    k1_ms = sum(a.elapsed_time(b) for a, b in k1_events) / len(k1_events)
    value = n * m / (ms_step * 1e-3)  # the whole matrix, all ranks together

    # roofline of the dominant kernel (the column-slab stream of this rank)
    words = (ncols + 63) // 64
    rw = opts.get("resident_words", 0)
    sw = opts["slab_words"]
    peak, peak_kind = measured_peaks()
    # An update whose rows are already equal moves no row, so the bytes of all
    # updates over the time are no bandwidth (they may exceed the peak); the
    # launch's DRAM bytes (ncu) are, or, without them, what no launch on these
    # sources can do without: the schedule in once and the matrix out once.
    update_bytes = m * 4 * words * 8
    traffic = profiled_traffic(args.workload, sw or None) if world == 1 and not rw else None
    alg_bytes = 8 * stats["ops"] + n * W * 8
    achieved = (traffic or alg_bytes) / (k1_ms * 1e-3) / 1e9
    roofline = {"bound": "hbm", "kernel": "stream_kernel" + (" (resident slabs)" if rw else ""),
                "achieved": achieved, "peak": peak,
                "peak_source": f"{peak_kind} MEASURED_PEAKS hbm_gbs" if peak_kind == "measured" else "fallback",
                "unit": "GB/s", "frac": achieved / peak, "traffic": traffic,
                "achieved_is": "DRAM bytes of the launch (ncu) / kernel time" if traffic else
                               "schedule in once + matrix out once / kernel time",
                "algorithmic_bytes_per_launch": alg_bytes, "kernel_ms": k1_ms,
                "update_bytes_per_launch": update_bytes,
                "update_bytes_are": "4 row segments per event, as if no update were skipped"}
    if traffic:
        roofline["dram_GBps"] = achieved
        roofline["dram_frac"] = achieved / peak

    result = {"metric": METRIC, "value": value, "unit": "bit-updates/s", "n_gpus": world, "steps": args.steps,
              "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True, "scaling": "strong",
              "vs_baseline": None, "dtype": "u64", "data": "synthetic",
              "config": {"workload": w["desc"], "n": n, "m": m, "global_batch": m,
                         "parallelism": f"source columns split over {world} GPUs, sizes all-gathered"
                                        if world > 1 else "single GPU",
                         "l2": "inputs larger than L2 (S %.2f GB, events %.0f MB)" % (n * W * 8 / 1e9, m * 16 / 1e6),
                         "window_events": opts["window_events"] or "chosen by the library",
                         "slab_words": None if rw else (sw or "chosen at launch"),
                         "smem_rows": None if rw else (opts["smem_rows"] or "default"),
                         "resident_words": rw or None,
                         "ctas": -(-words // rw) if rw else -(-tn.tn_row_words(ncols) // sw) if sw else None,
                         "autotuned": tuned is not None,
                         "levels": stats["levels"], "ops": stats["ops"], "windows": stats["windows"],
                         "global_memory_windows": stats["windows"] - stats["local_windows"]},
              "events_per_s": m / (ms_step * 1e-3),
              "roofline": roofline, "gpu_launches": launches, "clocks": clocks.summary(),
              "largest_out_component": {"node": int(am), "size": int(out.max().item())}}

    if rank == 0 and not args.no_e2e:
        # end to end through the host-buffer C-ABI call (same plan options), pinned
        # inputs copied in and the sizes copied out inside every timed call
        hu = torch.from_numpy(u.view(np.int32)).pin_memory()
        hv = torch.from_numpy(v.view(np.int32)).pin_memory()
        ht = torch.from_numpy(t).pin_memory()
        hout = torch.empty(n, dtype=torch.int32).pin_memory()
        ham = torch.empty(1, dtype=torch.int32).pin_memory()
        e2e_warm, e2e_steps = min(args.warmup, 1), min(args.steps, 3)
        for i in range(e2e_warm + e2e_steps):
            if i == e2e_warm:
                torch.cuda.synchronize()
                t0 = time.perf_counter()
            tn.tn_out_component_sizes_host_ptrs(hu.data_ptr(), hv.data_ptr(), ht.data_ptr(), m, n,
                                                hout.data_ptr(), ham.data_ptr(), **opts)
        e2e_s = (time.perf_counter() - t0) / e2e_steps
        assert np.array_equal(hout.numpy(), out.cpu().numpy()), "host entry point disagrees with device path"
        result["e2e"] = {"value": n * m / e2e_s, "unit": "bit-updates/s", "h2d_bytes_per_step": m * 16,
                         "d2h_bytes_per_step": n * 4 + 4, "ms_per_step": e2e_s * 1e3, "steps": e2e_steps,
                         "warmup": e2e_warm}

    if rank == 0 and not args.no_cpu_baseline:
        result["cpu_baseline"] = cpu_baseline_line(u, v, t, n, args.cpu_seconds, seed=w["seed"])
    if rank == 0:
        print(json.dumps(result), flush=True)
    if dist:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
