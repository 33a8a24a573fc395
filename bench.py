#!/usr/bin/env python
"""Benchmark: alias-table build and bulk sampling at n = 10^9 on GB300.

One step = one pass of the whole hot path over one batch: build the alias
table of n = 10^9 binary32 weights (exact total, light/heavy look-back scan,
split search, sweep) and draw k = 10^9 samples from it.  Steps cycle through
the paper's three n = 10^9 input shapes (uniform (0,1], Zipf 0.8 and Zipf 1.5,
randomly permuted; Sec. 10 "Input Data"), generated on the device from fixed
seeds.  Inputs (4 GB) exceed the 129 MB L2, so no flush is needed between
steps.

Printed JSON line (rank 0): ``value`` is the build throughput over all ranks
in Gweights/s; ``sample`` gives the sampling throughput (with a bare random
gather's rate and the sector-limited roofline beside it); ``e2e`` repeats the
step through the C ABI's host-buffer entry points with the host<->device
copies inside the timed region (two table objects double-buffered; the
serial one-table figure, its phases and the host link's rate per buffer
beside it); ``roofline`` is the dominant kernel against the measured HBM
copy bandwidth, with its DRAM traffic from the committed ncu summaries;
``cpu_baseline`` times the CPU oracle on a bounded sample of the same
workload.  The other rows ride on the same line: ``psa_plus`` (PSA+ builds),
``two_level`` (two-level tables, with ``os_nd`` output-sensitive sampling),
``many_tables`` (4096 tables built and sampled in one CUDA graph against one
table at a time), ``serving`` (a Poisson request stream against one request
at a time, then ``serving.load_sweep``: both paths at 0.5, 0.8 and 0.95 of
the plain path's saturation rate, ``--serve-loads``) and ``small_exact`` (n =
10^6 u32 weights, k = 10^6: build and sample latency in microseconds, L2
resident, checked bit for bit against the oracle), each with the oracle
timed beside it where it applies.

``--impl reference`` times the CPU oracle itself (the reference arm of this
repository) on bounded samples of the same workload.

Multi-GPU: the path does not shard (one table per GPU); under torchrun every
rank runs an independent replica and ``value`` sums their work over the
slowest rank's time.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "alias build Gweights/s + sample Gsamples/s at n=1e9 (% HBM roofline); p99 ms"
UNIT = "Gweights/s"
DISTS = {  # name -> (generator kind, Zipf exponent, seed)
    "uniform": ("f32_uniform", 1.0, 7),
    "zipf0.8": ("f32_zipf", 0.8, 5),
    "zipf1.5": ("f32_zipf", 1.5, 6),
}
# algorithmic bytes per unit (weights for the build kernels, samples for the query)
ALGO_BYTES = {"stats": 4, "stats_combine": 0, "classify": 4, "tilescan": 0, "split": 0, "sweep": 16, "sample": 16}
BUILD_BYTES_PER_WEIGHT = 24  # three 4-B weight reads + 12-B (threshold, alias) payload
SECTOR_BYTES_PER_SAMPLE = 36  # a random gather's floor: one 32-B sector + a 4-B coalesced store
KERNEL_NAMES = {"stats": "k_stats", "stats_combine": "k_stats_combine", "classify": "k_classify",
                "tilescan": "k_tilescan", "split": "k_split", "sweep": "k_sweep", "sample": "k_sample"}


def parse():
    ap = argparse.ArgumentParser(description=__doc__.splitlines()[0])
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=6)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--n", type=int, default=10 ** 9)
    ap.add_argument("--k", type=int, default=10 ** 9)
    ap.add_argument("--dists", default="uniform,zipf0.8,zipf1.5")
    ap.add_argument("--e2e-steps", type=int, default=3)
    ap.add_argument("--cpu-sample", type=int, default=20_000_000,
                    help="weights (and samples) per distribution for the CPU-oracle baseline")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-clocks", action="store_true")
    ap.add_argument("--no-two-level", action="store_true")
    ap.add_argument("--no-psa-plus", action="store_true")
    ap.add_argument("--batch-tables", type=int, default=4096,
                    help="tables of the many-distribution workload (0: skip it)")
    ap.add_argument("--batch-steps", type=int, default=10)
    ap.add_argument("--serve-requests", type=int, default=100_000,
                    help="requests of the serving workload (0: skip it)")
    ap.add_argument("--serve-rate", type=float, default=20_000.0, help="Poisson arrival rate, requests/s")
    ap.add_argument("--serve-loads", default="0.5,0.8,0.95",
                    help="comma-separated fractions of the plain path's saturation rate to offer in a load "
                         "sweep after the serving run (empty: no sweep)")
    ap.add_argument("--no-small", action="store_true",
                    help="skip the small exact configuration (n = 10^6 u32 weights, L2-resident latency)")
    ap.add_argument("--serve-sweep-requests", type=int, default=20_000, help="requests per load-sweep point")
    return ap.parse_args()


def measured_peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


_CSRC = "paper_1903_00227_gb300/csrc/"
_PSA = (_CSRC + "wrs_kernels.cuh", _CSRC + "wrs_pack.cuh", _CSRC + "wrs_device.cuh")
KERNEL_SOURCES = {  # the files each measured kernel is compiled from
    "psa": _PSA,
    "two_level": _PSA + (_CSRC + "wrs_twolevel.cuh",),
    "os_nd": _PSA + (_CSRC + "wrs_twolevel.cuh", _CSRC + "wrs_osnd.cuh"),
    "psa_plus": _PSA + (_CSRC + "wrs_twolevel.cuh", _CSRC + "wrs_psaplus.cuh"),
}


def kernel_family(name: str) -> str:
    if name.startswith("k_pp"):
        return "psa_plus"
    return "os_nd" if name.startswith("k_os") else ("two_level" if name.startswith("k2_") else "psa")


def source_sha(family: str = "psa") -> str:
    h = hashlib.sha256()
    for rel in KERNEL_SOURCES[family]:
        with open(os.path.join(ROOT, rel), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def traffic_for(stage: str, units: int):
    """DRAM bytes per launch from the committed ncu summary, if it was taken
    on the current source of that kernel; else None.  `stage` is a build
    stage or a kernel name."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(path):
        return None
    with open(path) as f:
        d = json.load(f)
    name = KERNEL_NAMES.get(stage, stage)
    e = d.get("kernels", {}).get(name)
    if not e or e.get("source_sha") != source_sha(kernel_family(name)):
        return None
    return float(e["dram_bytes_per_unit"]) * units


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int, enabled: bool):
        self.proc = None
        self.path = os.path.join(os.environ.get("WRS_CLOCKS_DIR", tempfile.gettempdir()),
                                 f"clocks_bench_{os.getpid()}.csv")
        self.gpu = gpu_index
        if enabled:
            try:
                os.makedirs(os.path.dirname(self.path), exist_ok=True)
                self.fh = open(self.path, "w")
                self.proc = subprocess.Popen(
                    ["nvidia-smi", "-i", str(gpu_index), f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                     "-lms", "200"], stdout=self.fh, stderr=subprocess.DEVNULL)
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
        self.fh.close()
        sm, mx, reasons = [], [], set()
        names = ("hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap")
        with open(self.path) as f:
            for line in f:
                p = [x.strip() for x in line.split(",")]
                if len(p) < 9:
                    continue
                try:
                    sm.append(float(p[1]))
                    mx.append(float(p[2]))
                except ValueError:
                    continue
                for name, v in zip(names, p[5:9]):
                    if v.lower().startswith("active"):
                        reasons.add(name)
        if not sm:
            return None
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(mx), "reasons": sorted(reasons),
                "samples": len(sm)}


def reduce_max(values, device):
    """Max over ranks of a list of floats (identity on one rank)."""
    import torch
    import torch.distributed as dist

    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return [float(v) for v in values]
    t = torch.tensor([float(v) for v in values], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return t.tolist()


def job_rates(world: int, steps: int, n: int, k: int, t_build_ms: float, t_sample_ms: float):
    """Whole-job throughput of `world` replicas that each built `steps` tables
    of n weights and drew `steps` x k samples, timed by the slowest rank:
    (Gweights/s, Gsamples/s)."""
    return (world * steps * n / (t_build_ms * 1e-3) / 1e9, world * steps * k / (t_sample_ms * 1e-3) / 1e9)


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def cpu_oracle_run(names, n_s: int, repeats: int = 1):
    """Time the CPU oracle (quantize + Alg. 2 sweep, then n_s queries) on the
    first n_s weights of each distribution's recipe.  Returns totals."""
    from oracle import wrs_oracle as O
    from paper_1903_00227_gb300 import workloads as WL

    tb = ts = 0.0
    nw = nsmp = 0
    steps = []
    for r in range(repeats):
        for name in names:
            kind, s, seed = DISTS[name]
            w = WL.generate(kind, n_s, seed, s)
            t0 = time.perf_counter()
            qz = O.quantize(w)
            tab = O.sweep(qz)
            t1 = time.perf_counter()
            O.sample(tab.thr, tab.alias, tab.Qp, n_s, 2, 0)
            t2 = time.perf_counter()
            tb += t1 - t0
            ts += t2 - t1
            nw += n_s
            nsmp += n_s
            steps.append((t2 - t0) * 1e3)
    return tb, ts, nw, nsmp, steps


def cpu_other_builders(names, n_s: int):
    """The oracle's other sequential builders on the same bounded sample, as
    they stand (one thread): Vose's method in binary64 (Alg. 1, the paper's
    sequential baseline) and the exact PSA (Alg. 3) with 64 subproblems run
    one after another."""
    from oracle import wrs_oracle as O
    from paper_1903_00227_gb300 import workloads as WL

    tv = tp = 0.0
    nw = 0
    for name in names:
        kind, s, seed = DISTS[name]
        w = WL.generate(kind, n_s, seed, s)
        t0 = time.perf_counter()
        O.vose_f64(w)
        t1 = time.perf_counter()
        O.psa(O.quantize(w), 64)
        t2 = time.perf_counter()
        tv += t1 - t0
        tp += t2 - t1
        nw += n_s
    return {"vose_f64_gweights_s": nw / tv / 1e9, "psa64_gweights_s": nw / tp / 1e9}


def cpu_rows(names, n_s: int, batch_tables: int):
    """The oracle timed beside each of the other rows, one thread, on bounded
    samples of the same recipes (quantisation included in every build)."""
    from oracle import wrs_oracle as O
    from paper_1903_00227_gb300 import workloads as WL

    res = {}
    tq = tpp = t2b = t2s = 0.0
    nw = 0
    tl_z = qz_z = None
    for name in names:
        kind, s, seed = DISTS[name]
        w = WL.generate(kind, n_s, seed, s)
        t0 = time.perf_counter()
        qz = O.quantize(w)
        t1 = time.perf_counter()
        O.psa_plus(qz, 2048)
        t2 = time.perf_counter()
        tl = O.build_2lvl(qz)
        t3 = time.perf_counter()
        O.sample_2lvl(tl, n_s, 3, 0)
        t4 = time.perf_counter()
        tq += t1 - t0
        tpp += t2 - t1
        t2b += t3 - t2
        t2s += t4 - t3
        nw += n_s
        if name == "zipf1.5":
            tl_z, qz_z = tl, qz
    sample = f"first {n_s:,} weights of each of {', '.join(names)}; one thread"
    res["psa_plus"] = {"build_gweights_s": nw / (tq + tpp) / 1e9, "cores": 1, "sample": sample}
    res["two_level"] = {"build_gweights_s": nw / (tq + t2b) / 1e9, "sample_gsamples_s": nw / t2s / 1e9,
                        "cores": 1, "sample": sample}
    if tl_z is not None:
        k = 10 ** 9
        t0 = time.perf_counter()
        items, _ = O.os_nd(qz_z, tl_z, k, 5, 0)
        dt = time.perf_counter() - t0
        res["os_nd"] = {"gsamples_s": k / dt / 1e9, "pairs": int(len(items)), "seconds": dt, "cores": 1,
                        "sample": f"first {n_s:,} weights of zipf1.5, k = 10^9; one thread"}
    if batch_tables > 0:
        nb, kb, kinds, seeds = WL.batch_plan(batch_tables, 4)
        m = min(256, len(nb))
        ws_ = [WL.generate(kinds[t], nb[t], seeds[t], 1.0) for t in range(m)]
        t0 = time.perf_counter()
        for t in range(m):
            qz = O.quantize(ws_[t])
            tab = O.sweep(qz)
            if kb[t]:
                O.sample(tab.thr, tab.alias, tab.Qp, kb[t], 11, t)
        dt = time.perf_counter() - t0
        res["many_tables"] = {"gweights_s": sum(nb[:m]) / dt / 1e9, "tables_per_s": m / dt, "cores": 1,
                              "sample": f"first {m} tables of the workload, quantize + Alg. 2 sweep + "
                                        "their samples; one thread"}
    return res


def cpu_psa_all_cores(names, n_s: int):
    """The oracle's exact PSA (Alg. 3) with P = host threads subproblems, its
    P - 1 splits and P packs run on P host threads (the oracle's own split
    and pack steps; ctypes releases the interpreter lock), on the same bounded
    sample; quantisation and the two traversals with their prefix sums run on
    one thread, as the oracle writes them."""
    from oracle import wrs_oracle as O
    from paper_1903_00227_gb300 import workloads as WL

    nt = max(1, os.cpu_count() or 1)
    tq = tt = 0.0
    nw = 0
    phases = {"begin_s": 0.0, "splits_s": 0.0, "packs_s": 0.0, "end_s": 0.0}
    for name in names:
        kind, s, seed = DISTS[name]
        w = WL.generate(kind, n_s, seed, s)
        t0 = time.perf_counter()
        qz = O.quantize(w)
        t1 = time.perf_counter()
        ph = {}
        O.psa_threads(qz, nt, nt, ph)
        t2 = time.perf_counter()
        tq += t1 - t0
        tt += t2 - t1
        nw += n_s
        for key in phases:
            phases[key] += ph[key]
    return {"psa_all_cores_gweights_s": nw / (tq + tt) / 1e9, "psa_all_cores_threads": nt,
            "psa_all_cores_phase_s": {"quantize_s": tq, **phases}}


def cpu_sample_all_cores(n_s: int):
    """The oracle's sampler on every host core: threads draw disjoint ranges
    of sample indices with the oracle's indexed query (ctypes releases the
    interpreter lock during the C call), from a table of n_s uniform weights."""
    from concurrent.futures import ThreadPoolExecutor

    import numpy as np

    from oracle import wrs_oracle as O
    from paper_1903_00227_gb300 import workloads as WL

    kind, s, seed = DISTS["uniform"]
    qz, tab = O.build_table(WL.generate(kind, n_s, seed, s))
    nt = max(1, os.cpu_count() or 1)
    k = 4 * n_s
    chunks = [np.arange(i * k // nt, (i + 1) * k // nt, dtype=np.uint64) for i in range(nt)]
    t0 = time.perf_counter()
    with ThreadPoolExecutor(nt) as ex:
        list(ex.map(lambda c: O.sample_at(tab.thr, tab.alias, tab.Qp, 2, 0, c), chunks))
    dt = time.perf_counter() - t0
    return {"sample_gsamples_s_all_cores": k / dt / 1e9, "sample_threads": nt}


def cpu_baseline(names, n_s: int):
    tb, ts, nw, nsmp, _ = cpu_oracle_run(names, n_s)
    out = {"value": nw / tb / 1e9, "unit": UNIT, "cores": 1, "kind": "oracle",
           "sample_gsamples_s": nsmp / ts / 1e9,
           "sample": f"first {n_s:,} weights of each of {', '.join(names)} (same recipes), "
                     f"exact quantize + Alg. 2 sweep, then {n_s:,} queries each; single thread"}
    out.update(cpu_other_builders(names, n_s))
    out.update(cpu_psa_all_cores(names, n_s))
    out.update(cpu_sample_all_cores(n_s))
    out["cpu_model"] = cpu_model()
    out["host_threads"] = os.cpu_count()
    return out


def cpu_model() -> str:
    try:
        with open("/proc/cpuinfo") as f:
            for line in f:
                if line.lower().startswith(("model name", "cpu part")):
                    return line.split(":", 1)[1].strip()
    except OSError:
        pass
    import platform

    return platform.machine()


def config(args, names):
    return {"workload": f"n={args.n:.0e} binary32 weights ({', '.join(names)}; randomly permuted), "
                        f"table build + k={args.k:.0e} samples per step, steps cycle the distributions",
            "n": args.n, "k": args.k, "dists": names, "tile": 2048,
            "l2": "inputs larger than L2 (4 GB weights, 16 GB table vs 129 MB L2)",
            "parallelism": "replicas"}


def run_reference(args, names):
    ws, rank, _ = dist_env()
    if rank != 0:
        return 0
    n_s = min(args.cpu_sample, args.n) // 4  # each step: one distribution, bounded sample
    for i in range(args.warmup):
        cpu_oracle_run([names[i % len(names)]], n_s)
    tb = ts = 0.0
    nw = 0
    steps = []
    for i in range(args.steps):
        b, s, w_, _, st = cpu_oracle_run([names[i % len(names)]], n_s)
        tb += b
        ts += s
        nw += w_
        steps += st
    value = nw / tb / 1e9
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": statistics.mean(steps), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "u128", "data": "synthetic",
            "config": config(args, names), "impl": "reference",
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
                             "sample": f"each step: first {n_s:,} weights of one distribution, "
                                       f"quantize + sweep + {n_s:,} queries, single thread"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


TWO_LEVEL_BYTES_PER_WEIGHT = 20  # two 4-B weight reads + 12-B payload (upper levels: < 0.1%)


def run_two_level(args, torch, wrs, weights, names, stream, peak):
    """The two-level ("2lvl-sweep") table on the same inputs: build and k
    samples per distribution, CUDA events on the launching stream."""
    n, k = args.n, args.k
    sh = stream.cuda_stream
    t2 = wrs.AliasTable2(n)
    out = torch.empty(k, dtype=torch.int32, device="cuda")
    per = {}
    for name in names:
        w = weights[name]
        for _ in range(2):
            t2.build(w, stream=sh)
            t2.sample(k, 1, out=out, stream=sh)
        torch.cuda.synchronize()
        bt, st = [], []
        for i in range(max(3, args.steps // 2)):
            e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
            e0.record(stream)
            t2.build(w, stream=sh)
            e1.record(stream)
            t2.sample(k, 100 + i, out=out, stream=sh)
            e2.record(stream)
            e2.synchronize()
            bt.append(e0.elapsed_time(e1))
            st.append(e1.elapsed_time(e2))
        if t2.status() != wrs.OK:
            raise RuntimeError("two-level build failed")
        bm, sm_ = statistics.mean(bt), statistics.mean(st)
        per[name] = {"build_ms": bm, "build_gweights_s": n / (bm * 1e-3) / 1e9,
                     "build_frac": TWO_LEVEL_BYTES_PER_WEIGHT * n / (bm * 1e-3) / 1e9 / peak,
                     "sample_ms": sm_, "sample_gsamples_s": k / (sm_ * 1e-3) / 1e9}
    levels = t2.levels()
    t2.free()
    bmean = statistics.mean(v["build_ms"] for v in per.values())
    smean = statistics.mean(v["sample_ms"] for v in per.values())
    return {"build_gweights_s": n / (bmean * 1e-3) / 1e9, "sample_gsamples_s": k / (smean * 1e-3) / 1e9,
            "roofline_build": {"bound": "hbm", "achieved": TWO_LEVEL_BYTES_PER_WEIGHT * n / (bmean * 1e-3) / 1e9,
                               "peak": peak, "unit": "GB/s", "traffic_k2_group": traffic_for("k2_group", n),
                               "frac": TWO_LEVEL_BYTES_PER_WEIGHT * n / (bmean * 1e-3) / 1e9 / peak,
                               "algorithmic_bytes_per_weight": TWO_LEVEL_BYTES_PER_WEIGHT},
            "levels": levels, "per_dist": per,
            "note": "wrs_table2_*: Alg. 2 per group of 2048, group totals as the next level (Sec. 6); "
                    "a different table from the headline's PSA table, same sampling distribution"}


PSA_PLUS_BYTES_PER_WEIGHT = 20  # two 4-B weight reads + 12-B payload (the leftovers' passes come on top)


def run_psa_plus(args, torch, wrs, table, weights, names, stream, peak):
    """PSA+ builds (wrs_table_build_psa_plus) of the same inputs into the
    headline's table object, CUDA events on the launching stream; the sampler
    is the headline's (same table format)."""
    n = args.n
    sh = stream.cuda_stream
    per = {}
    for name in names:
        w = weights[name]
        for _ in range(2):
            table.build_psa_plus(w, stream=sh)
        torch.cuda.synchronize()
        bt = []
        for i in range(max(3, args.steps // 2)):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record(stream)
            table.build_psa_plus(w, stream=sh)
            e1.record(stream)
            e1.synchronize()
            bt.append(e0.elapsed_time(e1))
        if table.status() != wrs.OK:
            raise RuntimeError("PSA+ build failed")
        left = table.psa_plus_leftovers()
        bm = statistics.mean(bt)
        per[name] = {"build_ms": bm, "build_gweights_s": n / (bm * 1e-3) / 1e9,
                     "build_frac": PSA_PLUS_BYTES_PER_WEIGHT * n / (bm * 1e-3) / 1e9 / peak,
                     "leftover_fraction": left / n}
    bmean = statistics.mean(v["build_ms"] for v in per.values())
    ach = PSA_PLUS_BYTES_PER_WEIGHT * n / (bmean * 1e-3) / 1e9
    return {"build_gweights_s": n / (bmean * 1e-3) / 1e9,
            "roofline_build": {"bound": "hbm", "achieved": ach, "peak": peak, "unit": "GB/s", "frac": ach / peak,
                               "algorithmic_bytes_per_weight": PSA_PLUS_BYTES_PER_WEIGHT},
            "per_dist": per,
            "note": "wrs_table_build_psa_plus: Alg. 2 per tile of 2048 until an item outside the tile is needed, "
                    "then PSA on the leftovers (Sec. 4.2); a different table from PSA's, same distribution"}


def run_os_nd(args, torch, wrs, weights, stream):
    """OS-ND output-sensitive sampling (wrs_table2_sample_os) on the two-level
    table of the skewed inputs, against k alias queries of the same table
    (timed for k <= 10^9; the alias time of larger k is that rate)."""
    n = args.n
    sh = stream.cuda_stream
    t2 = wrs.AliasTable2(n)
    cap = n + 128 * (n // wrs.TABLE2_GROUP + 1) + 1
    items = torch.empty(cap, dtype=torch.int32, device="cuda")
    counts = torch.empty(cap, dtype=torch.int64, device="cuda")
    npairs = torch.zeros(1, dtype=torch.int64, device="cuda")
    qout = torch.empty(min(args.k, 10 ** 9), dtype=torch.int32, device="cuda")
    res = {}
    for name in [d for d in ("zipf1.5", "zipf0.8") if d in weights]:
        w = weights[name]
        t2.build(w, stream=sh)
        ks = (10 ** 9, 10 ** 12) if name == "zipf1.5" else (10 ** 12,)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        kq = qout.numel()
        t2.sample(kq, 3, out=qout, stream=sh)
        e0.record(stream)
        t2.sample(kq, 4, out=qout, stream=sh)
        e1.record(stream)
        e1.synchronize()
        alias_rate = kq / (e0.elapsed_time(e1) * 1e-3)
        for k in ks:
            ts = []
            for i in range(3):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                rc = wrs.table2_sample_os(t2.handle, w.data_ptr(), wrs.F32, k, 50 + i, 0, items.data_ptr(),
                                          counts.data_ptr(), cap, npairs.data_ptr(), sh)
                e1.record(stream)
                e1.synchronize()
                assert rc == wrs.OK, wrs.status_str(rc)
                if i:
                    ts.append(e0.elapsed_time(e1))
            m = int(npairs.item())
            assert m <= cap and int(counts[:m].sum().item()) == k
            ms = statistics.mean(ts)
            res[f"{name}_k{k:.0e}"] = {"k": k, "pairs": m, "ms": ms, "gsamples_s": k / (ms * 1e-3) / 1e9,
                                       "alias_queries_ms_equivalent": k / alias_rate * 1e3,
                                       "speedup_vs_alias": (k / alias_rate * 1e3) / ms}
    t2.free()
    return res


def run_batched(args, torch, WL, wrs, stream):
    """Many-distribution workload: 4096 tables, sizes log-uniform in [32, 2^20],
    binary32 uniform or Zipf(1.0) by seed, k log-uniform in [1, 4096].  One
    step builds and samples every table.  The batched path (seven build
    launches + one sample launch over all tables, captured once in a CUDA
    graph, sweep grouping from the autotuner) against the plain path (one
    wrs_table per distribution: its build and sample calls, table after
    table, on one stream).  Both must give the same samples."""
    sh = stream.cuda_stream
    n, k, kinds, seeds = WL.batch_plan(args.batch_tables, 4)
    batch = wrs.AliasBatch(n)
    off = batch.offsets
    buf = torch.empty(off[-1], dtype=torch.float32, device="cuda")
    for t in range(len(n)):
        WL.generate_device(kinds[t], n[t], seeds[t], 1.0, out=buf[off[t]:off[t] + n[t]])
    koff = batch.set_samples(k)
    out_b = torch.empty(max(koff[-1], 1), dtype=torch.int32, device="cuda")
    out_p = torch.empty_like(out_b)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    tuned_ms = batch.tune(buf, stream=sh)
    tune_s = time.perf_counter() - t0
    for _ in range(3):
        batch.build(buf, stream=sh)
        batch.sample(11, 0, out=out_b, stream=sh)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):  # captured on torch's side stream, replayed on `stream`
        batch.build(buf)
        batch.sample(11, 0, out=out_b)
    for _ in range(3):
        graph.replay()
    torch.cuda.synchronize()
    times = []
    for _ in range(args.batch_steps):
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        graph.replay()
        e1.record(stream)
        e1.synchronize()
        times.append(e0.elapsed_time(e1))
    rc, st = batch.status()
    if rc != wrs.OK:
        raise RuntimeError(f"batched build failed: {wrs.status_str(rc)}")

    tables = [wrs.AliasTable(nt) for nt in n]
    views = [buf[off[t]:off[t] + n[t]] for t in range(len(n))]
    outs = [out_p[koff[t]:koff[t] + k[t]] for t in range(len(n))]

    def plain_step():
        for t, tab in enumerate(tables):
            tab.build(views[t], stream=sh)
            if k[t]:
                tab.sample(k[t], 11, t, out=outs[t], stream=sh)

    plain_step()
    torch.cuda.synchronize()
    ptimes = []
    for _ in range(max(2, args.batch_steps // 3)):
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        plain_step()
        e1.record(stream)
        e1.synchronize()
        ptimes.append(e0.elapsed_time(e1))
    identical = bool(torch.equal(out_b[:koff[-1]], out_p[:koff[-1]]))
    for tab in tables:
        tab.free()
    groups = batch.groups()
    batch.free()
    total_w, total_k = sum(n), sum(k)
    bms, pms = statistics.mean(times), statistics.mean(ptimes)
    srt = sorted(times)
    return {
        "workload": f"{len(n)} tables, sizes log-uniform in [32, 2^20] (total {total_w} binary32 weights), "
                    f"uniform (0,1] or Zipf 1.0 by seed, k log-uniform in [1, 4096] (total {total_k})",
        "batched": {"ms_per_step": bms, "p99_ms": srt[min(len(srt) - 1, int(round(0.99 * (len(srt) - 1))))],
                    "gweights_s": total_w / (bms * 1e-3) / 1e9, "tables_per_s": len(n) / (bms * 1e-3),
                    "launches_per_step": 8 + (1 if any(x <= 2048 for x in n) else 0), "cuda_graph": True,
                    "tuned_groups": groups, "tuned_sweep_ms": tuned_ms, "tune_seconds": tune_s,
                    "one_block_tables": sum(1 for x in n if x <= 2048),
                    "roofline_build": {"algorithmic_bytes": 24 * total_w,
                                       "frac": 24 * total_w / (bms * 1e-3) / 1e9 / measured_peaks()[0],
                                       "note": "24 B/weight over all tables' weights against the measured copy "
                                               "bandwidth; the step also draws the samples"}},
        "plain": {"ms_per_step": pms, "gweights_s": total_w / (pms * 1e-3) / 1e9,
                  "tables_per_s": len(n) / (pms * 1e-3),
                  "launches_per_step": 7 * len(n) + sum(1 for x in k if x),
                  "note": "one wrs_table per distribution, wrs_table_build + wrs_sample per table on one stream"},
        "speedup": pms / bms,
        "identical_samples": identical,
    }


def run_serving(args, torch):
    """Serving workload: a seeded Poisson stream of requests, 30% build+sample
    (binary32 Zipf 1.0 weights uploaded from pinned host memory, sizes
    log-uniform in [2^10, 2^24]) and 70% sample-only against resident tables,
    k log-uniform in [1, 10^5], under a 40 GB device-memory budget with LRU
    eviction.  The continuous-batching server against the plain path (one
    request at a time) on the same stream; both must give the same samples."""
    from paper_1903_00227_gb300 import serve as S

    reqs = S.request_stream(args.serve_requests, rate=args.serve_rate, seed=5)
    srv = S.Server(budget=40 << 30, max_inflight=3, tick_requests=2048, tick_samples=1 << 24)
    t0 = time.perf_counter()
    reserved = srv.reserve(reqs)
    setup_s = time.perf_counter() - t0
    served = srv.run(reqs)
    srv.cache.clear_resident()
    plain = srv.run_plain(reqs)
    same = bool((served["checksum"] == plain["checksum"]).all())
    out = {"workload": f"{len(reqs)} requests, Poisson {args.serve_rate:g}/s, 30% build+sample (Zipf 1.0, "
                       f"n log-uniform in [2^10, 2^24]), 70% sample-only, k log-uniform in [1, 10^5], "
                       f"40 GB budget, LRU eviction",
           "served": S.summarize(served, reqs), "plain": S.summarize(plain, reqs),
           "identical_samples": same, "table_objects_reserved": reserved, "reserve_seconds": setup_s,
           "objects_created_total": srv.cache.created, "objects_freed": srv.cache.freed}
    loads = [float(x) for x in args.serve_loads.split(",") if x.strip()]
    if loads:
        # offered loads below the plain path's saturation rate, which the run
        # above measured (its arrivals outpace the plain path), so that both
        # paths are compared at a load each can sustain
        sat = out["plain"]["requests_per_s"]
        points = []
        for f in loads:
            rq = S.request_stream(args.serve_sweep_requests, rate=f * sat, seed=6)
            srv.cache.clear_resident()
            a = srv.run(rq)
            srv.cache.clear_resident()
            b = srv.run_plain(rq)
            points.append({"load": f, "rate": f * sat, "served": S.summarize(a, rq), "plain": S.summarize(b, rq),
                           "identical_samples": bool((a["checksum"] == b["checksum"]).all())})
        out["load_sweep"] = {"plain_saturation_rate": sat, "requests_per_point": args.serve_sweep_requests,
                             "points": points}
    srv.close()
    return out


def run_small(torch, WL, wrs, stream, reps: int = 50):
    """The small exact configuration: n = 10^6 u32 weights uniform in [1, 2^24]
    (seed 1), built as 64 split pieces (the table does not depend on the
    split count), then k = 10^6 samples (seed 2, stream 0).  Table (4 MB of
    weights, 16 MB of buckets) and samples stay in L2, so the figures are
    latencies in microseconds (median of `reps` CUDA-event timings on the
    launching stream), not an HBM claim.  The table and samples are checked
    against the oracle once."""
    from oracle import wrs_oracle as O
    import numpy as np

    n, k = 1_000_000, 1_000_000
    w = WL.u32_uniform(n, 1)
    w_dev = torch.from_numpy(w.view(np.int32).copy()).cuda()
    out = torch.empty(k, dtype=torch.int32, device="cuda")
    sh = stream.cuda_stream
    tb, ts = [], []
    with wrs.AliasTable(n) as t:
        for i in range(reps + 3):
            e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
            e0.record(stream)
            t.build(w_dev, stream=sh)
            e1.record(stream)
            t.sample(k, seed=2, stream_id=0, out=out, stream=sh)
            e2.record(stream)
            e2.synchronize()
            if i >= 3:
                tb.append(e0.elapsed_time(e1) * 1e3)
                ts.append(e1.elapsed_time(e2) * 1e3)
        if t.status() != wrs.OK:
            raise RuntimeError("small configuration: build failed")
        thr, alias, _ = t.download()
    qz, tab = O.build_table(w)
    want = O.sample(tab.thr, tab.alias, tab.Qp, k, 2, 0)
    exact = bool(np.array_equal(thr, tab.thr) and np.array_equal(alias, tab.alias)
                 and np.array_equal(out.cpu().numpy().view(np.uint32), want))
    b_us, s_us = statistics.median(tb), statistics.median(ts)
    return {"workload": "n=1e6 u32 weights uniform in [1, 2^24] (seed 1), 64 split pieces, k=1e6 samples "
                        "(seed 2, stream 0)",
            "build_us": b_us, "sample_us": s_us, "build_gweights_s": n / (b_us * 1e-6) / 1e9,
            "sample_gsamples_s": k / (s_us * 1e-6) / 1e9, "reps": reps, "bit_exact_vs_oracle": exact,
            "l2_resident": True, "note": "4 MB weights and 16 MB table fit in the 129 MB L2: latency, no HBM claim"}


def run_e2e(args, torch, wrs, table, weights, names, stream, ws):
    """The step through the C ABI's host-buffer entry points, with every host
    <-> device copy inside the timed region: wrs_table_build_host uploads
    the step's weights from pinned memory and builds, wrs_sample_host draws k
    samples and returns them in pinned memory.  `value`: a stream of steps on
    two table objects and two CUDA streams, step i+1's upload and build
    issued before step i's sampling (double buffering: the link carries one
    step's weights while the GPU samples the other's table).  `serial`: one
    table, one step at a time."""
    n, k = args.n, args.k
    K = args.e2e_steps
    h_in = {}
    for name in names:  # each distribution's weights in pinned host memory (prepared once, untimed)
        h_in[name] = torch.empty(n, dtype=torch.float32, pin_memory=True)
        h_in[name].copy_(weights[name])
    h_out = [torch.empty(k, dtype=torch.int32, pin_memory=True) for _ in range(2)]
    torch.cuda.synchronize()
    # the host link's rate on this machine for each pinned buffer the step uses
    # (whole buffer, best of 2), for context: the upload reads h_in, the
    # download writes h_out
    def copy_rate(dst, src, nbytes):
        best = 0.0
        for _ in range(2):
            e0, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            e0.record(stream)
            dst.copy_(src, non_blocking=True)
            e1.record(stream)
            e1.synchronize()
            best = max(best, nbytes / (e0.elapsed_time(e1) * 1e-3) / 1e9)
        return best

    dbuf = torch.empty(max(n, k), dtype=torch.int32, device="cuda")
    up = {name: copy_rate(dbuf[:n].view(torch.float32), h_in[name], 4 * n) for name in names}
    down = [copy_rate(h, dbuf[:k], 4 * k) for h in h_out]
    del dbuf
    link = {"h2d": min(up.values()), "d2h": min(down), "h2d_per_input": up, "d2h_per_output": down}

    def build_host(t, name, sh):
        rc = wrs.table_build_host(t.handle, h_in[name].data_ptr(), n, wrs.F32, sh)
        assert rc == wrs.OK, wrs.status_str(rc)

    def sample_host(t, i, slot, sh):
        rc = wrs.sample_host(t.handle, k, 5000 + i, 0, h_out[slot].data_ptr(), sh)
        assert rc == wrs.OK, wrs.status_str(rc)

    # serial: one table, one step at a time (first call allocates the staging buffers)
    sh0 = stream.cuda_stream
    times, t_up, t_down, t_bld, per_step = [], [], [], [], []
    for i in range(K + 1):
        name = names[i % len(names)]
        torch.cuda.synchronize()
        e0, em, e1 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        e0.record(stream)
        build_host(table, name, sh0)
        em.record(stream)
        sample_host(table, i, 0, sh0)
        e1.record(stream)
        e1.synchronize()
        if i > 0:
            times.append(e0.elapsed_time(e1))
            t_up.append(e0.elapsed_time(em))
            t_down.append(em.elapsed_time(e1))
            t_bld.append(sum(table.stage_ms().values()))  # the build's own kernels (stage events)
            per_step.append({"input": name, "upload_build_ms": t_up[-1], "build_kernels_ms": t_bld[-1],
                             "upload_gbs": 4 * n / max(1e-9, (t_up[-1] - t_bld[-1]) * 1e-3) / 1e9,
                             "sample_download_ms": t_down[-1]})
    t_serial = reduce_max([statistics.mean(times)], "cuda")[0]

    # pipelined: two table objects on two streams
    tables = [table, wrs.AliasTable(n)]
    streams = [stream, torch.cuda.Stream()]
    shs = [x.cuda_stream for x in streams]
    build_host(tables[1], names[0], shs[1])  # warm-up: staging buffers of the second object
    sample_host(tables[1], 0, 1, shs[1])
    torch.cuda.synchronize()
    steps = max(2 * K, 6)
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(streams[0])
    streams[1].wait_event(e0)
    build_host(tables[0], names[0], shs[0])
    for i in range(steps):
        cur, nxt = i % 2, (i + 1) % 2
        if i + 1 < steps:
            build_host(tables[nxt], names[(i + 1) % len(names)], shs[nxt])
        sample_host(tables[cur], i, cur, shs[cur])  # returns with the samples in host memory
    done = torch.cuda.Event()
    done.record(streams[1])
    streams[0].wait_event(done)
    e1.record(streams[0])
    e1.synchronize()
    t_pipe = reduce_max([e0.elapsed_time(e1) / steps], "cuda")[0]
    for t in tables:
        if t.status() != wrs.OK:
            raise RuntimeError("end-to-end build failed")
    tables[1].free()
    del h_in, h_out
    return {"value": ws * n / (t_pipe * 1e-3) / 1e9, "unit": UNIT, "h2d_bytes_per_step": 4 * n,
            "d2h_bytes_per_step": 4 * k, "ms_per_step": t_pipe, "steps": steps,
            "serial": {"value": ws * n / (t_serial * 1e-3) / 1e9, "ms_per_step": t_serial,
                       "upload_build_ms": statistics.mean(t_up), "build_kernels_ms": statistics.mean(t_bld),
                       "sample_download_ms": statistics.mean(t_down), "steps": per_step},
            "host_link_gbs": link,
            "note": "wrs_table_build_host (H2D of the weights) + wrs_sample_host (D2H of the samples) per step; "
                    "two table objects and two streams, step i+1's upload and build issued before step i's "
                    "sampling; serial = one table, one step at a time"}


def run_ours(args, names):
    import torch

    ws, rank, local = dist_env()
    if ws > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl")
    torch.cuda.set_device(local)
    import __graft_entry__ as g

    if rank == 0 or ws == 1:
        g.build()
    if ws > 1:
        torch.distributed.barrier()
    from paper_1903_00227_gb300 import workloads as WL
    from paper_1903_00227_gb300 import wrs

    n, k = args.n, args.k
    stream = torch.cuda.current_stream()
    sh = stream.cuda_stream
    weights = {}
    for name in names:
        kind, s, seed = DISTS[name]
        weights[name] = WL.generate_device(kind, n, seed, s)
    table = wrs.AliasTable(n)
    table.set_timing(True)
    out = torch.empty(k, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()

    def step(i, record):
        name = names[i % len(names)]
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e2 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        table.build(weights[name], stream=sh)
        e1.record(stream)
        table.sample(k, seed=1000 + i, stream_id=0, out=out, stream=sh)
        e2.record(stream)
        e2.synchronize()
        if record:
            st = table.stage_ms()
            return name, e0.elapsed_time(e1), e1.elapsed_time(e2), st
        return None

    for i in range(args.warmup):
        step(i, False)
    if table.status() != wrs.OK:
        raise RuntimeError(f"build failed: {wrs.status_str(table.status())}")
    if ws > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    clocks = Clocks(local, enabled=(rank == 0 and not args.no_clocks))
    time.sleep(0.3)
    recs = [step(args.warmup + i, True) for i in range(args.steps)]
    torch.cuda.synchronize()
    clk = clocks.stop()
    if ws > 1:
        torch.distributed.barrier()
    status = table.status()
    if status != wrs.OK:
        raise RuntimeError(f"build failed in the timed region: {wrs.status_str(status)}")

    t_build = sum(r[1] for r in recs)
    t_sample = sum(r[2] for r in recs)
    step_ms = [r[1] + r[2] for r in recs]
    t_build, t_sample = reduce_max([t_build, t_sample], "cuda")
    K = args.steps
    value, sample_rate = job_rates(ws, K, n, k, t_build, t_sample)

    # per-kernel mean durations (events on the launching stream)
    stage_ms = {s: statistics.mean(r[3][s] for r in recs) for s in wrs.STAGES}
    stage_ms["sample"] = statistics.mean(r[2] for r in recs)
    peak, peak_kind = measured_peaks()
    units = {s: n for s in wrs.STAGES}
    units["sample"] = k
    dom = max(stage_ms, key=stage_ms.get)
    achieved = ALGO_BYTES[dom] * units[dom] / (stage_ms[dom] * 1e-3) / 1e9
    roofline = {"bound": "hbm", "kernel": KERNEL_NAMES[dom], "achieved": achieved, "peak": peak,
                "unit": "GB/s", "frac": achieved / peak, "traffic": traffic_for(dom, units[dom]),
                "peak_source": peak_kind, "algorithmic_bytes_per_unit": ALGO_BYTES[dom]}
    if roofline["traffic"]:  # DRAM bytes actually moved per launch (ncu) over the live duration
        dram = roofline["traffic"] / (stage_ms[dom] * 1e-3) / 1e9
        roofline["dram_achieved"] = dram
        roofline["dram_frac"] = dram / peak
    build_mean = t_build / K
    ach_build = BUILD_BYTES_PER_WEIGHT * n / (build_mean * 1e-3) / 1e9
    per_kernel = {KERNEL_NAMES[s]: {"ms": stage_ms[s],
                                    "gbs": (ALGO_BYTES[s] * units[s] / (stage_ms[s] * 1e-3) / 1e9)
                                    if ALGO_BYTES[s] else None} for s in stage_ms}
    per_dist = {}
    for name in names:
        rs = [r for r in recs if r[0] == name]
        if rs:
            bm = statistics.mean(r[1] for r in rs)
            sm_ = statistics.mean(r[2] for r in rs)
            per_dist[name] = {"build_ms": bm, "build_gweights_s": n / (bm * 1e-3) / 1e9,
                              "build_frac": BUILD_BYTES_PER_WEIGHT * n / (bm * 1e-3) / 1e9 / peak,
                              "sample_ms": sm_, "sample_gsamples_s": k / (sm_ * 1e-3) / 1e9}

    # practical ceiling of random 16-B bucket gathers from a table this size
    gather = None
    if k > 0:
        gt = []
        for i in range(4):
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            WL.random_gather(wrs.table_buckets(table.handle), n, k, 77 + i, out.data_ptr(), sh)
            e1.record(stream)
            e1.synchronize()
            if i:
                gt.append(e0.elapsed_time(e1))
        gms = statistics.mean(gt)
        gather = {"gsamples_s": k / (gms * 1e-3) / 1e9, "ms": gms,
                  "sampler_fraction": gms / (t_sample / K),
                  "note": "random 16-B gathers from the same table with no RNG or coin: the random-access ceiling"}

    small = None
    if not args.no_small:
        small = run_small(torch, WL, wrs, stream)

    # end to end through the C ABI with host buffers (copies inside the timed region)
    e2e = None
    if args.e2e_steps > 0:
        e2e = run_e2e(args, torch, wrs, table, weights, names, stream, ws)

    psa_plus = None
    if not args.no_psa_plus:
        psa_plus = run_psa_plus(args, torch, wrs, table, weights, names, stream, peak)

    two_level = None
    if not args.no_two_level:
        two_level = run_two_level(args, torch, wrs, weights, names, stream, peak)
        two_level["os_nd"] = run_os_nd(args, torch, wrs, weights, stream)

    batched = None
    if args.batch_tables > 0:
        batched = run_batched(args, torch, WL, wrs, stream)
    serving = None
    if args.serve_requests > 0:
        serving = run_serving(args, torch)

    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline(names, min(args.cpu_sample, n))
        rows = cpu_rows(names, min(args.cpu_sample // 4, n), args.batch_tables)
        for key, row in (("psa_plus", psa_plus), ("two_level", two_level), ("many_tables", batched)):
            if row is not None and key in rows:
                row["cpu_oracle"] = rows[key]
        if two_level is not None and two_level.get("os_nd") is not None and "os_nd" in rows:
            two_level["os_nd"]["cpu_oracle"] = rows["os_nd"]

    if rank == 0:
        srt = sorted(step_ms)
        p99 = srt[min(len(srt) - 1, int(round(0.99 * (len(srt) - 1))))]
        line = {
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": K, "warmup": args.warmup,
            "ms_per_step": statistics.mean(step_ms), "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "u128", "data": "synthetic", "config": config(args, names),
            "sample": {"value": sample_rate, "unit": "Gsamples/s", "ms": t_sample / K,
                       "random_gather_ceiling": gather,
                       "sector_roofline": {"bytes_per_sample": SECTOR_BYTES_PER_SAMPLE,
                                           "frac": sample_rate * SECTOR_BYTES_PER_SAMPLE / peak,
                                           "note": "one 32-B sector per random bucket + a 4-B coalesced store"}},
            "p99_ms": p99,
            "roofline": roofline,
            "roofline_build": {"bound": "hbm", "achieved": ach_build, "peak": peak, "unit": "GB/s",
                               "frac": ach_build / peak, "algorithmic_bytes_per_weight": BUILD_BYTES_PER_WEIGHT,
                               "peak_source": peak_kind},
            "kernels": per_kernel, "per_dist": per_dist,
            "e2e": e2e, "cpu_baseline": cpu, "clocks": clk, "psa_plus": psa_plus, "two_level": two_level,
            "many_tables": batched, "serving": serving, "small_exact": small,
            "gpu_launches": K * (len(wrs.STAGES) + 1),
            "context": {"paper_psa_build_gweights_s_n1e9": 0.99, "paper_psa_query_gsamples_s_n1e9": 1.662,
                        "paper_hardware": "4x Xeon Gold 6138, 158 threads (context only)"},
        }
        print(json.dumps(line), flush=True)
    table.free()
    if ws > 1:
        torch.distributed.destroy_process_group()
    return 0


def main():
    args = parse()
    names = [d for d in args.dists.split(",") if d]
    for d in names:
        if d not in DISTS:
            raise SystemExit(f"unknown distribution {d}")
    if args.impl == "reference":
        return run_reference(args, names)
    return run_ours(args, names)


if __name__ == "__main__":
    sys.exit(main())
