"""The work that users of this library have it do, as cases that can be timed.

Every case goes through the public binding (``paper_1903_00227_gb300.wrs``)
on weights that are on the device already, as a user's program holds them.
``call`` names the entry point; sizes come from the benchmark, the tests and
the serving workload, or are round (and deliberately unround) numbers between.

All outputs are whole numbers (thresholds, indices, counts), compared for
equality, so ``exact`` has no value to give.
"""
from __future__ import annotations

import math

import torch

from paper_1903_00227_gb300 import workloads as WL
from paper_1903_00227_gb300 import wrs


def listed():
    return [
        # The smallest served request: a distribution of one tile, built and
        # sampled a few hundred times (launches and latency).
        {"name": "request_small", "call": "table", "dist": "f32_zipf", "s": 1.0, "n": 1500, "k": 200, "skip": 0},
        # Integer weights, the small exact configuration of the benchmark:
        # 10^6 u32 weights built as 64 split pieces, 10^6 samples.
        {"name": "exact_u32_1m", "call": "table", "dist": "u32_uniform", "s": 0.0, "n": 1_000_000, "k": 1_000_000,
         "skip": 0, "splits": 64},
        # The headline builds: the paper's input shapes, 10^9 and 10^8
        # weights (the latter a ragged number of tiles).
        {"name": "build_uniform_1e9", "call": "build", "dist": "f32_uniform", "s": 0.0, "n": 1_000_000_000,
         "skip": 0},
        {"name": "build_zipf08_1e8", "call": "build", "dist": "f32_zipf", "s": 0.8, "n": 100_000_007, "skip": 0},
        {"name": "build_zipf15_1e9", "call": "build", "dist": "f32_zipf", "s": 1.5, "n": 1_000_000_000, "skip": 0},
        # Bulk sampling, the other half of the headline: as many samples as
        # buckets, from a 16 GB table.
        {"name": "sample_1e9", "call": "sample", "dist": "f32_uniform", "s": 0.0, "n": 1_000_000_000,
         "k": 1_000_000_000, "skip": 0},
        # Many samples from a table that stays on the chip (a vocabulary, the
        # edges of a small graph).
        {"name": "sample_resident", "call": "sample", "dist": "f32_zipf", "s": 1.0, "n": 300_007, "k": 100_000_000,
         "skip": 0},
        # The other two builders on a mid-sized input; two-level tables are
        # built and sampled.
        {"name": "psa_plus_1e8", "call": "psa_plus", "dist": "f32_uniform", "s": 0.0, "n": 100_000_000, "skip": 0},
        {"name": "two_level_1e8", "call": "two_level", "dist": "f32_zipf", "s": 0.8, "n": 100_000_000,
         "k": 30_000_000, "skip": 0},
        # The many-distributions workload of the benchmark: uneven tables,
        # built together and sampled together.
        {"name": "batch_4096", "call": "batch", "tables": 4096, "plan": 1, "n_lo": 32, "n_hi": 1 << 20,
         "k_hi": 4096},
        # A server's coalesced sample requests against resident tables.
        {"name": "served_requests", "call": "many", "tables": 64, "plan": 1, "n_lo": 1024, "n_hi": 1 << 21,
         "tasks": 1000, "k_hi": 100_000},
        # Output-sensitive sampling: the histogram of many draws from a
        # million items.
        {"name": "histogram_os", "call": "os", "dist": "f32_zipf", "s": 1.0, "n": 1_000_000, "k": 100_000_000,
         "skip": 0},
    ]


def _log(rng, lo, hi):
    return min(hi, max(lo, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))))


def draw(rng):
    call = rng.choice(["table", "table", "build", "build", "sample", "sample", "psa_plus", "two_level", "batch",
                       "many", "os"])
    if call == "batch":
        n_hi = _log(rng, 2048, 1 << 20)
        return {"call": call, "tables": _log(rng, 16, 4096), "plan": rng.randrange(1, 1000), "n_lo": 32, "n_hi": n_hi,
                "k_hi": _log(rng, 64, 4096)}
    if call == "many":
        return {"call": call, "tables": _log(rng, 4, 256), "plan": rng.randrange(1, 1000), "n_lo": 1024,
                "n_hi": _log(rng, 1 << 14, 1 << 21), "tasks": _log(rng, 16, 4000), "k_hi": _log(rng, 100, 100_000)}
    dist = rng.choice(["f32_uniform", "f32_zipf", "f32_zipf", "u32_uniform"])
    c = {"call": call, "dist": dist, "s": round(rng.uniform(0.5, 2.0), 2) if dist == "f32_zipf" else 0.0,
         # one array in four does not start on a 16-byte boundary: a slice of a larger one
         "skip": rng.choice([0, 0, 0, 1])}
    if call == "table":
        c.update(n=_log(rng, 1 << 10, 1 << 24), k=_log(rng, 1, 100_000))
    elif call == "build":
        c.update(n=_log(rng, 100_000, 1_000_000_000))
    elif call == "sample":
        c.update(n=_log(rng, 10_000, 1_000_000_000), k=_log(rng, 10_000, 1_000_000_000))
    elif call == "psa_plus":
        c.update(n=_log(rng, 100_000, 100_000_000))
    elif call == "two_level":
        c.update(n=_log(rng, 10_000, 100_000_000), k=_log(rng, 10_000, 100_000_000))
    else:
        c.update(n=_log(rng, 10_000, 10_000_000), k=_log(rng, 1_000_000, 100_000_000))
    return c


class _Buckets:
    """The library's bucket memory as a tensor of two 64-bit words per bucket
    (threshold; alias with a zero reserved word above it).  Keeps the owner."""

    def __init__(self, owner, ptr, n):
        self.owner = owner
        self.__cuda_array_interface__ = {"shape": (n, 2), "typestr": "<i8", "data": (ptr, False), "version": 3}


def _bucket_view(owner, ptr, n):
    return torch.as_tensor(_Buckets(owner, ptr, n), device="cuda")


def _weights(case, seed):
    skip = case["skip"]
    n = case["n"]
    dt = torch.int32 if case["dist"] == "u32_uniform" else torch.float32
    buf = torch.empty(n + skip, dtype=dt, device="cuda")
    w = buf[skip:]
    WL.generate_device(case["dist"], n, seed, case["s"], out=w)
    return w


def _plan_batch(case):
    """Sizes, sample counts and kinds of the batch's tables: the case's own,
    whatever the seed of their weights."""
    sizes, ks, kinds, _ = WL.batch_plan(case["tables"], case["plan"], n_lo=case["n_lo"], n_hi=case["n_hi"],
                                        k_hi=case["k_hi"])
    return sizes, ks, kinds


def _plan_many(case):
    """Table sizes, and per task its table (some are hot) and sample count."""
    sizes = WL.log_uniform_ints(case["tables"], case["n_lo"], case["n_hi"], case["plan"], 11)
    which = WL.log_uniform_ints(case["tasks"], 1, case["tables"], case["plan"], 12) - 1
    ks = WL.log_uniform_ints(case["tasks"], 1, case["k_hi"], case["plan"], 13)
    return [int(n) for n in sizes], [int(t) for t in which], [int(k) for k in ks]


def prepare(case, seed):
    call = case["call"]
    st = {"call": call, "seed": seed * 7919 + 2, "case": case}
    if call == "batch":
        sizes, ks, kinds = _plan_batch(case)
        b = wrs.AliasBatch(sizes)
        w = torch.zeros(b.offsets[-1], dtype=torch.float32, device="cuda")
        for t, (n, kind) in enumerate(zip(sizes, kinds)):
            WL.generate_device(kind, n, seed * 1_000_003 + t, 1.0, out=w[b.offsets[t]:b.offsets[t] + n])
        k_off = b.set_samples(ks)
        view = _bucket_view(b, wrs.batch_buckets(b.handle), b.offsets[-1])
        view.zero_()  # the gaps between tables hold no bucket: give them one value
        st.update(batch=b, w=w, view=view, out=torch.empty(max(k_off[-1], 1), dtype=torch.int32, device="cuda"))
        return st
    if call == "many":
        sizes, which, ks = _plan_many(case)
        tables = []
        for t, n in enumerate(sizes):
            tb = wrs.AliasTable(n)
            tb.build(WL.generate_device("f32_zipf", n, seed * 1009 + t, 1.0))
            tables.append(tb)
        tasks, off = [], 0
        for i, (t, k) in enumerate(zip(which, ks)):
            tb = tables[t]
            tasks.append([wrs.table_buckets(tb.handle), wrs.table_device_header(tb.handle), tb.n, k, seed * 31 + i,
                          i, off, 0])
            off += k
        st.update(tables=tables, tasks=torch.tensor(tasks, dtype=torch.int64, device="cuda"), ntasks=len(tasks),
                  total=off, out=torch.empty(off, dtype=torch.int32, device="cuda"))
        return st
    w = _weights(case, seed)
    st["w"] = w
    if call in ("two_level", "os"):
        t = wrs.AliasTable2(case["n"])
        st["table"] = t
        if call == "os":
            t.build(w)
        else:
            st["out"] = torch.empty(case["k"], dtype=torch.int32, device="cuda")
        return st
    t = wrs.AliasTable(case["n"])
    st["table"] = t
    if call == "sample":
        t.build(w)
        del st["w"]
    else:
        st["view"] = _bucket_view(t, wrs.table_buckets(t.handle), case["n"])
    if "k" in case:
        st["out"] = torch.empty(case["k"], dtype=torch.int32, device="cuda")
    return st


def run(state):
    call, case = state["call"], state["case"]
    if call == "batch":
        b = state["batch"]
        b.build(state["w"])
        return [state["view"], b.sample(state["seed"], out=state["out"])]
    if call == "many":
        rc = wrs.sample_many(state["tasks"].data_ptr(), state["ntasks"], state["total"], state["out"].data_ptr(),
                             torch.cuda.current_stream().cuda_stream)
        if rc != wrs.OK:
            raise RuntimeError(wrs.status_str(rc))
        return state["out"]
    t = state["table"]
    if call == "table":
        if case.get("splits"):
            t.build_opts(state["w"], splits=case["splits"])
        else:
            t.build(state["w"])
        return [state["view"], t.sample(case["k"], state["seed"], out=state["out"])]
    if call == "build":
        t.build(state["w"])
        return state["view"]
    if call == "sample":
        return t.sample(case["k"], state["seed"], out=state["out"])
    if call == "psa_plus":
        t.build_psa_plus(state["w"])
        return state["view"]
    if call == "two_level":
        t.build(state["w"])
        return t.sample(case["k"], state["seed"], out=state["out"])
    # "os": the pairs come in no particular order; the histogram they make is one value per item
    items, counts = t.sample_os(state["w"], case["k"], state["seed"])
    return torch.zeros(case["n"], dtype=torch.int64, device="cuda").index_add_(0, items, counts)


def work(case):
    """Bytes of one pass: weights read once, buckets (16 B) and samples (4 B)
    written once, and of a table that is only sampled the buckets that can be
    reached (16 B each, at most one per sample)."""
    call = case["call"]
    if call == "batch":
        sizes, ks, _ = _plan_batch(case)
        return {"bytes": 20 * sum(sizes) + 4 * sum(ks), "flops": 0}
    if call == "many":
        sizes, _, ks = _plan_many(case)
        return {"bytes": 4 * sum(ks) + 16 * min(sum(ks), sum(sizes)), "flops": 0}
    n, k = case["n"], case.get("k", 0)
    if call == "sample":
        return {"bytes": 16 * min(n, k) + 4 * k, "flops": 0}
    if call == "os":  # weights read, one count per item written
        return {"bytes": 4 * n + 8 * n, "flops": 0}
    return {"bytes": 20 * n + 4 * k, "flops": 0}
