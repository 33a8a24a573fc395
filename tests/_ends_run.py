"""Tables of the largest u32 words: the light threshold is 0xFFFFFFFF itself,
so a word past the end cannot be told from a light one by its value.  Nothing
may be stored past the last bucket: single tables of capacity n (the header
lies behind the buckets), batches (the next table lies there), and the
allocation-free build into the front of a larger buffer.

Used by tests/test_gpu_ends.py; run as ``WRS_CHECK=1 python -m tests._ends_run``
the same cases go through libwrs_check.so, which counts every bucket store.
"""
import sys

import numpy as np
import torch

from oracle import wrs_oracle as O
from paper_1903_00227_gb300 import workloads as WL
from paper_1903_00227_gb300 import wrs
from tests import _gpu as G

SIZES = [2049, 4112, 4224, 5000, (1 << 22) + 1, (1 << 22) + 77]
RESERVED = wrs.check_build()  # what a bucket stored once has in its reserved word
PATTERN = 0x5A5A5A5A


def largest(n, lower=0):
    """n words 0xFFFFFFFF; with lower = 1 one of them is 0xFFFFFFFE."""
    w = np.full(n, 0xFFFFFFFF, np.uint32)
    w[n // 2] -= lower
    return w


def _same(got, w, what):
    thr, alias, res = got
    _, tab = O.build_table(w)
    assert np.array_equal(thr, tab.thr) and np.array_equal(alias, tab.alias), what
    assert (res == RESERVED).all(), what


def single(n, lower):
    w = largest(n, lower)
    with wrs.AliasTable(n) as t:
        for acc in (wrs.ACC_AUTO, wrs.ACC_U128):
            t.build_opts(G.to_device(w), acc=acc)
            assert t.status() == wrs.OK, (n, acc)
            assert t.check_failures() == 0, (n, acc)
            info = t.info()
            assert info.n == n and info.Q == int(w.sum(dtype=np.uint64)) and info.status == wrs.OK
            _same(t.download(), w, (n, acc))


def batch(total_above_fine):
    sizes = [2049, 3000, 5000, 4112, 100, 4112] + ([(1 << 22) + 5, 2049] if total_above_fine else [])
    ws = [WL.u32_uniform(n, t) if t % 2 else largest(n) for t, n in enumerate(sizes)]
    with wrs.AliasBatch(sizes) as b:
        packed = b.pack([G.to_device(w) for w in ws])
        for _ in range(3):
            b.build(packed)
            rc, st = b.status()
            assert rc == wrs.OK, st
            got = b.download()
            for t, w in enumerate(ws):
                lo = b.offsets[t]
                _same([a[lo:lo + len(w)] for a in got], w, (t, len(w)))


def noalloc(n):
    w = largest(n)
    w_dev = G.to_device(w)
    buckets = torch.full(((n + 256) * 4,), PATTERN, dtype=torch.int32, device="cuda")
    header = torch.zeros(wrs.DEVICE_HEADER_BYTES // 4, dtype=torch.int32, device="cuda")
    rc = wrs.build_noalloc(w_dev.data_ptr(), n, wrs.U32, buckets.data_ptr(), header.data_ptr(),
                           torch.cuda.current_stream().cuda_stream)
    assert rc == wrs.OK
    torch.cuda.synchronize()
    assert int(header[0]) == wrs.OK
    words = buckets.cpu().numpy().view(np.uint32).reshape(-1, 4)
    assert (words[n:] == PATTERN).all(), "stored behind the caller's buckets"
    thr = words[:n, 0].astype(np.uint64) | (words[:n, 1].astype(np.uint64) << np.uint64(32))
    _same((thr, words[:n, 2], words[:n, 3]), w, n)


def main():
    assert wrs.check_build() == 1, "the binding did not load libwrs_check.so (set WRS_CHECK=1)"
    for n in SIZES:
        for lower in (0, 1):
            single(n, lower)
    for above in (False, True):
        batch(above)
    for n in SIZES[:4]:
        noalloc(n)
    print("largest words: all cases passed", flush=True)


if __name__ == "__main__":
    sys.exit(main())
