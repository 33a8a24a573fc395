"""The packing code of the sweep, compiled by the host compiler and run warp by
warp (sweep_host.cpp): every bucket stored exactly once, none outside the
table, and the table of Alg. 2, in every key mode, tile size and task length."""
import ctypes

import numpy as np
import pytest

from oracle import wrs_oracle as O
from paper_1903_00227_gb300 import workloads as WL
from tests._host import host_library

U32_MAX = 0xFFFFFFFF


@pytest.fixture(scope="module")
def sweep(tmp_path_factory):
    f = host_library(tmp_path_factory.mktemp("sweep")).sweep_host
    f.argtypes = [ctypes.c_void_p, ctypes.c_uint64, ctypes.c_int, ctypes.c_uint32, ctypes.c_uint32, ctypes.c_int,
                  ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
    f.restype = ctypes.c_int
    return f


def _check(sweep, w, tile, group, wide):
    n = len(w)
    _, want = O.build_table(w)
    words = np.ascontiguousarray(w).view(np.uint32)
    tab = np.zeros((n, 4), np.uint32)
    status, failed = ctypes.c_uint32(), ctypes.c_uint64()
    assert sweep(words.ctypes.data, n, int(w.dtype == np.float32), tile, group, int(wide), tab.ctypes.data,
                 ctypes.byref(status), ctypes.byref(failed)) == 0
    assert failed.value == 0, f"{failed.value} buckets or aliases outside the table, or other failed checks"
    assert status.value == O.OK
    assert (tab[:, 3] == 1).all(), "a bucket was not stored exactly once"
    thr = tab[:, 0].astype(np.uint64) | (tab[:, 1].astype(np.uint64) << np.uint64(32))
    assert np.array_equal(thr, want.thr) and np.array_equal(tab[:, 2], want.alias)


@pytest.mark.parametrize("n", [2049, 4112, 4224, 5000])
@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("lower", [0, 1])
def test_largest_u32_words_stay_inside_the_table(sweep, n, wide, lower):
    """All words 0xFFFFFFFF (lower = 0): the light threshold is the largest
    word, so no fill word past the end can be told apart by its value.  With
    one word lower by one, all but that word are heavy."""
    w = np.full(n, U32_MAX, np.uint32)
    w[n // 2] -= lower
    for tile, group in ((2048, 1), (2048, 4), (256, 1), (256, 4)):
        _check(sweep, w, tile, group, wide)


def _giant(n):
    w = WL.f32_uniform(n, 3)
    w[n // 3] = 2.0 ** 9  # its q needs more than 32 bits, every light's does not
    return w


KINDS = {
    "u32": lambda n: WL.u32_uniform(n, 1),
    "equal": lambda n: np.full(n, 77, np.uint32),
    "few values": lambda n: np.random.default_rng(n).integers(0, 3, n).astype(np.uint32) + (np.arange(n) == 0),
    "uniform": lambda n: WL.f32_uniform(n, 2),
    "giant": _giant,
    "zipf2": lambda n: WL.f32_zipf(n, 2.0, 4),
    "long light runs": lambda n: np.where(np.arange(n) % 1500 == 7, 1000, 1).astype(np.float32),
    "subnormal": lambda n: (np.random.default_rng(n).integers(0, 1 << 20, n) * 2.0 ** -149).astype(np.float32),
    "powers": lambda n: np.exp2(np.random.default_rng(n).integers(0, 60, n)).astype(np.float32),
    "sorted": lambda n: np.sort(WL.f32_uniform(n, 5)),
}


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("n", [1, 127, 2049, 9001])
def test_sweep_on_the_host_matches_the_oracle(sweep, kind, n):
    w = KINDS[kind](n)
    if w.dtype != np.float32:
        w = w.astype(np.uint32)
    for tile, group, wide in ((2048, 4, False), (256, 1, False), (256, 3, True)):
        _check(sweep, w, tile, group, wide)
