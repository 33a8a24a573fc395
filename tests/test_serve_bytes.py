"""The serving budget counts what a table's allocation takes: never less, and
at most one percent and the fixed part's rounding more."""
import ctypes

from paper_1903_00227_gb300 import serve as S
from tests._host import host_library


def test_table_bytes_covers_the_allocation(tmp_path):
    f = host_library(tmp_path).table_bytes_host
    f.argtypes, f.restype = [ctypes.c_uint64], ctypes.c_uint64
    caps = [1 << c for c in range(10, 32)] + [1, 255, 257, 2049, 100_003, (1 << 22) - 1, (1 << 22) + 1, 5_000_001,
                                              10 ** 9, 4_000_000_019]
    for cap in caps:
        need, got = f(cap), S.table_bytes(cap)
        assert need <= got <= need + need // 100 + (4 << 10), (cap, need, got)
