"""The build at the edges of its dispatch: one launch up to 2048 weights, tile
sizes (fine tiles up to 2^22 weights), the sweep's key modes, dense and sparse
heavies, long light runs, ragged ends, unaligned weights.  Tables are integers:
equal to the oracle's, bucket for bucket."""
import numpy as np
import pytest
import torch

from oracle import wrs_oracle as O
from paper_1903_00227_gb300 import workloads as WL
from paper_1903_00227_gb300 import wrs
from tests import _gpu as G

pytestmark = pytest.mark.gpu

FINE_MAX = 1 << 22


def _runs(n, rng):
    """Stretches of equal small weights, zeros, dense and sparse heavies."""
    w = np.ones(n, np.float32)
    w[n // 5: n // 3] = 0
    w[n // 3: n // 2] = rng.random(n // 2 - n // 3).astype(np.float32) * 4
    w[n // 2::700] = 900.0
    return w


CASES = {
    "u32": lambda n: WL.u32_uniform(n, 3),
    "uniform": lambda n: WL.f32_uniform(n, 4),
    "zipf0.8": lambda n: WL.f32_zipf(n, 0.8, 5),
    "zipf2": lambda n: WL.f32_zipf(n, 2.0, 6),                   # Q >= 2^64
    "runs": lambda n: _runs(n, np.random.default_rng(7)),
    "subnormal": lambda n: (np.random.default_rng(8).integers(0, 1 << 20, n) * 2.0 ** -149).astype(np.float32),
    "sorted": lambda n: np.sort(WL.f32_uniform(n, 9)),
}


@pytest.mark.parametrize("kind", CASES)
@pytest.mark.parametrize("n", [1, 257, 2047, 2048, 2049, FINE_MAX - 1, FINE_MAX, FINE_MAX + 1])
def test_sweep_matches_oracle(kind, n):
    w = CASES[kind](n)
    _, tab = O.build_table(w)
    buf = torch.zeros(n + 1, dtype=torch.float32 if w.dtype == np.float32 else torch.int32, device="cuda")
    with wrs.AliasTable(n + 5) as t:
        for skip in (0, 1):  # 16-byte aligned, and one word off
            buf[skip:skip + n].copy_(G.to_device(w))
            t.build(buf[skip:skip + n])
            assert t.status() == wrs.OK
            thr, alias, _ = t.download()
            assert np.array_equal(thr, tab.thr) and np.array_equal(alias, tab.alias)


@pytest.mark.parametrize("kind", ["narrow", "wide", "mixed", "u32"])
@pytest.mark.parametrize("n", [1, 2049, 3 * 2048, 40_007])
def test_psa_plus_and_groups_in_both_key_widths(kind, n):
    """Tiles and groups whose sums fit 64 bits stage their buckets, others
    store them at once; a table may hold both kinds."""
    if kind == "u32":
        w = WL.u32_uniform(n, 12)
    else:
        w = WL.f32_uniform(n, 11)
        if kind == "wide":  # n q up to 2^80
            w = (w * np.float32(2.0) ** np.random.default_rng(13).integers(-20, 20, n)).astype(np.float32)
        elif kind == "mixed":
            w[::5000] = 2.0 ** 40
    qz = O.quantize(w)
    tab, left = O.psa_plus(qz, 2048, return_left=True)
    with wrs.AliasTable(n) as t:
        t.build_psa_plus(G.to_device(w))
        assert t.status() == wrs.OK
        thr, alias, _ = t.download()
        assert np.array_equal(thr, tab.thr) and np.array_equal(alias, tab.alias)
    ref = O.build_2lvl(qz)
    with wrs.AliasTable2(n) as t2:
        t2.build(G.to_device(w))
        assert t2.status() == wrs.OK
        thr, alias, *_ = t2.download()
        assert np.array_equal(thr, ref.thr) and np.array_equal(alias, ref.alias)
