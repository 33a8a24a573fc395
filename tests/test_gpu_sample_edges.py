"""The sampler's dispatch (tables in the L2 or beyond) and the search for a
block's first task among many: equal to the oracle, index for index."""
import numpy as np
import pytest
import torch

from oracle import wrs_oracle as O
from paper_1903_00227_gb300 import workloads as WL
from paper_1903_00227_gb300 import wrs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, (1 << 22) - 1, 1 << 22, (1 << 22) + 1])
def test_sample_on_both_sides_of_the_small_table_limit(n):
    with wrs.AliasTable(n) as t:
        t.build(WL.generate_device("f32_zipf", n, 3, 1.0))
        thr, alias, _ = t.download()
        qp = t.info().qp
        for k in (1, 1023, 1024, 5_000_001):
            got = t.sample(k, 2 ** 62 + 1, 2 ** 40).cpu().numpy().view(np.uint32)
            assert np.array_equal(got, O.sample(thr, alias, qp, k, 2 ** 62 + 1, 2 ** 40))


@pytest.mark.parametrize("ntasks", [1, 2, 31, 32, 33, 34, 1000, 1025, 1057])
def test_many_tasks_find_their_blocks(ntasks):
    rng = np.random.default_rng(ntasks)
    ks = rng.choice([0, 0, 1, 7, 4095, 4096, 4097, 9000], ntasks)
    ks[-1] = 3
    n = 5000
    with wrs.AliasTable(n) as t:
        t.build(WL.generate_device("f32_zipf", n, 3, 1.0))
        thr, alias, _ = t.download()
        qp = t.info().qp
        off = np.concatenate([[0], np.cumsum(ks)])
        head = [wrs.table_buckets(t.handle), wrs.table_device_header(t.handle), n]
        tasks = torch.tensor([head + [int(k), 11 + i, i, int(o), 0] for i, (k, o) in enumerate(zip(ks, off))],
                             dtype=torch.int64, device="cuda")
        out = torch.full((int(off[-1]),), -1, dtype=torch.int32, device="cuda")
        assert wrs.sample_many(tasks.data_ptr(), ntasks, int(off[-1]), out.data_ptr(),
                               torch.cuda.current_stream().cuda_stream) == wrs.OK
        got = out.cpu().numpy().view(np.uint32)
    for i, k in enumerate(ks):
        if k:
            assert np.array_equal(got[off[i]:off[i + 1]], O.sample(thr, alias, qp, int(k), 11 + i, i)), i
