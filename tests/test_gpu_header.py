"""The public header's f32 word: 1 for binary32 weights, 0 for u32, whatever
key width the sweep chose (wrs_device_header of include/wrs.h)."""
import numpy as np
import pytest
import torch

from oracle import wrs_oracle as O
from paper_1903_00227_gb300 import workloads as WL
from paper_1903_00227_gb300 import wrs
from tests import _gpu as G

pytestmark = pytest.mark.gpu

F32_WORD = 11  # status, tile_counter, beta, shift, Q (4 words), qp (2), light_max, f32


def _giant(n):
    w = WL.f32_uniform(n, 3)
    w[n // 3] = 2.0 ** 9  # the light words' units fit 32 bits, this one's do not
    return w


@pytest.mark.parametrize("kind", ["u32", "uniform", "giant", "zipf2"])
@pytest.mark.parametrize("n", [1500, 5000, 70_001])
def test_header_says_binary32_or_not(kind, n):
    w = {"u32": lambda: WL.u32_uniform(n, 1), "uniform": lambda: WL.f32_uniform(n, 2), "giant": lambda: _giant(n),
         "zipf2": lambda: WL.f32_zipf(n, 2.0, 4)}[kind]()
    _, tab = O.build_table(w)
    dtype = wrs.F32 if w.dtype == np.float32 else wrs.U32
    w_dev = G.to_device(w)
    buckets = torch.zeros(n * 4, dtype=torch.int32, device="cuda")
    header = torch.zeros(wrs.DEVICE_HEADER_BYTES // 4, dtype=torch.int32, device="cuda")
    assert wrs.build_noalloc(w_dev.data_ptr(), n, dtype, buckets.data_ptr(), header.data_ptr(),
                             torch.cuda.current_stream().cuda_stream) == wrs.OK
    torch.cuda.synchronize()
    words = buckets.cpu().numpy().view(np.uint32).reshape(n, 4)
    thr = words[:, 0].astype(np.uint64) | (words[:, 1].astype(np.uint64) << np.uint64(32))
    assert np.array_equal(thr, tab.thr) and np.array_equal(words[:, 2], tab.alias)
    assert int(header[0]) == wrs.OK
    assert int(header[F32_WORD]) == (1 if dtype == wrs.F32 else 0)
