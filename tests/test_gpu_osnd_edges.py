"""OS-ND where its passes meet: groups of one and two members, ragged trees,
counts around the switch between inversion and rejection (c p = 10)."""
import numpy as np
import pytest

from paper_1903_00227_gb300 import workloads as WL
from tests.test_gpu_osnd import _run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 2049, 2050, 4095])
def test_osnd_small_and_ragged_groups(n):
    _run(WL.f32_zipf(n, 1.0, n), [1, 300, 10 * n, 25 * n, 10 ** 7])


def test_osnd_zero_weights_and_lopsided_nodes():
    w = WL.f32_uniform(6000, 4)
    w[::2] = 0
    w[1::64] = 2.0 ** -20
    w[5] = 4096.0
    _run(w.astype(np.float32), [129, 60_000, 10 ** 8])
