"""The tuner keeps a grouping that the sweep runs: at most four tiles a warp."""
import pytest
import torch

from paper_1903_00227_gb300 import workloads as WL
from paper_1903_00227_gb300 import wrs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[200_000, 50_000, 9000, 4000, 100, 1_000_000], [5_000_000, 300_000, 60_000, 7000]])
def test_tuned_groups_are_groups_that_run(sizes):
    with wrs.AliasBatch(sizes) as b:
        w = b.pack([torch.from_numpy(WL.f32_uniform(n, t)).cuda() for t, n in enumerate(sizes)])
        for _ in range(6):  # equal times decide between groups that are one launch: try more than once
            b.tune(w)
            assert all(g in (1, 2, 4) for g in b.groups())
