"""u32 tables of the largest words, where a word past the end would count as
light: no bucket is stored outside the table (see _ends_run.py)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("lower", [0, 1])
@pytest.mark.parametrize("n", [2049, 4112, 4224, 5000, (1 << 22) + 1, (1 << 22) + 77])
def test_single_table_of_capacity_n(n, lower):
    from tests import _ends_run as E

    E.single(n, lower)


@pytest.mark.parametrize("total_above_fine", [False, True])
def test_batch_beside_other_tables(total_above_fine):
    from tests import _ends_run as E

    E.batch(total_above_fine)


@pytest.mark.parametrize("n", [2049, 4112, 4224, 5000])
def test_noalloc_leaves_the_callers_memory_alone(n):
    from tests import _ends_run as E

    E.noalloc(n)


def test_check_build_counts_each_bucket_once():
    r = subprocess.run([sys.executable, "-m", "tests._ends_run"], cwd=ROOT, env=dict(os.environ, WRS_CHECK="1"),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    assert "all cases passed" in r.stdout
