"""Hole filling at the edges of k_post's rounds: 512 slots one per thread, then
four in a row per thread, from 8193 absorbed on with the list in global
memory; the check of the array order is test_gpu_compaction's.  GPU."""
import pytest

import test_gpu_compaction as order

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_dead,where", [
    (4000, 512, "spread"), (4000, 513, "spread"), (4000, 515, "last"), (4001, 516, "spread"),
    (6000, 2559, "spread"), (6000, 2560, "first"), (6001, 2561, "spread"), (6001, 2562, "last"),
    (3000, 2999, "spread"), (20000, 8193, "spread"), (30000, 9001, "first"),
    (30001, 20000, "spread"),
])
def test_hole_filling_rounds(n, n_dead, where):
    order.test_hole_filling_order(n, n_dead, where)
