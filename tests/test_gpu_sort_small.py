"""Sorts of up to one chunk, which the scatter does alone, and the first sizes
past it; the check is test_gpu_sort's.  GPU."""
import pytest

import test_gpu_sort as whole

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,cells,order", [
    (2, 4096, "reversed"), (33, 1, "random"), (100, 128, "random"), (1023, 2048, "sorted"),
    (2047, 2049, "random"), (2048, 2048, "random"), (2048, 4096, "reversed"),
    (2048, 7, "one_cell"), (2049, 128, "random"), (4097, 4096, "random"),
])
def test_static_sort_of_one_chunk(n, cells, order):
    whole.test_static_sort_is_a_stable_argsort(n, cells, order)
