"""pic_profile_steps counts every kernel it launches: three a step, one more
with the profile sampler, five for each sort (histogram, tile sums, prefix,
scatter, copy back).  Needs a GPU."""
import pytest

from parity_util import mixed_state
from paper_2605_07083_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sort,sampler", [(0, 0), (0, 3), (4, 0), (4, 3)])
def test_launches_of_profiled_steps(sort, sampler):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07083_gb300 import build as B
    B.build()
    from paper_2605_07083_gb300 import pic
    p = W.single_diode_small(seed=6)
    d = pic.Diode(p)
    d.inject(0, *mixed_state(p, 3, 2000, 10)[0])
    if sort:
        d.tune(sort_period=sort)
    if sampler:
        d.set_profile_period(sampler)
    prof = d.profile(10)
    assert prof["push_launches"] == 10
    assert prof["launches"] == 10 * (4 if sampler else 3) + 5 * (10 // sort if sort else 0)
    d.close()
