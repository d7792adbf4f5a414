"""Sampled steps that run outside the step graphs (a period of at least 16
steps per distinct sampling phase) against the sampler after every step: the
same sums, samples and particles to the last bit.  Needs a GPU."""
import numpy as np
import pytest

from parity_util import mixed_state
from paper_2605_07083_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pic():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07083_gb300 import build as B
    B.build()
    from paper_2605_07083_gb300 import pic
    pic.load()
    return pic


def _params(window_start, seed=3):
    p = W.single_diode_small(seed=seed)
    p.update(window_start=window_start, n_gas=3e22)
    return p


@pytest.mark.parametrize("sort", [0, 8])
@pytest.mark.parametrize("period,window", [(16, 0), (17, 5), (31, 64), (100, 101), (5000, 3)])
def test_split_samples_are_those_of_every_step(pic, period, window, sort):
    st = mixed_state(_params(0), 11, 5003, 2001)
    total, runs = 203, []
    # one diode: one phase, sampled steps by themselves.  With diodes of other
    # phases beside it (enough that the period has fewer than 16 steps per
    # phase) the sampler follows every step.
    phases = period // 16 + 1
    for n in (1, phases if phases <= 4 else 1):
        ps = [_params(window + i, seed=3 + i) for i in range(n)]
        d = pic.Diode(ps if n > 1 else ps[0])
        for i in range(n):
            for sp in range(3):
                d.inject(sp, *st[sp], instance=i)
        if sort:
            d.tune(sort_period=sort)
        d.set_profile_period(period)
        if not runs:
            for k in (1, 90, 17, 95):           # 203 in calls that end anywhere
                d.step(k)
        else:
            for _ in range(total):
                d.step(1)
        runs.append((d.profiles(0) if window < total else None, [d.state(sp, 0) for sp in range(3)]))
        d.close()
    (pa, sa), (pb, sb) = runs
    assert pa["samples"] == pb["samples"] == len(range(window, total, period))
    assert np.array_equal(pa["counts"], pb["counts"]) and np.array_equal(pa["phi"], pb["phi"])
    for x, y in zip(sa, sb):
        for k in x:
            assert np.array_equal(x[k], y[k]), k
