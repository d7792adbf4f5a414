"""The two ways k_mid takes its collision candidates give the same state: a
batch whose expected candidates per step select the one for many (records
with the particle, constants in shared memory up to 64 diodes, from global
memory beyond) against the same diodes on handles of their own, which expect
few.  Bit for bit: draws are keyed by particle and step.  GPU."""
import numpy as np
import pytest

from parity_util import by_id, mixed_state
from paper_2605_07083_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_inst,capacity", [(2, 131072), (64, 4096), (65, 4096)])
def test_many_candidates_match_few(n_inst, capacity):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07083_gb300 import build as B
    B.build()
    from paper_2605_07083_gb300 import pic
    ps = []
    for i in range(n_inst):
        p = W.single_diode_small(seed=70 + i)
        # 0.3 to 0.6 candidates per particle and step; ionisation on; an ion
        # lost now and then is replenished
        p.update(n_gas=2e23, dt=2e-12, replenish=1, window_start=1 + i % 2, V=40.0,
                 E_cap_e_eV=400.0, E_cap_i_eV=400.0, weight=p["weight"] * 40.0,
                 capacity=(capacity,) * 3, T_e0_eV=30.0)
        ps.append(p)
    states = [mixed_state(p, 80 + i, 700 + 13 * i, 500) for i, p in enumerate(ps)]
    both = pic.Diode(ps)
    for i, st in enumerate(states):
        for sp in range(3):
            both.inject(sp, *st[sp], instance=i)
    both.step(5)
    collisions = 0
    for i in range(0, n_inst, max(1, n_inst // 6)):
        d = pic.Diode(ps[i])
        for sp in range(3):
            d.inject(sp, *states[i][sp])
        d.step(5)
        assert np.array_equal(both.rho_fixed(i), d.rho_fixed())
        for sp in range(3):
            a, b = by_id(both.state(sp, instance=i)), by_id(d.state(sp))
            for k in a:
                assert np.array_equal(a[k], b[k]), (i, sp, k)
        da, db = both.diagnostics(i), d.diagnostics()
        for k in ("count", "collisions", "candidates", "emitted", "replenished"):
            assert np.array_equal(da[k], db[k]), (i, k)
        collisions += int(da["collisions"][1:].sum())
        d.close()
    assert collisions > 100            # the case really exercises the collisions
    both.close()
