"""Whole steps of small diodes in one kernel (chosen on the device inside the
step graphs) against the three kernels launched one by one: array order,
charge, field, tallies (the FP64 energies too) bit for bit.  The diode counts
give clusters of 16 to 1 blocks; the cases reach partial quads, an empty
species, replenishment, ionisation, more candidates than a block lists, more
absorbed particles than a warp's lanes and than the staged list, and growth
past the point where the choice changes.  GPU."""
import numpy as np
import pytest

from parity_util import mixed_state
from paper_2605_07083_gb300 import workloads as W

pytestmark = pytest.mark.gpu

KEYS = ("z", "vx", "vy", "vz", "id")


def _diodes(n_inst, kind):
    ps, states = [], []
    for i in range(n_inst):
        p = W.single_diode_small(seed=300 + i)
        p.update(window_start=3, weight=p["weight"] * 8.0, capacity=(65536, 65536, 65536))
        n_emit, n_pairs = 900 + 37 * i % 500, 401
        if kind == "empty":
            n_emit = n_pairs = 0
        elif kind == "dense":              # ionisation and replenishment, many candidates
            p.update(n_gas=2e23, dt=2e-12, V=40.0, replenish=1, E_cap_e_eV=400.0,
                     E_cap_i_eV=400.0)
            n_emit = 9000
        elif kind == "hot":                # most particles leave within a few steps
            p.update(n_gas=0.0, T_e0_eV=1e5, dt=1e-11, replenish=1, Nz=127 + i)
            n_emit, n_pairs = 700, 9000
        elif kind == "wide":               # more cells than one warp solves for
            p.update(Nz=(600, 1999, 513)[i % 3], dt=2e-13)
        elif kind == "emission":           # 3000 electrons a step: outgrows the choice
            p.update(gamma_emit=p["gamma_emit"] * 1000.0, capacity=(1 << 18, 65536, 65536))
        ps.append(p)
        empty = {sp: [np.zeros(0, np.float32)] * 4 for sp in range(3)}
        states.append(mixed_state(p, 500 + i, n_emit, n_pairs) if n_emit else empty)
    return ps, states


@pytest.mark.parametrize("n_inst,kind,steps", [
    (1, "plain", 200), (1, "empty", 70), (1, "dense", 40), (1, "hot", 12), (1, "emission", 130),
    (20, "plain", 33), (39, "dense", 9), (39, "hot", 9), (100, "plain", 17), (100, "dense", 9),
    (170, "plain", 9), (1, "wide", 70), (5, "wide", 40), (100, "wide", 9),
])
def test_fused_steps_match_the_three_kernels(n_inst, kind, steps):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07083_gb300 import build as B
    B.build()
    from paper_2605_07083_gb300 import pic
    ps, states = _diodes(n_inst, kind)
    runs = []
    for graphs in (True, False):
        d = pic.Diode(ps)
        if not graphs:
            d.tune(graph_steps=-1)
        for i, st in enumerate(states):
            for sp in range(3):
                d.inject(sp, *st[sp], instance=i)
        d.step(steps)
        d.step(3)
        runs.append([([d.state(sp, instance=i) for sp in range(3)], d.rho_fixed(i), d.field(i),
                      d.diagnostics(i)) for i in range(0, n_inst, max(1, n_inst // 8))])
        d.close()
    absorbed = 0
    for a, b in zip(*runs):
        for sp in range(3):
            for k in KEYS:
                assert np.array_equal(a[0][sp][k], b[0][sp][k]), (sp, k)
        assert np.array_equal(a[1], b[1])
        assert np.array_equal(a[2][0], b[2][0]) and np.array_equal(a[2][1], b[2][1])
        for k in a[3]:
            assert np.array_equal(np.asarray(a[3][k]), np.asarray(b[3][k]), equal_nan=True), k
        absorbed += int(a[3]["count"].sum())
    assert absorbed > 0 or kind == "empty"
