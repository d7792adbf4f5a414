"""A diode that replenishment makes outgrow the 32-bit histograms of a block
while the fused kernel runs its steps: the charge, counts and particles of the
three kernels launched one by one, to the last bit.  GPU.

36000 hot ions of one diode leave in every step and come back as pairs whose
cold electrons stay: 2.3M electrons after 64 steps.  140 diodes give a block per
diode and one cell all of them (the sum of the fractions' high parts would pass
2^32 at 2.1M); 76 diodes give two blocks, each past 2^20 particles at the end."""
import numpy as np
import pytest

from paper_2605_07083_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_inst,cells", [(140, 1), (76, 3)])
def test_growth_by_replenishment_keeps_the_charge_exact(n_inst, cells):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07083_gb300 import build as B
    B.build()
    from paper_2605_07083_gb300 import pic
    ions, steps = 36000, 64
    ps = []
    for i in range(n_inst):
        p = W.single_diode_small(seed=40 + i)
        p.update(Nz=cells, V=0.0, dt=1e-6, n_gas=0.0, T_wall_K=0.0, T_e0_eV=0.0, T_i0_eV=100.0,
                 weight=1e-12, gamma_emit=0.0, replenish=1, window_start=3,
                 capacity=(32, 32, 32))
        ps.append(p)
    ps[0].update(gamma_emit=100.5 * ps[0]["weight"] / ps[0]["dt"],
                 capacity=(8192, 2600000, ions + 32))
    rng = np.random.default_rng(9)
    z = (rng.random(ions) * ps[0]["L"] * 0.999).astype(np.float32)
    v = [(rng.standard_normal(ions) * 5e4).astype(np.float32) for _ in range(3)]
    runs = []
    for graphs in (True, False):
        d = pic.Diode(ps)
        if not graphs:
            d.tune(graph_steps=-1)
        d.inject(2, z, *v)
        d.step(steps)
        rho = d.rho_fixed(0)
        d.step(1)
        runs.append((rho, d.rho_fixed(0), [d.state(sp) for sp in range(3)], d.diagnostics(0)))
        d.close()
    a, b = runs
    n = a[3]["n_live"]
    assert n[1] > (1 << 21) + 100000 and n[0] >= 100
    assert np.array_equal(a[0], b[0]) and np.array_equal(a[1], b[1])
    assert a[1].sum() == (n[2] - n[0] - n[1]) * (1 << 24)
    for x, y in zip(a[2], b[2]):
        for k in x:
            assert np.array_equal(x[k], y[k]), k
    for k in a[3]:
        assert np.array_equal(np.asarray(a[3][k]), np.asarray(b[3][k]), equal_nan=True), k
