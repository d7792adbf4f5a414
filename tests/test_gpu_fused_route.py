"""Which way the steps of small diodes run: the cases that compare the fused
kernel with the three kernels do reach it, in every cluster size, and none of
the forms that exclude it do.  GPU."""
import numpy as np
import pytest

from parity_util import mixed_state
from paper_2605_07083_gb300 import workloads as W
from test_gpu_fused import _diodes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pic():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07083_gb300 import build as B
    B.build()
    from paper_2605_07083_gb300 import pic
    return pic


def _run(pic, n_inst, kind, steps, **tune):
    ps, states = _diodes(n_inst, kind)
    d = pic.Diode(ps)
    if tune:
        d.tune(**tune)
    for i, st in enumerate(states):
        for sp in range(3):
            d.inject(sp, *st[sp], instance=i)
    d.step(steps)
    n = d.fused_steps()
    d.close()
    return n


# steps beyond a power-of-two graph of at least 8 run one by one
@pytest.mark.parametrize("n_inst,kind,steps,fused", [
    (1, "plain", 200, 200), (1, "empty", 70, 64), (1, "dense", 40, 40), (1, "hot", 12, 8),
    (20, "plain", 33, 32), (39, "dense", 9, 8), (39, "hot", 9, 8), (100, "plain", 17, 16),
    (100, "dense", 9, 8), (170, "plain", 9, 8), (1, "wide", 70, 64), (5, "wide", 40, 40),
    (100, "wide", 9, 8)])
def test_small_diodes_take_the_fused_kernel(pic, n_inst, kind, steps, fused):
    assert _run(pic, n_inst, kind, steps) == fused


@pytest.mark.parametrize("tune", [{"graph_steps": -1}, {"sort_period": 5},
                                  {"wait_polls": (1 << 20) + 1}])
def test_single_launches_sorts_and_own_wait_limits_take_the_three(pic, tune):
    assert _run(pic, 1, "plain", 64, **tune) == 0


def test_a_growing_diode_changes_over(pic):
    """125000 electrons and 300 more a step: the choice changes between two of
    the decisions (every 64 steps), and the particles are those of single
    launches."""
    p = W.single_diode_small(seed=77)
    p.update(gamma_emit=300.5 * p["weight"] / p["dt"], capacity=(1 << 19, 4096, 4096))
    state = mixed_state(p, 78, 125000, 1000)
    runs = []
    for graphs in (True, False):
        d = pic.Diode(p)
        if not graphs:
            d.tune(graph_steps=-1)
        for sp in range(3):
            d.inject(sp, *state[sp])
        d.step(700)
        runs.append(([d.state(sp) for sp in range(3)], d.rho_fixed(), d.fused_steps()))
        d.close()
    (sa, ra, fa), (sb, rb, fb) = runs
    assert 0 < fa < 640 and fa % 64 == 0 and fb == 0
    assert np.array_equal(ra, rb)
    for x, y in zip(sa, sb):
        for k in x:
            assert np.array_equal(x[k], y[k]), k


@pytest.mark.parametrize("n_pairs,pcand,fused", [(30000, 0.005, True), (60000, 0.02, False)])
def test_more_candidates_than_a_list_holds_take_the_three(pic, n_pairs, pcand, fused):
    """128 diodes, a block each: 300 candidates are in its list of 1024, 2400
    cost a second pass over its particles, which the three kernels do not need."""
    ps = []
    for i in range(128):
        p = W.single_diode_small(seed=200 + i)
        # n sigma g at the energy bound gives the electrons' probability
        g = np.sqrt(2 * 400.0 * W.E_CHARGE / W.M_E)
        p.update(window_start=1 << 40, E_cap_e_eV=400.0, E_cap_i_eV=400.0, gamma_emit=0.0,
                 n_gas=-np.log1p(-pcand) / (p["sigma_el_e"] * g * p["dt"]),
                 capacity=(1024, n_pairs + 4096, n_pairs + 4096))
        ps.append(p)
    state = mixed_state(ps[0], 5, 100, n_pairs)
    d = pic.Diode(ps)
    for i in range(128):
        for sp in range(3):
            d.inject(sp, *state[sp], instance=i)
    d.step(8)
    assert d.fused_steps() == (8 if fused else 0)
    d.close()


@pytest.mark.parametrize("ions,fused", [(20, 16), (4000, 8)])
def test_thousands_of_absorbed_particles_take_the_three(pic, ions, fused):
    """Hot ions that leave in every step and are replaced.  4000 of them keep
    the one warp that adds up their energies busy for longer than a step of the
    three kernels takes; how many there are is known from the first decision's
    last step on."""
    ps = []
    for i in range(76):
        p = W.single_diode_small(seed=40 + i)
        p.update(V=0.0, dt=1e-6, n_gas=0.0, T_e0_eV=0.0, T_i0_eV=100.0, weight=1e-12,
                 gamma_emit=0.0, replenish=1, window_start=1 << 40,
                 capacity=(32, 100000, ions + 32))
        ps.append(p)
    rng = np.random.default_rng(9)
    z = (rng.random(ions) * ps[0]["L"] * 0.999).astype(np.float32)
    v = [(rng.standard_normal(ions) * 5e4).astype(np.float32) for _ in range(3)]
    d = pic.Diode(ps)
    for i in range(76):
        d.inject(2, z, *v, instance=i)
    d.step(8)
    d.step(8)
    assert d.fused_steps() == fused
    d.close()
