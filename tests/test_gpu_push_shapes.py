"""The push kernel in every shape, a few and many collision candidates: the
partition of the particles over blocks, warps and chunks changes no bit of the
particles, charge and tallies.  Single launches, so that no step runs in the
fused kernel of small diodes.  GPU.

Many candidates: a probability of 2 % of room for 3 x 2^21 particles, above one
per thread of a block per SM, selects the kernels whose candidate records carry
the particle; 0.5 % do not.  4096 cells leave 64-quad chunks room for one wide
block per SM, the default for that room as long as the live counts are not
known before a step: the particles come after a first, empty step.  A chosen
size or chunk selects the others."""
import numpy as np
import pytest

from parity_util import mixed_state
from paper_2605_07083_gb300 import workloads as W

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


@pytest.mark.parametrize("cells,many", [(128, False), (128, True), (2048, True), (4096, False),
                                        (4096, True)])
def test_results_do_not_depend_on_the_push_shape(pic, cells, many):
    p = W.single_diode_small(seed=61) if cells == 128 else W.single_diode_production(seed=62)
    # the probability at the energy bound, of electrons
    g = np.sqrt(2 * p["E_cap_e_eV"] * W.E_CHARGE / W.M_E)
    prob = 0.02 if many else 0.005
    p.update(Nz=cells, replenish=1, window_start=2,
             n_gas=-np.log1p(-prob) / (p["sigma_el_e"] * g * p["dt"]),
             capacity=(1 << 21,) * 3)
    st = mixed_state(p, 63, 30001, 10003)
    shapes = [{}, {"push_threads": 128}, {"push_threads": 320}, {"push_chunk": 32},
              {"push_threads": 160, "push_chunk": 32}, {"push_blocks_per_sm": 1}]
    runs = []
    for shape in shapes:
        d = pic.Diode(p)
        d.tune(graph_steps=-1, **shape)
        d.step(1)
        for sp in range(3):
            d.inject(sp, *st[sp])
        d.step(12)
        runs.append(([d.state(sp) for sp in range(3)], d.rho_fixed(), d.diagnostics()))
        d.close()
    sa, ra, da = runs[0]
    assert da["candidates"].sum() > 1000 and da["count"].sum() > 0
    for (sb, rb, db), shape in zip(runs[1:], shapes[1:]):
        assert np.array_equal(ra, rb), shape
        for x, y in zip(sa, sb):
            for k in x:
                assert np.array_equal(x[k], y[k]), (shape, k)
        for k in ("count", "ke", "collisions", "candidates", "emitted", "replenished"):
            assert np.array_equal(da[k], db[k]), (shape, k)


@pytest.mark.parametrize("shift,skip", [(0, ()), (1, ()), (3, ("vx",)), (0, ("z", "id")),
                                        (2, ("vx", "vy", "vz", "id"))])
def test_state_into_unaligned_and_missing_arrays(pic, shift, skip):
    """pic_get_state into device arrays off the 16-byte boundaries, and with
    some of them null: the host's copy of the same state, and nothing beyond."""
    import ctypes as C

    import torch
    p = W.single_diode_small(seed=64)
    d = pic.Diode(p)
    for sp, s in mixed_state(p, 65, 5003, 1001).items():
        d.inject(sp, *s)
    want = d.state(0)
    n = want["z"].size
    keys = ("z", "vx", "vy", "vz", "id")
    out = {k: torch.full((n + 8,), 77, device="cuda",
                         dtype=torch.int32 if k == "id" else torch.float32) for k in keys}
    torch.cuda.synchronize()
    ptrs = [None if k in skip else C.c_void_p(out[k].data_ptr() + 4 * shift) for k in keys]
    live = C.c_int64()
    assert pic.load().pic_get_state(d.handle, 0, 0, *ptrs, n, C.byref(live), 1) == 0
    assert live.value == n
    for k in keys:
        got = out[k].cpu().numpy()
        assert (np.concatenate([got[:shift], got[shift + n:]]) == 77).all(), k
        if k in skip:
            assert (got == 77).all(), k
        else:
            assert np.array_equal(got[shift:shift + n].view(want[k].dtype), want[k]), k
    d.close()
