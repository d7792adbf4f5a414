"""The deposit that bins a warp's particles cell by cell (a state kept sorted)
against the one atomic per particle: the same charge and particles to the last
bit, for warps that span one cell up to more than the bins hold, with particles
absorbed and a last warp that is partly idle.  Needs a GPU."""
import numpy as np
import pytest

from paper_2605_07083_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _state(p, n, span, seed):
    """n particles in array order; each run of 128 lies in `span` cells, at
    nodes, just below them and between; the first run is about to be lost."""
    rng = np.random.default_rng(seed)
    dz = p["L"] / p["Nz"]
    i = np.arange(n)
    cell = (i // 128) * 3 % (p["Nz"] - span) + (i * 37) % 128 * span // 128
    frac = np.choose(i % 3, [np.zeros(n), np.full(n, 1.0 - 1e-6), rng.random(n)])
    z = np.float32((cell + frac) * dz)
    v = [rng.normal(0.0, 1e4, n).astype(np.float32) for _ in range(3)]
    v[2][:100] = np.float32(-3e6)
    z = np.clip(z, 0, np.nextafter(np.float32(p["L"]), np.float32(0)))
    return z, v[0], v[1], v[2]


@pytest.mark.parametrize("span", [1, 2, 4, 5, 8, 9, 40])
@pytest.mark.parametrize("n", [127, 8195])
def test_binned_deposit_is_the_plain_one(n, span):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07083_gb300 import build as B
    B.build()
    from paper_2605_07083_gb300 import pic
    p = W.single_diode_small(seed=5)
    out = []
    for period in (0, 100000):              # the sort itself never falls due
        d = pic.Diode(p)
        if period:
            d.tune(sort_period=period)
        for sp in range(3):
            d.inject(sp, *_state(p, n, span, 20 + sp))
        got = [d.rho_fixed()]
        for _ in range(4):
            d.step(1)
            got.append(d.rho_fixed())
        for sp in range(3):
            s = d.state(sp)
            got += [s[k] for k in sorted(s)]
        out.append(got)
        d.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
