"""Hole filling of the absorbed slots: the array order after a step in which a
given set of particles leaves, against the rule on the host (the live tail
slots move, in order, into the dead slots below the new count).  Exact.  GPU."""
import numpy as np
import pytest

from paper_2605_07083_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,n_dead,where", [
    (5, 1, "last"), (5, 5, "all"), (4000, 3, "spread"), (4000, 513, "first"),
    (4000, 700, "last"), (12000, 6000, "spread"), (12000, 11990, "spread"), (12000, 12000, "all"),
])
def test_hole_filling_order(n, n_dead, where):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07083_gb300 import build as B
    B.build()
    from paper_2605_07083_gb300 import pic
    rng = np.random.default_rng(n + n_dead)
    dead = {"last": np.arange(n - n_dead, n), "first": np.arange(n_dead), "all": np.arange(n),
            "spread": np.sort(rng.choice(n, n_dead, replace=False))}[where]
    p = W.single_diode_small()
    p.update(n_gas=0.0, gamma_emit=0.0, V=0.0, replenish=0, weight=1.0)
    z = (rng.uniform(0.2, 0.8, n) * p["L"]).astype(np.float32)
    vz = np.zeros(n, np.float32)
    vz[dead] = np.float32(2.0 * p["L"] / p["dt"]) * np.where(rng.random(dead.size) < 0.5, -1, 1)
    vx = rng.standard_normal(n).astype(np.float32)
    d = pic.Diode(p)
    d.inject(1, z, vx, -vx, vz)
    d.step(1)
    got = d.state(1)
    d.close()
    slots = np.arange(n)
    alive = np.ones(n, bool)
    alive[dead] = False
    new = n - n_dead
    order = slots[:new].copy()
    order[~alive[:new]] = slots[new:][alive[new:]]
    assert np.array_equal(got["id"], order.astype(np.uint32))
    assert np.array_equal(got["vx"], vx[order]) and np.array_equal(got["vy"], -vx[order])
