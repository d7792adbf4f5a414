"""Tensors that the binding makes on the current stream and the library uses on
the handle's.  GPU."""
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


@pytest.mark.parametrize("form", ["double", "strided"])
def test_converted_arrays_are_complete_when_they_are_read(pic, form):
    """FP64 or strided tensors are converted on the current stream, here behind
    50 ms of other work; the handle's stream must not read them before."""
    import torch
    p = W.single_diode_small(seed=70)
    state = mixed_state(p, 71, 4001, 10)[0]
    d = pic.Diode(p)
    if form == "double":
        arrays = [torch.from_numpy(a).cuda().double() for a in state]
    else:
        arrays = [torch.stack([torch.from_numpy(a).cuda()] * 2, 1)[:, 0] for a in state]
    # the blocks that the conversions will take hold something else
    used = [torch.full((state[0].size,), 0.5 * p["L"], device="cuda") for _ in range(64)]
    torch.cuda.synchronize()
    del used
    torch.cuda._sleep(100_000_000)
    d.inject(0, *arrays)
    got = d.state(0)
    for k, a in zip(("z", "vx", "vy", "vz"), state):
        assert np.array_equal(got[k], a), k
    d.close()


def test_state_tensors_are_not_written_while_their_memory_is_in_use(pic):
    """Freed tensors whose last writes are still queued behind other work on
    the current stream: their memory comes back as the state's tensors, which
    must be written after those writes."""
    import torch
    p = W.single_diode_small(seed=72)
    d = pic.Diode(p)
    d.inject(0, *mixed_state(p, 73, 4001, 10)[0])
    want = d.state(0)
    d.state(0, device=True)                # (a kernel's first launch may wait for the GPU)
    n = want["z"].size
    old = [torch.zeros(n, device="cuda") for _ in range(64)]
    torch.cuda.synchronize()
    torch.cuda._sleep(100_000_000)
    for t in old:
        t.fill_(-1.0)
    del old, t
    got = d.state(0, device=True)
    torch.cuda.synchronize()
    for k in ("z", "vx", "vy", "vz"):
        assert np.array_equal(got[k].cpu().numpy(), want[k]), k
    d.close()
