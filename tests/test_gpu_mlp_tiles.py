"""The surrogate kernels at the edges of their sample tiles (8, 16, 32 and 128
samples, one wave of 152 blocks each) against the FP64 oracle MLP.  GPU.

Tolerances: FP32 sums of up to 128 products of O(1) terms through three
layers keep about 1e-6 relative to the outputs' size; 1e-5 of the largest
value (and 1e-4 relative where a value is not small) leaves a factor of ten."""
import ctypes as C

import numpy as np
import pytest

from oracle import mlp_oracle as M
from test_gpu_mlp import _bf16_theta, _ptr, _setup, env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

SMS = 152


@pytest.mark.parametrize("batch", [1, 9, 8 * SMS, 8 * SMS + 1, 16 * SMS + 5, 32 * SMS + 1])
def test_forward_tiles(env, batch):  # noqa: F811
    torch, pic, lib = env
    theta, x, _, master, w = _setup(torch, lib, 11, batch)
    xd = torch.from_numpy(x).cuda()
    y = torch.full((batch + 8, 4), 7.0, dtype=torch.float32, device="cuda")
    assert lib.pic_mlp_forward(_ptr(master), _ptr(w), _ptr(xd), batch, _ptr(y), None) == 0
    torch.cuda.synchronize()
    yo, _ = M.forward(_bf16_theta(theta), x.astype(np.float64))
    got = y.cpu().numpy()
    np.testing.assert_allclose(got[:batch], yo, rtol=1e-4, atol=1e-5 * np.abs(yo).max())
    assert (got[batch:] == 7.0).all()            # nothing past the batch is written


@pytest.mark.parametrize("batch,old_scratch", [(1, False), (33, False), (33, True),
                                               (8 * SMS, False), (8 * SMS + 1, False),
                                               (16 * SMS + 3, False), (16 * SMS + 3, True)])
def test_gradient_tiles(env, batch, old_scratch):  # noqa: F811
    """old_scratch: room for one partial per 32 samples only (the least the
    entry point takes), which selects tiles of 32."""
    torch, pic, lib = env
    theta, x, t, master, w = _setup(torch, lib, 12, batch)
    xd, td = torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()
    least = (batch + 31) // 32 * (M.param_count() + 1) * 4
    nbytes = least if old_scratch else lib.pic_mlp_scratch_bytes(batch)
    assert nbytes >= least
    scratch = torch.empty(nbytes // 4, dtype=torch.float32, device="cuda")
    g = torch.empty(M.param_count(), dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    args = (_ptr(master), _ptr(w), _ptr(xd), _ptr(td), batch, _ptr(g), _ptr(loss), _ptr(scratch))
    assert lib.pic_mlp_grad(*args, least - 4, None) == pic.PIC_EINVAL
    assert lib.pic_mlp_grad(*args, nbytes, None) == 0
    torch.cuda.synchronize()
    Lo, go = M.loss_and_grad(_bf16_theta(theta), x.astype(np.float64), t.astype(np.float64))
    assert loss.item() == pytest.approx(Lo, rel=1e-5)
    np.testing.assert_allclose(g.cpu().numpy().astype(np.float64), go, rtol=1e-3,
                               atol=1e-5 * np.abs(go).max())


def test_scratch_of_the_largest_batch_serves_all(env):  # noqa: F811
    torch, pic, lib = env
    sizes = [lib.pic_mlp_scratch_bytes(b) for b in range(1, 6000)]
    assert all(a <= b for a, b in zip(sizes, sizes[1:]))
