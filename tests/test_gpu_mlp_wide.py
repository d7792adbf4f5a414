"""Predictions of large batches, whose warps take several groups of samples in
turn: batches that select 12, 16 and 20 warps a block (the fewest idle in the
last round of 152 blocks), each of two rounds or more and ragged, against the
FP64 oracle.  GPU.  The tolerance is that of the tiled predictions: FP32 sums of
up to 128 products through three layers."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from test_gpu_mlp import _bf16_theta, _ptr, _setup, env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,warps,rounds", [(41213, 12, 3), (38909, 16, 2), (48635, 20, 2)])
def test_wide_prediction_rounds(env, batch, warps, rounds):  # noqa: F811
    torch, pic, lib = env
    per_sm = -(-(-(-batch // 8)) // 152)
    slots = {n: -(-per_sm // n) * n for n in (16, 20, 12)}
    assert min(slots, key=slots.get) == warps and slots[warps] == rounds * warps
    theta, x, _, master, w = _setup(torch, lib, 13, batch)
    xd = torch.from_numpy(x).cuda()
    y = torch.full((batch + 8, 4), 7.0, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    assert lib.pic_mlp_forward(_ptr(master), _ptr(w), _ptr(xd), batch, _ptr(y), None) == 0
    torch.cuda.synchronize()
    yo, _ = M.forward(_bf16_theta(theta), x.astype(np.float64))
    got = y.cpu().numpy()
    np.testing.assert_allclose(got[:batch], yo, rtol=1e-4, atol=1e-5 * np.abs(yo).max())
    assert (got[batch:] == 7.0).all()
