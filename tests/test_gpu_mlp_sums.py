"""The order in which the network's gradient and loss are summed over the
batch.  GPU.

With all parameters zero the output is 0, and one target value for every
sample makes every sample's output-bias gradient the same FP32 number d, known
exactly: what is left is the rounding of the sum.  A sum of like terms is off
by at most its longest chain of additions times 2^-24: the samples of a tile,
the rounds of sixteen partials (32 for the loss) and the tree over them.  Added
one after another, 152 tiles' partials are off by 36 such units for these
targets, 38 partials of 32 samples by 2."""
import numpy as np
import pytest

from oracle import mlp_oracle as M
from test_gpu_mlp import _ptr, env  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.mark.parametrize("batch,tile", [(100, 8), (1211, 8), (1216, 8), (2432, 16), (4096, 32)])
@pytest.mark.parametrize("target", [1.9075, 1.96, 1.9925])
def test_summation_error_of_gradient_and_loss(env, batch, tile, target):  # noqa: F811
    torch, pic, lib = env
    n = M.param_count()
    zero = torch.zeros(n, dtype=torch.float32, device="cuda")
    w = torch.zeros(n, dtype=torch.bfloat16, device="cuda")
    x = torch.zeros((batch, 5), dtype=torch.float32, device="cuda")
    t = torch.full((batch, 4), target, dtype=torch.float32, device="cuda")
    nbytes = lib.pic_mlp_scratch_bytes(batch)
    scratch = torch.empty(nbytes // 4, dtype=torch.float32, device="cuda")
    g, loss = torch.empty(n, device="cuda"), torch.empty(1, device="cuda")
    torch.cuda.synchronize()
    assert lib.pic_mlp_grad(_ptr(zero), _ptr(w), _ptr(x), _ptr(t), batch, _ptr(g), _ptr(loss),
                            _ptr(scratch), nbytes, None) == 0
    torch.cuda.synchronize()
    diff = np.float32(0) - np.float32(target)
    d = np.float32(2) * diff / np.float32(batch * 4)
    want = float(d) * batch
    parts = -(-batch // tile)
    chain = tile + (-(-parts // 16) - 1) + 4
    got = g[-4:].double().cpu().numpy()
    assert (np.abs(got - want) <= chain * U * abs(want)).all(), (got - want) / want / U
    # squares of a tile over 32 lanes in 16 rows, its tree, the tiles over 32
    # lanes, their tree; the square and the division round too
    chain = 16 + 5 + (-(-parts // 32) - 1) + 5 + 2
    want = float(diff) ** 2
    assert abs(loss.item() - want) <= chain * U * want, (loss.item() - want) / want / U
