"""The counting sort at the edges of its chunks, tiles and counters, against a
stable argsort of the fixed-point cell rule on the host.  Exact.  GPU."""
import ctypes as C

import numpy as np
import pytest

from paper_2605_07083_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CHUNK, TILE = 8192, 4096


@pytest.mark.parametrize("n,cells,order", [
    (1, 1, "random"), (31, 4096, "random"), (CHUNK - 1, 2, "random"), (CHUNK, 127, "one_cell"),
    (CHUNK + 1, 4095, "reversed"), (3 * CHUNK + 513, TILE // 4, "random"),
    (40 * CHUNK + 7, 103, "sorted"), (200003, 4096, "random"), (70 * CHUNK, 2048, "random"),
])
def test_static_sort_is_a_stable_argsort(n, cells, order):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07083_gb300 import build as B
    B.build()
    from paper_2605_07083_gb300 import pic
    lib = pic.load()
    L = 5e-3
    rng = np.random.default_rng(n + cells)
    z = W.clamp_inside((rng.random(n) * L).astype(np.float32), L)
    if order == "sorted":
        z = np.sort(z)
    elif order == "reversed":
        z = np.sort(z)[::-1].copy()
    elif order == "one_cell":
        z[:] = np.float32(0.3 * L)
    fields = [z] + [rng.standard_normal(n).astype(np.float32) for _ in range(3)]
    ids = rng.integers(0, 1 << 31, n).astype(np.int32)
    # one element off 16-byte alignment, the least a caller's float array has
    src = [torch.from_numpy(np.concatenate([a[:1], a])).cuda()[1:] for a in fields + [ids]]
    out = [torch.empty_like(a) for a in src]
    stream = torch.cuda.current_stream().cuda_stream
    rc = lib.pic_sort_by_cell_static(*[C.c_void_p(a.data_ptr()) for a in src], n, cells, L,
                                     *[C.c_void_p(a.data_ptr()) for a in out], C.c_void_p(stream))
    assert rc == pic.PIC_OK
    torch.cuda.synchronize()
    cell = np.clip(np.floor(z * np.float32(cells / L)), 0, cells - 1).astype(np.int64)
    perm = np.argsort(cell, kind="stable")
    for a, b in zip(fields + [ids], out):
        assert np.array_equal(b.cpu().numpy(), a[perm])
