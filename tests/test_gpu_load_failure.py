"""A checkpoint load that fails after its buffer was accepted leaves the handle
as it was: the caller's allocator refuses the block for the profile sums, and
the next injection goes after the particles that the handle really holds.
Needs a GPU."""
import ctypes as C

import numpy as np
import pytest

from parity_util import mixed_state
from paper_2605_07083_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("saved,held", [(9001, 2003), (2003, 9001)])
def test_injection_after_a_failed_load(saved, held):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2605_07083_gb300 import build as B
    B.build()
    from paper_2605_07083_gb300 import pic
    p = W.single_diode_small(seed=6)
    a = pic.Diode(p)                       # the checkpoint, with profile sums
    a.set_profile_period(5)
    a.inject(0, *mixed_state(p, 21, saved, 10)[0])
    blob = a.save()
    a.close()

    good, keep = pic._torch_allocator()
    refuse = [False]

    @C.CFUNCTYPE(C.c_void_p, C.c_size_t, C.c_void_p, C.c_void_p)
    def alloc(nbytes, stream, ctx):
        return None if refuse[0] else keep[0](nbytes, stream, ctx)

    mine = pic.PicAllocator()
    mine.alloc, mine.free, mine.ctx = alloc, keep[1], None
    stream = torch.cuda.Stream()
    h = pic.pic_create([pic.make_config(p)], C.c_void_p(stream.cuda_stream), C.byref(mine))
    first = mixed_state(p, 22, held, 10)[0]
    more = mixed_state(p, 23, 501, 10)[0]
    pic.pic_inject(h, 0, 0, *first)
    refuse[0] = True
    with pytest.raises(pic.PicError) as e:
        pic.pic_load(h, blob)
    assert e.value.code == pic.PIC_ENOMEM
    refuse[0] = False
    pic.pic_inject(h, 0, 0, *more)
    st = pic.pic_get_state(h, 0, 0)
    for k, x, y in zip(("z", "vx", "vy", "vz"), first, more):
        assert np.array_equal(st[k], np.concatenate([x, y])), k
    assert np.array_equal(st["id"], np.arange(st["z"].size, dtype=np.uint32))
    pic.pic_load(h, blob)                  # with the block granted it loads
    assert pic.pic_diagnostics(h)["n_live"] == [saved + 5, 0, 0]
    pic.pic_destroy(h)
