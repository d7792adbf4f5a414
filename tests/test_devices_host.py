"""What the library's host side does, in a process with two devices among other
things, on a stand-in for the CUDA runtime (fake_cudart.c): no GPU, nothing is
launched.
Each case runs in a process of its own, which loads the library against the
stand-in."""
import os
import subprocess
import sys

import pytest

from conftest import ROOT

DEVICE, MANAGED = 2, 3                       # cudaMemoryType
HANDLE = '''
import ctypes as C, sys
lib = C.CDLL(sys.argv[1])
fake = C.CDLL("libcudart.so.13")
word = lambda name: C.c_int.in_dll(fake, name)
last_kernel = lambda name: name.encode() in C.c_char_p.in_dll(fake, "fake_last_kernel").value
from paper_2605_07083_gb300 import pic, workloads as W
for name, (res, args) in pic.ENTRY_POINTS.items():
    getattr(lib, name).restype, getattr(lib, name).argtypes = res, args
fake.fake_array.argtypes = [C.c_void_p, C.c_size_t, C.c_int, C.c_int]
def create():                                # on device 1, with a stream of device 1
    word("fake_device").value = 1
    h, cfg = C.c_void_p(), pic.make_config(dict(W.single_diode_small(), capacity=(4096,) * 3))
    assert lib.pic_create(C.byref(cfg), 1, C.c_void_p(0x1000), None, C.byref(h)) == 0
    return h
def array(n, kind, device):
    a = (C.c_uint32 * n)()
    fake.fake_array(a, C.sizeof(a), kind, device)
    return a
'''


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_2605_07083_gb300 import build as B
    lib = B.build()
    out = tmp_path_factory.mktemp("fake")
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-Wno-builtin-declaration-mismatch",
                    "-Wl,-soname,libcudart.so.13", os.path.join(ROOT, "tests", "fake_cudart.c"),
                    "-o", str(out / "libcudart.so.13")], check=True)

    def go(body):
        env = dict(os.environ, LD_LIBRARY_PATH=str(out), PYTHONPATH=ROOT)
        r = subprocess.run([sys.executable, "-c", HANDLE + body, lib], env=env, text=True,
                           capture_output=True, timeout=120)
        assert r.returncode == 0, r.stdout + r.stderr
    return go


@pytest.mark.parametrize("kind,device,direct", [(DEVICE, 1, True), (DEVICE, 0, False),
                                                (MANAGED, 0, True), (0, 0, False)])
def test_only_arrays_of_the_handles_device_are_read_by_kernels(run, kind, device, direct):
    """One array of several elsewhere (or not known to the runtime) sends the
    whole call through cudaMemcpyAsync, which carries it over or refuses it."""
    run(f'''
h = create()
a = [array(512, {DEVICE}, 1) for _ in range(4)] + [array(512, {kind}, {device})]
n = C.c_int64()
copies = word("fake_copies").value
assert lib.pic_inject(h, 0, 0, 512, a[0], a[1], a[4], a[3], 1) == 0
assert (word("fake_copies").value == copies) == {direct}
assert lib.pic_get_state(h, 0, 0, *a, 512, C.byref(n), 1) == 0
assert last_kernel("k_state_copy" if {direct} else "k_read")
''')


@pytest.mark.parametrize("elements,offset,direct", [(512, 0, True), (511, 0, False), (600, 88, True),
                                                    (600, 89, False)])
def test_a_count_beyond_the_array_is_not_read_by_kernels(run, elements, offset, direct):
    """512 particles from (to) an array with `elements` of them, from `offset`
    on: past its end cudaMemcpyAsync is asked, which refuses what does not fit
    (the stand-in copies: the memory behind the array is there)."""
    run(f'''
h = create()
whole = (C.c_float * 1024)()
fake.fake_array(whole, 4 * {elements}, {DEVICE}, 1)
short = C.byref(whole, 4 * {offset})
a = [array(512, {DEVICE}, 1) for _ in range(3)]
copies = word("fake_copies").value
assert lib.pic_inject(h, 0, 0, 512, a[0], short, a[1], a[2], 1) == 0
assert (word("fake_copies").value == copies) == {direct}
n = C.c_int64()
assert lib.pic_get_state(h, 0, 0, a[0], short, a[1], a[2], None, 512, C.byref(n), 1) == 0
assert last_kernel("k_state_copy" if {direct} else "k_read")
''')


@pytest.mark.parametrize("call", [
    "lib.pic_synchronize(h)", "lib.pic_diagnostics(h, 0, C.byref(pic.PicDiag()))",
    "lib.pic_get_state(h, 0, 0, *a, 512, C.byref(n), 1)",
    "lib.pic_get_state(h, 0, 0, None, None, None, None, None, 512, C.byref(n), 0)",
    "lib.pic_get_rho_fixed(h, 0, rho, 129)", "lib.pic_checkpoint_bytes(h, C.byref(size))"])
def test_reads_work_whichever_device_is_current(run, call):
    """A thread that reads a handle need not have selected the handle's device
    (launches on another device's stream are refused), and finds its own device
    current afterwards."""
    run(f'''
h = create()
a = [array(512, {DEVICE}, 1) for _ in range(5)]
n, size, rho = C.c_int64(), C.c_size_t(), (C.c_int64 * 129)()
assert lib.pic_get_rho_fixed(h, 0, rho, 129) == 0      # the empty state's charge is deposited
word("fake_device").value = 0
assert {call} == 0
assert word("fake_refused").value == 0 and word("fake_device").value == 0
''')


def test_network_kernels_are_set_up_on_every_device(run):
    """The raised shared-memory limit of a kernel holds for one device: the
    first call on a second one sets it there, later calls on neither."""
    run(f'''
a = array(1 << 16, {DEVICE}, 0)
counts = (C.c_int * 2).in_dll(fake, "fake_attributes")
for device in (0, 1, 1, 0):
    word("fake_device").value = device
    assert lib.pic_mlp_forward(a, a, a, 10, a, None) == 0
    seen = list(counts)
    if device == 1:
        assert seen[1] == seen[0] > 0
assert list(counts) == seen
''')


@pytest.mark.parametrize("window,period,steps", [(0, 100, 50), (70, 100, 130), (1000, 33, 250),
                                                 (0, 100, 3)])
def test_prepared_steps_capture_nothing_at_any_phase_of_the_samples(run, window, period, steps):
    """Sampled steps run by themselves, so the stretches between them start
    anywhere: after one preparation no later call of as many steps captures."""
    run(f'''
h = C.c_void_p()
word("fake_device").value = 1
p = dict(W.single_diode_small(), capacity=(4096,) * 3, window_start={window})
cfg = pic.make_config(p)
assert lib.pic_create(C.byref(cfg), 1, C.c_void_p(0x1000), None, C.byref(h)) == 0
t = pic.PicTuning(size=C.sizeof(pic.PicTuning), wait_polls=5)   # three kernels a step
assert lib.pic_tune(h, C.byref(t)) == 0
assert lib.pic_set_profile_period(h, {period}) == 0
assert lib.pic_prepare_steps(h, {steps}) == 0
captures = word("fake_captures").value
for _ in range(40):
    assert lib.pic_step(h, {steps}) == 0
assert word("fake_graph_launches").value > 0 and captures > 0
assert word("fake_captures").value == captures
''')


@pytest.mark.parametrize("cells,room,live,tune,wide", [
    (4096, 3 << 20, 20000, {}, False), (4096, 3 << 20, 900000, {}, False),
    (4096, 3 << 20, 1100000, {}, True), (4096, 3 << 20, 0, {}, False),
    (4096, 1 << 23, 0, {}, True), (4096, 1 << 23, 20000, {}, False),
    (4096, 3 << 20, 1100000, {"push_threads": 320}, False), (2048, 3 << 20, 1100000, {}, False)])
def test_one_wide_push_block_only_for_many_particles(run, cells, room, live, tune, wide):
    """The grids that leave two push blocks too few warps take one wide block
    per SM from a million particles on; the first step after an injection
    decides, and by the room where there are none."""
    run(f'''
h = C.c_void_p()
word("fake_device").value = 1
p = dict(W.single_diode_production(), Nz={cells}, capacity=({room} // 3,) * 3)
cfg = pic.make_config(p)
assert lib.pic_create(C.byref(cfg), 1, C.c_void_p(0x1000), None, C.byref(h)) == 0
t = pic.PicTuning(size=C.sizeof(pic.PicTuning), graph_steps=-1, **{tune})
assert lib.pic_tune(h, C.byref(t)) == 0
for sp in (0, 1):
    if {live}:
        a = [(C.c_float * ({live} // 2))() for _ in range(4)]
        assert lib.pic_inject(h, 0, sp, {live} // 2, *a, 0) == 0
for _ in range(3):
    assert lib.pic_step(h, 2) == 0
fake.fake_count.argtypes = [C.c_char_p]
steps, one = fake.fake_count(b"k_post"), fake.fake_count(b"k_push_wide")
assert steps == 6 and one == (6 if {wide} else 0)
''')
