"""The library's host side against failing allocations, without a GPU: the CUDA runtime's memory calls are
those of fake_cudart.c (kernels do nothing), preloaded in a child process."""
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PROLOGUE = """
import ctypes as C, sys
fake = C.CDLL(sys.argv[1])
lib = C.CDLL(sys.argv[2])
fake.fake_fail_from.argtypes = [C.c_size_t]
lib.ot_octree_build.argtypes = [C.c_void_p, C.c_int, C.c_void_p, C.c_void_p, C.c_void_p]
lib.ot_octree_destroy.argtypes = [C.c_void_p]
MALLOC, POOL, OOM = 1, 2, -3
def build(level):
    h = C.c_void_p()
    prm = (C.c_int * 3)(level, level, 1)
    return lib.ot_octree_build(None, 0, prm, None, C.byref(h)), h
def destroy(h):
    assert lib.ot_octree_destroy(h) == 0
def map_level(h):
    v = C.c_int(-1)
    assert lib.ot_octree_get_map_level(h, C.byref(v)) == 0
    return v.value
"""


@pytest.fixture(scope="module")
def child(tmp_path_factory):
    from paper_2605_20565_gb300 import _build
    lib = _build.build()
    fake = str(tmp_path_factory.mktemp("fake") / "fake_cudart.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-w", "-o", fake, os.path.join(HERE, "fake_cudart.c")], check=True)

    def run(script):
        env = dict(os.environ, LD_PRELOAD=fake)
        r = subprocess.run([sys.executable, "-c", PROLOGUE + script, fake, lib], env=env, cwd=ROOT, timeout=120,
                           capture_output=True, text=True)
        assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
    return run


@pytest.mark.parametrize("level,bytes_", [(1, 1), (1, 8 * 16), (3, 1), (0, 16)])
def test_a_map_level_without_memory_leaves_the_octree_as_it_was(child, level, bytes_):
    """Either allocation of ot_octree_set_map_level fails (bytes_: from which size on): the call reports it, the
    level stays, and nothing that the octree holds was freed; with memory again the same call succeeds."""
    child(f"""
st, h = build(3)
assert st == 0 and map_level(h) == 3
assert lib.ot_octree_set_map_level(h, 2, None) == 0
live = fake.fake_live(POOL), fake.fake_live(MALLOC)
for _ in range(3):
    fake.fake_fail_from({bytes_})
    assert lib.ot_octree_set_map_level(h, {level}, None) == OOM
    assert map_level(h) == 2 and (fake.fake_live(POOL), fake.fake_live(MALLOC)) == live
fake.fake_fail_from(1 << 62)
assert lib.ot_octree_set_map_level(h, {level}, None) == 0 and map_level(h) == {level}
assert lib.ot_octree_set_map_level(h, 2, None) == 0 and map_level(h) == 2
assert (fake.fake_live(POOL), fake.fake_live(MALLOC)) == live
destroy(h)
assert fake.fake_live(POOL) == 0
""")


@pytest.mark.parametrize("old_first", [False, True])
def test_pools_end_with_their_context(child, old_first):
    """Octrees after a context was destroyed and made again (cudaDeviceReset) take their memory from a
    pool of the new one, which is given back with its last octree whatever was left in the old one."""
    child(f"""
st, a = build(2)
st2, b = build(1)
assert st == 0 and st2 == 0
fake.fake_new_context()
st, c = build(2)
assert st == 0 and fake.fake_dead_pool() == 0
if {old_first}:
    destroy(a)
assert fake.fake_trims() == 0
destroy(c)
assert fake.fake_trims() == 1 and fake.fake_dead_pool() == 0
if not {old_first}:
    destroy(a)
destroy(b)
st, d = build(3)
assert st == 0
destroy(d)
assert fake.fake_trims() == 2 and fake.fake_dead_pool() == 0
""")


def test_memory_is_released_after_a_wait_that_captures_allow(child):
    """Destroying an octree, changing its map and dropping its tables wait for the device before pool
    memory is released, without cudaDeviceSynchronize (an error while a stream is captured anywhere)."""
    child("""
st, h = build(3)
assert st == 0
for level in (2, 1, 3):
    assert lib.ot_octree_set_map_level(h, level, None) == 0
for enable in (1, 1, 0, 1):
    assert lib.ot_octree_build_mates(h, enable, None) == 0
st, g = build(2)
destroy(h)
destroy(g)
assert fake.fake_unwaited() == 0 and fake.fake_device_syncs() == 0 and fake.fake_live(POOL) == 0
""")


@pytest.mark.parametrize("why", ["leaves", "memory"])
def test_refused_leaves_leave_no_memory(child, why):
    """ot_octree_from_leaves that is refused, for its leaves or for want of memory, gives the pool's memory
    back when no octree lives, and only then."""
    child(f"""
lib.ot_octree_from_leaves.argtypes = [C.c_void_p, C.c_void_p, C.c_int64, C.c_int, C.c_void_p, C.c_void_p]
keys, levels = (C.c_uint64 * 8)(), (C.c_uint8 * 8)()
def refused():
    if {why == "leaves"}:
        fake.fake_copy_word(1, 1)  # the count of leaves out of place
        want = -4
    else:
        fake.fake_fail_from(1)
        want = OOM
    h = C.c_void_p(1)
    assert lib.ot_octree_from_leaves(keys, levels, 8, 1, None, C.byref(h)) == want and not h.value
    fake.fake_copy_word(0, 0)
    fake.fake_fail_from(1 << 62)
refused()
assert fake.fake_live(POOL) == 0 and fake.fake_trims() == 1
st, h = build(2)
live = fake.fake_live(POOL)
refused()
assert fake.fake_live(POOL) == live and fake.fake_trims() == 1
destroy(h)
assert fake.fake_live(POOL) == 0 and fake.fake_trims() == 2
""")


@pytest.mark.parametrize("mates", [False, True])
@pytest.mark.parametrize("tile", [1, 2, 3, 4, 5, 7, 48, 64])
def test_tiles_of_a_small_batch(child, tile, mates):
    """With fewer tiles than warps the tiles get smaller: the trilinear kernels' stay whole rows of 32 points (a
    tile that ends within a row would be done twice from there on), the delta kernels' at least 4
    points, and the tiles cover the points once."""
    child(f"""
class Group(C.Structure):
    _fields_ = [("kernel", C.c_int), ("x", C.c_void_p), ("y", C.c_void_p), ("z", C.c_void_p), ("n", C.c_int64),
                ("u", C.c_void_p), ("host", C.c_void_p)]
st, h = build(3)
if {mates}:
    assert lib.ot_octree_build_mates(h, 1, None) == 0
for n in (1, 31, 300, 1000, 6000):
    fake.fake_forget_batches()
    x = (C.c_double * n)()
    u = (C.c_float * (3 * n))()
    p = [C.addressof(a) for a in (x, x, x, u)]
    kinds = (2, 1) if {mates} else (1,)
    groups = (Group * len(kinds))(*(Group(k, *p[:3], n, p[3], None) for k in kinds))
    launch = (C.c_int * 7)(0, {tile}, 0, 0, 0, 0, -1)
    b = C.c_void_p()
    lib.ot_batch_create.argtypes = [C.c_void_p, C.c_void_p, C.c_int, C.c_void_p, C.c_int] + [C.c_void_p] * 3
    assert lib.ot_batch_create(h, groups, len(kinds), u, 0, launch, None, C.byref(b)) == 0
    assert fake.fake_batch_launches() == len(kinds)
    for i, kind in enumerate(kinds):
        pts, tiles = fake.fake_batch_pts(i), fake.fake_batch_tiles(i)
        assert fake.fake_batch_kernel(i) == kind and tiles == -(-n // pts)
        assert pts <= 32 * {tile} and pts % (32 if kind == 1 else 4) == 0
        # as small as it may be while there are fewer tiles than the 32 warps of the fake's 4 SMs
        assert tiles >= 32 or pts < 2 * (32 if kind == 1 else 4)
    lib.ot_batch_destroy.argtypes = [C.c_void_p]
    assert lib.ot_batch_destroy(b) == 0
destroy(h)
assert fake.fake_live(POOL) == 0
""")


def test_a_batch_without_memory_for_records_is_made_without(child):
    """Creating a batch with value records takes four allocations for them (the bits and count, the records,
    the node list, the cells' entries): whichever fails, the batch is made without records and keeps
    none of the others."""
    child("""
class Group(C.Structure):
    _fields_ = [("kernel", C.c_int), ("x", C.c_void_p), ("y", C.c_void_p), ("z", C.c_void_p), ("n", C.c_int64),
                ("u", C.c_void_p), ("host", C.c_void_p)]
st, h = build(3)
assert lib.ot_octree_build_mates(h, 1, None) == 0
n = 4096
x, u = (C.c_double * n)(), (C.c_float * (3 * n))()
px, pu = C.addressof(x), C.addressof(u)
groups = (Group * 1)(Group(1, px, px, px, n, pu, None))
lib.ot_batch_create.argtypes = [C.c_void_p, C.c_void_p, C.c_int, C.c_void_p, C.c_int] + [C.c_void_p] * 3
lib.ot_batch_destroy.argtypes = [C.c_void_p]
before = fake.fake_live(MALLOC)
def create():
    b = C.c_void_p()
    fake.fake_copy_word(1, 5)  # nodes of hot leaves
    st = lib.ot_batch_create(h, groups, 1, u, 0, None, None, C.byref(b))
    fake.fake_copy_word(0, 0)
    held = fake.fake_live(MALLOC) - before
    assert st == 0 and lib.ot_batch_destroy(b) == 0 and fake.fake_live(MALLOC) == before
    return held
assert create() == 5  # the tile counter, the cell means; records, node list, entries
for k in (3, 4, 5, 6):
    fake.fake_fail_nth(k)
    assert create() == 2
fake.fake_fail_nth(-1)
assert create() == 5
destroy(h)
""")


def test_what_a_reset_took_is_not_freed_again(child):
    """Octrees (with tables) and batches of a destroyed context are dropped without releasing anything: their
    addresses are not theirs any more, and may be a newer octree's."""
    child("""
class Group(C.Structure):
    _fields_ = [("kernel", C.c_int), ("x", C.c_void_p), ("y", C.c_void_p), ("z", C.c_void_p), ("n", C.c_int64),
                ("u", C.c_void_p), ("host", C.c_void_p)]
lib.ot_batch_create.argtypes = [C.c_void_p, C.c_void_p, C.c_int, C.c_void_p, C.c_int] + [C.c_void_p] * 3
lib.ot_batch_destroy.argtypes = [C.c_void_p]
x, u = (C.c_double * 64)(), (C.c_float * 192)()
px, pu = C.addressof(x), C.addressof(u)
def make():
    st, h = build(3)
    assert st == 0 and lib.ot_octree_build_mates(h, 1, None) == 0
    b = C.c_void_p()
    assert lib.ot_batch_create(h, (Group * 1)(Group(1, px, px, px, 64, pu, None)), 1, u, 0, None, None, C.byref(b)) == 0
    return h, b
old, old_batch = make()
fake.fake_new_context()
new, new_batch = make()
live = fake.fake_live(POOL | MALLOC)
assert lib.ot_batch_destroy(old_batch) == 0
destroy(old)
assert fake.fake_live(POOL | MALLOC) == live and fake.fake_bad_frees() == 0
assert lib.ot_batch_destroy(new_batch) == 0
destroy(new)
assert fake.fake_live(POOL) == 0 and fake.fake_bad_frees() == 0
""")


def test_ordered_copies_fit_their_allocation(child):
    """The ordered copies of a group's positions and results, for every size modulo their alignment, with hosts and
    without."""
    child("""
class Group(C.Structure):
    _fields_ = [("kernel", C.c_int), ("x", C.c_void_p), ("y", C.c_void_p), ("z", C.c_void_p), ("n", C.c_int64),
                ("u", C.c_void_p), ("host", C.c_void_p)]
lib.ot_batch_create.argtypes = [C.c_void_p, C.c_void_p, C.c_int, C.c_void_p, C.c_int] + [C.c_void_p] * 3
lib.ot_batch_destroy.argtypes = [C.c_void_p]
st, h = build(3)
x, u = (C.c_double * 64)(), (C.c_float * 192)()
px, pu = C.addressof(x), C.addressof(u)
launch = (C.c_int * 7)(0, 0, 0, 5, 0, 0, 0)
wrong = []
for n in [*range(64, 64 + 513), *range(4090, 4110), 100_003]:
    groups = (Group * 2)(Group(1, px, px, px, n, pu, pu), Group(1, px, px, px, n, pu, None))
    fake.fake_forget_batches()
    b = C.c_void_p()
    assert lib.ot_batch_create(h, groups, 2, u, 0, launch, None, C.byref(b)) == 0
    wrong += [n for g in range(2) if not fake.fake_batch_fits(0, g)]
    assert lib.ot_batch_destroy(b) == 0
assert not wrong, wrong
destroy(h)
""")
