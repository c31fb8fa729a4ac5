"""Octrees before and after cudaDeviceReset, in a child process that uses the C ABI and the CUDA runtime
only: those made after it are the oracle's, bit for bit, also when one made before it is destroyed
among them."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

SCRIPT = """
import ctypes as C, sys
import numpy as np
import oracle
lib, rt = C.CDLL(sys.argv[1]), C.CDLL("libcudart.so.13")
lib.ot_octree_leaves.argtypes = [C.c_void_p] * 4
rt.cudaMemcpy.argtypes = [C.c_void_p, C.c_void_p, C.c_size_t, C.c_int]
ball = np.array([[0.5, 0.5, 0.5, 0.2, 0.1]])
ko, lo = oracle.octree_build(ball, 3, 6)
def leaves(h):
    n, k, l = C.c_int64(), C.c_void_p(), C.c_void_p()
    assert lib.ot_octree_leaves(h, C.byref(n), C.byref(k), C.byref(l)) == 0
    keys, lev = np.empty(n.value, np.uint64), np.empty(n.value, np.uint8)
    assert rt.cudaMemcpy(keys.ctypes.data, k, keys.nbytes, 2) == 0 and rt.cudaMemcpy(lev.ctypes.data, l, lev.nbytes, 2) == 0
    assert np.array_equal(keys, ko) and np.array_equal(lev, lo)
def build():
    h = C.c_void_p()
    assert lib.ot_octree_build(ball.ctypes.data_as(C.c_void_p), 1, (C.c_int * 3)(3, 6, 1), None, C.byref(h)) == 0
    leaves(h)
    return h
old = build()
for _ in range(2):
    assert rt.cudaDeviceReset() == 0
    h, g = build(), build()
    assert lib.ot_octree_destroy(old) == 0  # of the context before: nothing of the new ones is released
    i = build()
    for t in (h, g, i):
        leaves(t)
    assert lib.ot_octree_destroy(h) == 0 and lib.ot_octree_destroy(i) == 0
    leaves(g)
    old = build()
"""


def test_octrees_after_a_device_reset():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2605_20565_gb300 as ot
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", SCRIPT, ot.library_path()], cwd=root, timeout=300, capture_output=True,
                       text=True)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-2000:]
