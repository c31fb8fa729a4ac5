"""Sorted spreading into force fields that start at any float of a larger buffer: the sums of a field of
its own, bit for bit, and nothing written beside them -- trees with tiles and of one level (which have a
kernel of their own), the allocating and the allocation-free call."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BALL = np.array([[0.5, 0.5, 0.5, 0.2, 0.1]])


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2605_20565_gb300 as ot
    lib = C.CDLL(ot.library_path())
    lib.ot_spread_noalloc.restype = C.c_int
    lib.ot_spread_noalloc.argtypes = [C.c_void_p, C.c_int] + [C.c_void_p] * 5 + [C.c_int64, C.c_void_p, C.c_void_p]
    return torch, ot, lib.ot_spread_noalloc


@pytest.mark.parametrize("offset", [0, 1, 2, 3])
@pytest.mark.parametrize("lmin,lmax", [(3, 5), (1, 1)])
@pytest.mark.parametrize("kernel", [2, 3])
def test_field_at_any_float(env, kernel, lmin, lmax, offset):
    torch, ot, noalloc = env
    tree = ot.ot_octree_build(BALL if lmax > 1 else np.zeros((0, 5)), lmin, lmax)
    N, n = ot.ot_octree_info(tree)[0], 700
    rng = np.random.default_rng(offset)
    v = rng.normal(size=(3, n))
    X = 0.5 + 0.2 * v / np.linalg.norm(v, axis=0)
    x = [torch.as_tensor(np.ascontiguousarray(X[d]), device="cuda") for d in range(3)]
    F = torch.as_tensor(rng.normal(size=(3, n)).astype(np.float32), device="cuda")
    start = torch.as_tensor(rng.normal(size=(N, 4)).astype(np.float32), device="cuda")
    want = start.clone()
    ot.ot_spread(tree, kernel, ot.OT_SORTED, *x, F, want)
    assert not torch.equal(want, start)
    for alloc in (True, False):
        buf = torch.full((4 * N + 8,), 7.0, dtype=torch.float32, device="cuda")
        f = buf[4 + offset:4 + offset + 4 * N].view(N, 4)
        assert (f.data_ptr() - buf.data_ptr()) % 16 == 4 * offset
        f.copy_(start)
        if alloc:
            ot.ot_spread(tree, kernel, ot.OT_SORTED, *x, F, f)
        else:
            s = C.c_void_p(torch.cuda.current_stream().cuda_stream)
            assert noalloc(tree.handle, kernel, *(a.data_ptr() for a in x), F.data_ptr(), None, n, f.data_ptr(),
                           s) == 0
        assert torch.equal(f, want)
        assert torch.all(buf[:4 + offset] == 7.0) and torch.all(buf[4 + offset + 4 * N:] == 7.0)
