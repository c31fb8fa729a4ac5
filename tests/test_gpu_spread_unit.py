"""Sorted spreading on trees of one level (8 leaves), where the sums over all markers are split over
threads and blocks: sizes around a block's 256 markers and around all blocks' 155,648, both
kernels, FP32 and FP64, closed and periodic, with markers outside the cube; two calls bit for bit, and the
allocation-free call's bits.  Forces of one sign, so that the largest sum is that of the terms'
magnitudes: FP32 1e-5 of it, FP64 1e-12 (sums of at most 100 terms in a row: 1e-14).  Many markers in
parallel: 2 million in less than 50 ms (2.2 s by one thread per leaf, 77 us by all of them)."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import oracle
    import paper_2605_20565_gb300 as ot
    lib = C.CDLL(ot.library_path())
    lib.ot_spread_noalloc.restype = C.c_int
    lib.ot_spread_noalloc.argtypes = [C.c_void_p, C.c_int] + [C.c_void_p] * 5 + [C.c_int64, C.c_void_p, C.c_void_p]
    return torch, ot, oracle, lib.ot_spread_noalloc


@pytest.mark.parametrize("kernel", [2, 3])
@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("n", [1, 32, 255, 256, 257, 5_000, 155_648, 155_649, 400_001])
def test_sums(env, n, periodic, kernel):
    torch, ot, oracle, noalloc = env
    ko, lo = oracle.octree_build(np.zeros((0, 5)), 1, 1)
    tree = ot.ot_octree_build(np.zeros((0, 5)), 1, 1)
    ot.ot_octree_set_periodic(tree, periodic)
    rng = np.random.default_rng(n)
    X = rng.random((3, n))
    if n > 1:
        X[0, ::50] = 1.5
    F = rng.uniform(0.5, 1.5, (3, n)).astype(np.float32)
    dV = rng.uniform(0.1, 0.2, n).astype(np.float32)
    inside = X[0] < 1
    kw = dict(periodic=True) if periodic else {}
    ref, _ = oracle.spread_delta(ko, lo, 1, kernel, *np.ascontiguousarray(X[:, inside]),
                                 F[:, inside].astype(np.float64), dV=dV[inside].astype(np.float64), **kw)
    x = [torch.as_tensor(np.ascontiguousarray(X[d]), device="cuda") for d in range(3)]
    for dtype, tol in ((torch.float32, 1e-5), (torch.float64, 1e-12)):
        Fd, dVd = (torch.as_tensor(a, device="cuda").to(dtype) for a in (F, dV))
        spread = ot.ot_spread if dtype == torch.float32 else ot.ot_spread_f64
        out = []
        for _ in range(2):
            f = torch.zeros((8, 4), dtype=dtype, device="cuda")
            spread(tree, kernel, ot.OT_SORTED, *x, Fd, f, dV=dVd)
            out.append(f)
        assert torch.equal(*out)
        assert np.abs(out[0].cpu().numpy()[:, :3] - ref[:, :3]).max() <= tol * np.abs(ref[:, :3]).max()
        if dtype == torch.float32 and n <= 150_635:
            f = torch.zeros((8, 4), dtype=dtype, device="cuda")
            s = C.c_void_p(torch.cuda.current_stream().cuda_stream)
            assert noalloc(tree.handle, kernel, *(a.data_ptr() for a in x), Fd.data_ptr(), dVd.data_ptr(), n,
                           f.data_ptr(), s) == 0
            assert torch.equal(f, out[0])
    assert bool(ot.ot_last_error(tree) & ot.OT_DEV_OUTSIDE) == (n > 1)


def test_many_markers_in_parallel(env):
    torch, ot, _, _ = env
    tree = ot.ot_octree_build(np.zeros((0, 5)), 1, 1)
    n = 2_000_000
    x = [torch.rand(n, dtype=torch.float64, device="cuda") for _ in range(3)]
    F = torch.rand((3, n), dtype=torch.float32, device="cuda")
    f = torch.zeros((8, 4), dtype=torch.float32, device="cuda")
    e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for _ in range(2):
        e[0].record()
        ot.ot_spread(tree, 2, ot.OT_SORTED, *x, F, f)
        e[1].record()
        torch.cuda.synchronize()
    assert e[0].elapsed_time(e[1]) < 50.0
