"""Sorted spreading and multi-direct forcing with markers in more home tiles than the block-per-tile form
takes (4096): the warp-per-run form against the oracle, both kernels, FP32 and FP64, closed cubes with
stencils past the faces and periodic ones, stencils that leave the finest level, forces that are not
finite, markers outside the cube; and the 150,000 scattered markers that the allocation-free call is
compared on.  Tolerance: 1e-5 of the largest value in FP32, 1e-12 in FP64, as everywhere."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

BALL = np.array([[0.45, 0.5, 0.55, 0.3, 0.01]])
TREES = {"uniform": (np.zeros((0, 5)), 7, 7), "ball": (BALL, 3, 8)}


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import oracle
    import paper_2605_20565_gb300 as ot
    leaves = {k: oracle.octree_build(*v) for k, v in TREES.items()}
    return torch, ot, oracle, leaves


def home_tiles(X, lmax, kernel, periodic):
    s = X * 2.0 ** lmax
    i0 = (np.floor(s - 0.5) - 1 if kernel == 2 else np.floor(s) - 1).astype(np.int64)
    i0 = i0 % (1 << lmax) if periodic else np.maximum(i0, 0)
    return len(np.unique(np.ravel_multi_index(i0 >> 2, 3 * (1 << (lmax - 2),))))


def markers(tree, n, seed):
    """Anywhere in the uniform tree; around the ball's surface, a tenth of them off the finest level."""
    rng = np.random.default_rng(seed)
    if tree == "uniform":
        X = rng.random((3, n))
        X[:, ::40] = rng.random((3, X[:, ::40].shape[1])) * 2.0 ** -7  # at three faces
        return X
    v = rng.normal(size=(3, n))
    r = 0.3 + np.where(rng.random(n) < 0.1, 0.06, 0.004) * rng.uniform(-1, 1, n)
    return np.ascontiguousarray(BALL[0, :3, None] + r * v / np.linalg.norm(v, axis=0))


def cuda(torch, X):
    return [torch.as_tensor(np.ascontiguousarray(X[d]), device="cuda") for d in range(3)]


@pytest.mark.parametrize("tree,periodic", [("uniform", False), ("uniform", True), ("ball", False)])
@pytest.mark.parametrize("kernel", [2, 3])
def test_spreading(env, tree, periodic, kernel):
    torch, ot, oracle, leaves = env
    lmax, n = TREES[tree][2], 60_000
    ko, lo = leaves[tree]
    t = ot.ot_octree_build(*TREES[tree])
    ot.ot_octree_set_periodic(t, periodic)
    X = markers(tree, n, kernel)
    assert home_tiles(X, lmax, kernel, periodic) > 4096
    rng = np.random.default_rng(8)
    F = rng.normal(size=(3, n)).astype(np.float32)
    dV = (rng.uniform(0.5, 2.0, n) * 2.0 ** (-3 * lmax)).astype(np.float32)
    ref, bad = oracle.spread_delta(ko, lo, lmax, kernel, *X, F.astype(np.float64), dV=dV.astype(np.float64),
                                   periodic=periodic)
    scale = np.abs(ref[:, :3]).max()
    x = cuda(torch, X)
    for dtype, tol in ((torch.float32, 1e-5), (torch.float64, 1e-12)):
        spread = ot.ot_spread if dtype == torch.float32 else ot.ot_spread_f64
        Fd, dVd = (torch.as_tensor(a, device="cuda").to(dtype) for a in (F, dV))
        out = []
        for _ in range(2):
            f = torch.zeros((ko.size, 4), dtype=dtype, device="cuda")
            spread(t, kernel, ot.OT_SORTED, *x, Fd, f, dV=dVd)
            out.append(f)
        assert torch.equal(*out)
        assert np.abs(out[0].cpu().numpy()[:, :3] - ref[:, :3]).max() <= tol * scale
        assert bool(ot.ot_last_error(t) & ot.OT_DEV_STENCIL) == (bad > 0) == (not periodic)
        # one force that is not finite: its stencil's cells only
        one = torch.zeros_like(Fd)
        one[:, 17] = 1.0
        g = torch.zeros_like(f)
        spread(t, kernel, ot.OT_SORTED, *x, one, g)
        reached = g[:, 0] != 0
        Fd[0, 17], Fd[1, 17] = np.inf, np.nan
        f = torch.zeros_like(f)
        spread(t, kernel, ot.OT_SORTED, *x, Fd, f, dV=dVd)
        assert 0 < int(reached.sum()) <= 64 and torch.equal(f[~reached], out[0][~reached])
        assert torch.all(f[reached, 0].isinf()) and torch.all(f[reached, 1].isnan())
        assert torch.equal(f[:, 2], out[0][:, 2])
        ot.ot_last_error(t)


@pytest.mark.parametrize("tree,periodic", [("uniform", False), ("uniform", True), ("ball", False)])
@pytest.mark.parametrize("n", [3_000, 40_000])
@pytest.mark.parametrize("kernel", [2, 3])
def test_multi_direct_forcing(env, tree, periodic, n, kernel):
    torch, ot, oracle, leaves = env
    lmax = TREES[tree][2]
    ko, lo = leaves[tree]
    t = ot.ot_octree_build(*TREES[tree])
    ot.ot_octree_set_periodic(t, periodic)
    X = markers(tree, n, n + kernel)
    assert n < 8192 or home_tiles(X, lmax, kernel, periodic) > 4096
    rng = np.random.default_rng(n)
    U = (0.3 * rng.normal(size=(3, n))).astype(np.float32)
    u0 = rng.normal(size=(ko.size, 4)).astype(np.float32)
    rho, dt, rounds = 1.3, 0.7, 3
    u, f, slip, skipped = u0.astype(np.float64), np.zeros((ko.size, 4)), [], 0
    for _ in range(rounds + 1):
        uk, bad = oracle.interp_delta(ko, lo, lmax, kernel, u, *X, periodic=periodic)
        slip.append(np.sqrt(((U - uk) ** 2).sum()))
        if len(slip) <= rounds:
            d, _ = oracle.spread_delta(ko, lo, lmax, kernel, *X, (U - uk) / dt, periodic=periodic)
            u[:, :3] += dt / rho * d[:, :3]
            f += d
        skipped += bad
    x, Ud = cuda(torch, X), torch.as_tensor(U, device="cuda")
    got = []
    for outside in (False, True):
        ud = torch.as_tensor(u0, device="cuda")
        if outside:  # two more markers, which add nothing, first and last
            x = [torch.cat([torch.full((1,), 1.25, dtype=a.dtype, device="cuda"), a, a[:1] - 3.0]) for a in x]
            Ud = torch.cat([Ud[:, :1], Ud, Ud[:, :1]], dim=1).contiguous()
        fd, sd = ot.ot_ibm_mdf(t, kernel, *x, Ud, ud, rho, dt, rounds, slip=True)
        got.append((ud, fd))
        bits = ot.ot_last_error(t)
        assert bool(bits & ot.OT_DEV_STENCIL) == (skipped > 0) and bool(bits & ot.OT_DEV_OUTSIDE) == outside
        assert torch.all(sd.isnan()) if outside else np.abs(sd.cpu().numpy() - slip).max() <= 1e-5 * max(slip)
        assert np.array_equal(ud[:, 3].cpu().numpy(), u0[:, 3])
        for a, b in ((ud, u), (fd, f)):
            assert np.abs(a.cpu().numpy()[:, :3] - b[:, :3]).max() <= 1e-5 * np.abs(b[:, :3]).max()


def test_150000_scattered_markers(env):
    """Their sums against FP64 atomics of the same forces (the weights of which the oracle holds elsewhere)."""
    torch, ot, _, _ = env
    from paper_2605_20565_gb300 import synth
    w = synth.single_bubble(n_markers=10, n_particles=10)
    t = ot.ot_octree_build(w.spheres, w.lmin, w.lmax)
    c, r, shell = w.spheres[0, :3], w.spheres[0, 3], w.spheres[0, 4]
    rng = np.random.default_rng(11)
    n = 150_000
    d = rng.normal(size=(3, n))
    X = c[:, None] + d / np.linalg.norm(d, axis=0) * (r + rng.uniform(-0.4, 0.4, n) * shell)
    assert home_tiles(X, w.lmax, 2, False) > 4096
    F = rng.normal(size=(3, n)).astype(np.float32)
    x, Fd = cuda(torch, X), torch.as_tensor(F, device="cuda")
    N = ot.ot_octree_info(t)[0]
    want = torch.zeros((N, 4), dtype=torch.float64, device="cuda")
    ot.ot_spread_f64(t, 2, ot.OT_ATOMIC, *x, Fd.double(), want)
    for dtype, tol in ((torch.float32, 1e-5), (torch.float64, 1e-12)):
        f = torch.zeros((N, 4), dtype=dtype, device="cuda")
        spread = ot.ot_spread if dtype == torch.float32 else ot.ot_spread_f64
        spread(t, 2, ot.OT_SORTED, *x, Fd.to(dtype), f)
        assert float((f - want)[:, :3].abs().max()) <= tol * float(want[:, :3].abs().max())
