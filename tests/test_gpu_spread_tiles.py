"""The sorted spreading by 4x4x4 tiles of finest cells, where its parts can go wrong: marker counts
around the one-block sort's limit and the warps' 32 markers, one tile with a run of tens of
thousands, trees of one tile or less per axis (stencils that wrap onto their own tile), deep trees
whose tile keys are sorted in two parts, forces that are not finite, and markers outside the cube.
Tolerance: the FP32 bound of 1e-5 of the largest value that the path holds to everywhere; FP64
1e-12.  The library reads positions to 2^-53, which at level 20 is 2^-33 of a cell and more than
that bound, so there the FP64 sums are held to those of the atomic mode, which shares the weights."""
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
    return torch, ot, oracle


def check(env, spheres, lmin, lmax, X, kernel, periodic=False, seed=0):
    """FP32 and FP64 sorted spreading of X (3, n) against the oracle; two FP32 calls bit for bit."""
    torch, ot, oracle = env
    ko, lo = oracle.octree_build(spheres, lmin, lmax)
    tree = ot.ot_octree_build(spheres, lmin, lmax)
    ot.ot_octree_set_periodic(tree, periodic)
    rng = np.random.default_rng(seed)
    n = X.shape[1]
    F = rng.normal(size=(3, n)).astype(np.float32)
    dV = (rng.uniform(0.5, 2.0, n) * 2.0 ** (-3 * lmax)).astype(np.float32)
    x = [torch.as_tensor(np.ascontiguousarray(X[d]), device="cuda") for d in range(3)]
    kw = dict(periodic=True) if periodic else {}
    ref, bad = oracle.spread_delta(ko, lo, lmax, kernel, *X, F.astype(np.float64), dV=dV.astype(np.float64), **kw)
    scale = np.abs(ref[:, :3]).max()
    outs = []
    for dtype, tol in ((torch.float32, 1e-5), (torch.float32, 1e-5), (torch.float64, 1e-12)):
        f = torch.zeros((ko.size, 4), dtype=dtype, device="cuda")
        spread = ot.ot_spread if dtype == torch.float32 else ot.ot_spread_f64
        spread(tree, kernel, ot.OT_SORTED, *x, torch.as_tensor(F, device="cuda").to(dtype), f,
               dV=torch.as_tensor(dV, device="cuda").to(dtype))
        want = ref
        if dtype == torch.float64 and lmax > 10:
            want = torch.zeros_like(f)
            spread(tree, kernel, ot.OT_ATOMIC, *x, torch.as_tensor(F, device="cuda").to(dtype), want,
                   dV=torch.as_tensor(dV, device="cuda").to(dtype))
            want = want.cpu().numpy()
        assert np.abs(f.cpu().numpy()[:, :3] - want[:, :3]).max() <= tol * scale
        outs.append(f)
    assert torch.equal(outs[0], outs[1])
    assert bool(ot.ot_last_error(tree) & ot.OT_DEV_STENCIL) == (bad > 0)


BALL = np.array([[0.5, 0.5, 0.5, 0.2, 0.1]])


@pytest.mark.parametrize("kernel", [2, 3])
@pytest.mark.parametrize("n", [1, 31, 32, 33, 1024, 8191, 8192, 8193, 40_000])
def test_marker_counts(env, n, kernel):
    rng = np.random.default_rng(n)
    v = rng.normal(size=(3, n))
    check(env, BALL, 3, 5, 0.5 + 0.2 * v / np.linalg.norm(v, axis=0), kernel, seed=n)


@pytest.mark.parametrize("n", [3_000, 20_000])
def test_one_long_run(env, n):
    rng = np.random.default_rng(3)
    X = np.array([[0.7], [0.5], [0.5]]) + rng.uniform(-0.01, 0.01, (3, n))
    X[:, ::100] = 0.5 + 0.2 * np.array([[0.0], [1.0], [0.0]])  # and a second run among it
    check(env, BALL, 3, 5, X, 2)


@pytest.mark.parametrize("kernel", [2, 3])
@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("lmax", [1, 2, 3, 4])
def test_few_tiles_per_axis(env, lmax, periodic, kernel):
    """Uniform trees of 2, 4, 8 and 16 cells per axis, markers everywhere (stencils over every
    face: dropped, or wrapped)."""
    rng = np.random.default_rng(lmax)
    check(env, np.zeros((0, 5)), lmax, lmax, rng.random((3, 500)), kernel, periodic)


@pytest.mark.parametrize("n", [500, 9_000])
def test_deep_tree(env, n):
    """Level 20 around a tiny sphere: 54-bit tile keys, which do not fit beside the marker index."""
    c = np.array([0.3, 0.6, 0.45])
    r = 20.0 * 2.0 ** -20
    rng = np.random.default_rng(n)
    v = rng.normal(size=(3, n))
    check(env, np.array([[*c, r, 5.0 * 2.0 ** -20]]), 1, 20, c[:, None] + r * v / np.linalg.norm(v, axis=0), 2)


def test_forces_that_are_not_finite_stay_in_their_stencils(env):
    torch, ot, oracle = env
    tree = ot.ot_octree_build(BALL, 3, 5)
    ko, lo = oracle.octree_build(BALL, 3, 5)
    rng = np.random.default_rng(9)
    v = rng.normal(size=(3, 400))
    X = np.ascontiguousarray(0.5 + 0.2 * v / np.linalg.norm(v, axis=0))
    F = rng.normal(size=(3, 400)).astype(np.float32)
    x = [torch.as_tensor(X[d], device="cuda") for d in range(3)]

    def spread(F):
        f = torch.zeros((ko.size, 4), dtype=torch.float32, device="cuda")
        ot.ot_spread(tree, 2, ot.OT_SORTED, *x, torch.as_tensor(F, device="cuda"), f)
        return f.cpu().numpy()[:, :3]

    clean = spread(F)
    one = np.zeros((3, 400), np.float32)
    one[:, 17] = 1.0
    reached = spread(one)[:, 0] != 0
    F[0, 17], F[1, 17] = np.inf, np.nan
    got = spread(F)
    assert 0 < reached.sum() <= 64
    assert np.array_equal(got[~reached], clean[~reached])
    assert np.all(np.isinf(got[reached, 0])) and np.all(np.isnan(got[reached, 1]))
    assert np.array_equal(got[:, 2], clean[:, 2])


def test_outside_markers_add_nothing(env):
    torch, ot, _ = env
    tree = ot.ot_octree_build(BALL, 3, 5)
    X = torch.tensor([[0.7, 1.5, 0.5], [0.5, 0.5, np.nan], [0.5, 0.5, 0.5]], dtype=torch.float64, device="cuda")
    F = torch.ones((3, 3), dtype=torch.float32, device="cuda")
    n = ot.ot_octree_info(tree)[0]
    f, g = (torch.zeros((n, 4), dtype=torch.float32, device="cuda") for _ in range(2))
    ot.ot_last_error(tree)
    ot.ot_spread(tree, 2, ot.OT_SORTED, X[0], X[1], X[2], F, f)
    assert ot.ot_last_error(tree) & ot.OT_DEV_OUTSIDE
    ot.ot_spread(tree, 2, ot.OT_SORTED, X[0, :1], X[1, :1], X[2, :1], F[:, :1].contiguous(), g)
    assert torch.equal(f, g) and ot.ot_last_error(tree) == 0
