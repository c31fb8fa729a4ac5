"""Delta-kernel interpolation by 8 lanes per marker, where its split can go wrong: marker counts
around 4 and 32, every parity of the stencil's first cell (markers in all 8 octants of all 8
children), stencils over the cube's faces (dropped or wrapped) and off the finest level, trees of
one block per axis, markers outside the cube -- with and without the parent-block table (the same
bits), in a batch and on its own.  Held to the oracle at the path's bounds, 1e-5 in FP32 and 1e-12
in FP64 of the largest value."""
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


@pytest.mark.parametrize("kernel", [2, 3])
@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("case,n", [("ball", 1), ("ball", 3), ("ball", 5), ("ball", 31), ("ball", 33), ("ball", 5000),
                                    ("lmax1", 200), ("lmax2", 200), ("lmax3", 300), ("coarse", 700)])
def test_against_oracle(env, case, n, periodic, kernel):
    torch, ot, oracle = env
    rng = np.random.default_rng(n)
    if case == "ball":
        spheres, lmin, lmax = np.array([[0.5, 0.5, 0.5, 0.2, 0.1]]), 3, 5
        v = rng.normal(size=(3, n))
        X = 0.5 + 0.2 * v / np.linalg.norm(v, axis=0)
    elif case == "coarse":  # markers everywhere in a tree that is refined near one corner
        spheres, lmin, lmax = np.array([[0.1, 0.1, 0.1, 0.1, 0.05]]), 2, 5
        X = rng.random((3, n))
    else:
        spheres, lmin = np.zeros((0, 5)), int(case[4:])
        lmax = lmin
        X = rng.random((3, n))
    ko, lo = oracle.octree_build(spheres, lmin, lmax)
    tree = ot.ot_octree_build(spheres, lmin, lmax)
    ot.ot_octree_set_periodic(tree, periodic)
    field = rng.normal(size=(ko.size, 4))
    f32 = field.astype(np.float32)
    x = [torch.as_tensor(np.ascontiguousarray(X[d]), device="cuda") for d in range(3)]
    kw = dict(periodic=True) if periodic else {}
    ref, bad = oracle.interp_delta(ko, lo, lmax, kernel, f32.astype(np.float64), *X, **kw)
    ref64, _ = oracle.interp_delta(ko, lo, lmax, kernel, field, *X, **kw)
    hosts = oracle.locate_ub(ko, lo, *X)
    outs = []
    for table in (False, True):
        ot.ot_octree_build_mates(tree, table)
        ot.ot_last_error(tree)
        h = torch.empty(n, dtype=torch.int32, device="cuda")
        g = torch.as_tensor(f32, device="cuda")
        u = ot.ot_interpolate(tree, kernel, *x, g, host_out=h)
        assert bool(ot.ot_last_error(tree) & ot.OT_DEV_STENCIL) == (bad > 0)
        u64 = ot.ot_interpolate_f64(tree, kernel, *x, torch.as_tensor(field, device="cuda"))
        ub, hb = torch.empty_like(u), torch.empty_like(h)
        batch = ot.ot_batch_create(tree, [dict(kernel=kernel, x=x[0], y=x[1], z=x[2], u=ub, host=hb)], g)
        ot.ot_batch_run(batch)
        torch.cuda.synchronize()
        assert np.abs(u.cpu().numpy() - ref).max() <= 1e-5 * np.abs(f32).max()
        assert np.abs(u64.cpu().numpy() - ref64).max() <= 1e-12 * np.abs(field).max()
        assert np.array_equal(h.cpu().numpy(), hosts)
        assert torch.equal(ub, u) and torch.equal(hb, h)
        outs.append((u, u64))
    assert torch.equal(outs[0][0], outs[1][0]) and torch.equal(outs[0][1], outs[1][1])


def test_outside(env):
    torch, ot, _ = env
    tree = ot.ot_octree_build(np.array([[0.5, 0.5, 0.5, 0.2, 0.1]]), 3, 5)
    field = torch.ones((ot.ot_octree_info(tree)[0], 4), dtype=torch.float32, device="cuda")
    X = torch.tensor([[0.7, -0.1, 0.5, 0.7], [0.5, 0.5, np.nan, 0.5], [0.5, 0.5, 0.5, 1.0]], dtype=torch.float64,
                     device="cuda")
    h = torch.empty(4, dtype=torch.int32, device="cuda")
    ot.ot_last_error(tree)
    u = ot.ot_interpolate(tree, 2, X[0], X[1], X[2], field, host_out=h).cpu().numpy()
    assert ot.ot_last_error(tree) & ot.OT_DEV_OUTSIDE
    assert np.allclose(u[:, 0], 1.0, atol=1e-6) and np.all(np.isnan(u[:, 1:]))
    assert h[0] >= 0 and torch.all(h[1:] == -1)
