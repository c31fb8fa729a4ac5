"""Delta-kernel interpolation in FP64, whose weights are evaluated by all lanes whatever the warp's number of
markers and whose 3-point stencil is dealt to them by cells: marker counts around the warps' 4 and 32
with markers outside the cube among them, hosts, the stencil bit, both searches, with and without the
tables (the same bits).  Against the oracle: 1e-12 of the largest value."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [2, 3])
@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 6, 31, 32, 33, 100, 6_000])
def test_against_oracle(n, periodic, kernel):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import oracle
    import paper_2605_20565_gb300 as ot
    spheres, lmin, lmax = np.array([[0.1, 0.2, 0.1, 0.15, 0.05]]), 2, 6  # over three faces
    ko, lo = oracle.octree_build(spheres, lmin, lmax)
    tree = ot.ot_octree_build(spheres, lmin, lmax)
    ot.ot_octree_set_periodic(tree, periodic)
    ot.ot_index_train(tree, root=ot.OT_ROOT_LINEAR, n_leaf_models=64)
    rng = np.random.default_rng(n + kernel)
    v = rng.normal(size=(3, n))
    X = np.abs(spheres[0, :3, None] + (0.15 + 0.06 * rng.uniform(-1, 1, n)) * v / np.linalg.norm(v, axis=0))
    X[:, ::7] = rng.random((3, X[:, ::7].shape[1]))
    out = np.zeros(n, bool)
    if n > 4:
        out[2::5] = True
        X[1, out] = rng.choice([1.0, -0.5, np.nan], out.sum())
    field = rng.normal(size=(ko.size, 4))
    inside = np.ascontiguousarray(X[:, ~out])
    ref, bad = oracle.interp_delta(ko, lo, lmax, kernel, field, *inside, periodic=periodic)
    hosts = oracle.locate_ub(ko, lo, *inside)
    x = [torch.as_tensor(np.ascontiguousarray(X[d]), device="cuda") for d in range(3)]
    f = torch.as_tensor(field, device="cuda")
    first = None
    for table in (False, True):
        ot.ot_octree_build_mates(tree, table)
        for search in (ot.OT_BINARY, ot.OT_LEARNED):
            ot.ot_last_error(tree)
            h = torch.full((n,), -9, dtype=torch.int32, device="cuda")
            u = ot.ot_interpolate_f64(tree, kernel, *x, f, search=search, host_out=h)
            bits = ot.ot_last_error(tree)
            assert bool(bits & ot.OT_DEV_STENCIL) == (bad > 0) and bool(bits & ot.OT_DEV_OUTSIDE) == bool(out.any())
            got, hg = u.cpu().numpy(), h.cpu().numpy()
            assert np.abs(got[:, ~out] - ref).max() <= 1e-12 * np.abs(field).max()
            assert np.all(np.isnan(got[:, out])) and np.array_equal(hg[~out], hosts) and np.all(hg[out] == -1)
            first = got if first is None else first
            assert np.array_equal(got, first, equal_nan=True)
