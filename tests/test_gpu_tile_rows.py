"""Batches whose tiles are not a power of two of rows, small enough that the tiles are made smaller: the
hosts and values of the single calls, bit for bit, for every form of the trilinear launch (searches,
level-mate rows, value records) and the delta kernels beside it."""
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
    import paper_2605_20565_gb300 as ot
    return torch, ot


@pytest.mark.parametrize("n", [33, 3_001, 60_000])
@pytest.mark.parametrize("tile", [3, 5, 7])
@pytest.mark.parametrize("form", ["search", "rows", "records"])
def test_same_as_single_calls(env, form, tile, n):
    torch, ot = env
    tree = ot.ot_octree_build(np.array([[0.5, 0.5, 0.5, 0.2, 0.05]]), 3, 6)
    if form != "search":
        ot.ot_octree_build_mates(tree)
    rng = np.random.default_rng(n + tile)
    field = torch.as_tensor(rng.normal(size=(ot.ot_octree_info(tree)[0], 4)).astype(np.float32), device="cuda")
    P = rng.random((3, n))
    d = rng.normal(size=(3, n))
    M = 0.5 + 0.2 * d / np.linalg.norm(d, axis=0)
    groups, want = [], []
    for kernel, X in ((ot.OT_TRILINEAR, P), (ot.OT_PESKIN4, M), (ot.OT_TRILINEAR, M)):
        x = [torch.as_tensor(np.ascontiguousarray(X[k]), device="cuda") for k in range(3)]
        h = torch.empty(n, dtype=torch.int32, device="cuda")
        want.append((ot.ot_interpolate(tree, kernel, *x, field, host_out=h), h))
        groups.append(dict(kernel=kernel, x=x[0], y=x[1], z=x[2],
                           u=torch.full((3, n), -9.0, dtype=torch.float32, device="cuda"),
                           host=torch.full((n,), -9, dtype=torch.int32, device="cuda")))
    b = ot.ot_batch_create(tree, groups, field, launch=dict(tile=tile, tri_tile=tile,
                                                            tri_records=0 if form == "records" else -1))
    for _ in range(2):
        ot.ot_batch_run(b)
    for g, (u, h) in zip(groups, want):
        assert torch.equal(g["u"], u) and torch.equal(g["host"], h)
    assert ot.ot_last_error(tree) & ot.OT_DEV_OUTSIDE == 0
