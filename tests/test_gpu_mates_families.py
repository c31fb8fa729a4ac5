"""The level-mate and parent-block tables by families of 8 sibling leaves, where the split into
families and single leaves can go wrong: trees with no family at all, of families only, of one
leaf, cells refined in some children, families at every face of the cube, clamped and periodic.
Trilinear and delta interpolation through the tables must give the bits of the per-query searches."""
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


TREES = {
    "one_leaf": (np.zeros((0, 5)), 0, 0),
    "eight": (np.zeros((0, 5)), 1, 1),
    "uniform3": (np.zeros((0, 5)), 3, 3),
    "corner": (np.array([[0.0, 0.0, 0.0, 0.01, 0.0]]), 0, 6),          # one refined child per level
    "faces": (np.array([[0.5, 0.0, 1.0, 0.2, 0.02], [0.0, 0.5, 0.5, 0.1, 0.02]]), 1, 6),
    "mixed": (np.array([[0.3, 0.6, 0.5, 0.15, 0.01], [0.7, 0.2, 0.8, 0.08, 0.0]]), 2, 7),
    "deep": (np.array([[0.4, 0.4, 0.4, 0.001, 0.0]]), 1, 12),           # deeper than the descriptors
}


@pytest.mark.parametrize("periodic", [False, True])
@pytest.mark.parametrize("name", list(TREES))
def test_tables_give_the_searches_bits(env, name, periodic):
    torch, ot, oracle = env
    spheres, lmin, lmax = TREES[name]
    ko, lo = oracle.octree_build(spheres, lmin, lmax)
    tree = ot.ot_octree_build(spheres, lmin, lmax)
    ot.ot_octree_set_periodic(tree, periodic)
    rng = np.random.default_rng(len(name))
    cen = oracle.leaf_centres(ko, lo)
    pick = rng.integers(0, ko.size, 20_000)
    half = 0.5 * 2.0 ** -lo[pick].astype(np.float64)
    P = cen[pick] + half[:, None] * rng.uniform(-1.0, 1.0, (pick.size, 3))  # in every kind of leaf
    P = np.clip(P, 0.0, np.nextafter(1.0, 0.0)).T
    x = [torch.as_tensor(np.ascontiguousarray(P[d]), device="cuda") for d in range(3)]
    field = torch.as_tensor(rng.normal(size=(ko.size, 4)), device="cuda")
    f32 = field.float()
    kernels = [1] if lmax == 0 else [1, 2, 3]
    out = []
    for table in (False, True):
        ot.ot_octree_build_mates(tree, table)
        out.append([ot.ot_interpolate(tree, k, *x, f32) for k in kernels] +
                   [ot.ot_interpolate_f64(tree, k, *x, field) for k in kernels])
    for a, b in zip(*out):
        assert torch.equal(a, b)
    host = oracle.locate_ub(ko, lo, *P)
    ref = oracle.interp_trilinear(ko, lo, f32.double().cpu().numpy(), *P, host, periodic=periodic)
    assert np.abs(out[1][0].cpu().numpy() - ref).max() <= 1e-5 * np.abs(ref).max()
