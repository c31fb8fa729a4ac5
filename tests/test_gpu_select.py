"""What the octree builder selects and lists: trees against the oracle's, bit for bit, where its
parts can go wrong -- spheres that touch cells to within rounding (the FP32 test has to leave those
to FP64), zero shells, spheres outside the cube or around all of it, level sizes around the
selection's 4096-item tiles, and refined cells that balance adds."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def cases():
    rng = np.random.default_rng(5)
    yield "touching", np.array([[0.5, 0.5, 0.5, 0.25, 0.0], [0.25, 0.25, 0.25, 0.125, 0.125]]), 1, 6
    yield "touching_far", np.array([[0.5, 0.5, 0.5, 0.0, 0.125 * np.sqrt(3.0)]]), 2, 6
    yield "by_an_ulp", np.array([[0.5, 0.5, 0.5, np.nextafter(0.25, 1.0), 0.0], [0.75, 0.5, 0.5, np.nextafter(0.125, 0.0), 0.0]]), 1, 7
    yield "around", np.array([[0.5, 0.5, 0.5, 3.0, 2.5]]), 2, 5
    yield "outside", np.array([[1.4, -0.3, 0.5, 0.6, 0.01], [1e6, 0.5, 0.5, 1e6 - 0.25, 1e-3]]), 1, 6
    yield "point", np.array([[0.123, 0.456, 0.789, 0.0, 0.0]]), 0, 9
    yield "huge", np.array([[0.5, 0.5, 0.5, 1e300, 1e300]]), 1, 4
    yield "many", np.column_stack([rng.random((40, 3)), rng.uniform(0.0, 0.1, 40), rng.uniform(0.0, 0.01, 40)]), 3, 7
    for lmin in (4, 5):  # 4096 candidates (one tile) and 32768
        yield f"tile{lmin}", np.array([[0.31, 0.52, 0.47, 0.21, 0.02]]), lmin, lmin + 2


@pytest.mark.parametrize("name,spheres,lmin,lmax", list(cases()), ids=[c[0] for c in cases()])
def test_trees(name, spheres, lmin, lmax):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import oracle
    import paper_2605_20565_gb300 as ot
    ko, lo = oracle.octree_build(spheres, lmin, lmax)
    for _ in range(2):  # the second one on recycled memory
        tree = ot.ot_octree_build(spheres, lmin, lmax)
        k, l = ot.ot_octree_copy_leaves(tree)
        assert np.array_equal(k.cpu().numpy().view(np.uint64), ko) and np.array_equal(l.cpu().numpy(), lo)
        del tree
