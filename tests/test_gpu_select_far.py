"""Octrees for spheres with centres so far away that squared distances leave FP32's range, and just within
it: the oracle's, bit for bit.  On an axis the FP64 distance of centre and cell rounds to the centre's
magnitude, so shells and radii of that size decide."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = {
    "covers_the_cube": [[1e25, 0.5, 0.5, 0.1, 2e25]],
    "surface_through_it": [[1e20, 0.5, 0.5, 1e20, 0.0]],
    "negative": [[-3e19, 0.5, 0.5, 3e19, 1.0]],
    "three_axes": [[2e19, -2e19, 2e19, 2e19 * 3 ** 0.5, 1e5]],
    "beyond_float": [[1e200, 0.5, 0.5, 1e200, 0.0], [0.3, 0.4, 0.5, 0.1, 0.01]],
    "never": [[1e25, 0.5, 0.5, 0.1, 1e24]],
    "largest_square": [[1.8e19, 0.5, 0.5, 1.8e19, 0.0], [0.0, 1.85e19, 0.5, 1.85e19, 0.0]],
    "overflowing_sum": [[1.2e19, 1.2e19, 1.2e19, 1.2e19 * 3 ** 0.5, 1e4]],
    "with_a_near_one": [[1e25, 0.5, 0.5, 0.1, 1e24], [0.6, 0.5, 0.4, 0.2, 0.02]],
}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("lmin", [0, 2])
def test_trees(name, lmin):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import oracle
    import paper_2605_20565_gb300 as ot
    spheres = np.array(CASES[name])
    ko, lo = oracle.octree_build(spheres, lmin, 5)
    tree = ot.ot_octree_build(spheres, lmin, 5)
    k, l = ot.ot_octree_copy_leaves(tree)
    assert np.array_equal(k.cpu().numpy().view(np.uint64), ko) and np.array_equal(l.cpu().numpy(), lo)
