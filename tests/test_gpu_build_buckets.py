"""The octree build's searches start from a table of its key sets' leading bits: leaves equal to the
oracle's, bit for bit, where buckets are empty (shells at the cube's corners, tiny deep ones), full
(all cells refined), one per key or absent (few keys)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

TREES = {
    "last corner": ([[0.97, 0.98, 0.96, 0.03, 0.01]], 1, 9),
    "first corner": ([[0.01, 0.02, 0.0, 0.02, 0.012]], 1, 9),
    "all refined": ([[0.5, 0.5, 0.5, 0.4, 2.0]], 2, 6),
    "deep": ([[0.3, 0.31, 0.62, 2e-4, 1e-4], [0.75, 0.2, 0.1, 1e-4, 2e-4]], 2, 14),
    "surface": ([[0.47, 0.52, 0.5, 0.3, 0.004]], 4, 8),
    "two levels": ([[0.5, 0.4, 0.6, 0.35, 0.02]], 5, 6),
}


@pytest.mark.parametrize("full", [1, 0])
@pytest.mark.parametrize("name", list(TREES))
def test_leaves(name, full):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2605_20565_gb300 as ot
    spheres, lmin, lmax = np.array(TREES[name][0]), *TREES[name][1:]
    ko, lo = oracle.octree_build(spheres, lmin, lmax, full)
    k, l = ot.ot_octree_copy_leaves(ot.ot_octree_build(spheres, lmin, lmax, full))
    assert np.array_equal(k.cpu().numpy().view(np.uint64), ko) and np.array_equal(l.cpu().numpy(), lo)
