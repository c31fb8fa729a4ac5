"""The radix sort behind ot_points_morton_order (and the spreading and the index training) at the
edges of its 4096-key tiles: whole and ragged last tiles, one key more than a tile, every pass
count (1 to 8 digits), digits that all coincide, and points outside the cube.  The permutation must
be numpy's stable order of the same cell keys."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 255, 4095, 4096, 4097, 8192, 12289, 300_001])
@pytest.mark.parametrize("level,clump", [(1, False), (3, False), (8, False), (8, True), (14, False)])
def test_order_at_tile_edges(n, level, clump):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2605_20565_gb300 as ot
    rng = np.random.default_rng(n * 31 + level)
    P = 0.3 + 1e-9 * rng.random((3, n)) if clump else rng.random((3, n))
    P[:, ::17] = np.where(rng.random((3, P[:, ::17].shape[1])) < 0.1, 1.5, P[:, ::17])  # some outside
    cell = np.floor(np.clip(P, 0.0, np.nextafter(1.0, 0.0)) * 2.0 ** level).astype(np.uint64)
    key = np.zeros(n, np.uint64)
    for b in range(level):
        for d in range(3):
            key |= ((cell[d] >> np.uint64(b)) & np.uint64(1)) << np.uint64(3 * b + d)
    key[np.any(P >= 1.0, axis=0)] = np.uint64((1 << (3 * level)) - 1)
    x, y, z = (torch.as_tensor(np.ascontiguousarray(P[d]), device="cuda") for d in range(3))
    perm = ot.ot_points_morton_order(x, y, z, level).cpu().numpy()
    assert np.array_equal(perm, np.argsort(key, kind="stable"))
