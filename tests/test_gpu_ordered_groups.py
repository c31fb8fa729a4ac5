"""Batches whose replays order several trilinear groups by cell, at sizes where the groups' ordered copies end
just past a 256-byte boundary (and around it): the hosts and values of the single calls, bit for bit, in
every group and replay, with hosts asked for in some groups only."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [64, 65, 128, 255, 256, 257, 258, 321, 353, 513, 4096, 4097, 4100, 30_017])
@pytest.mark.parametrize("level", [3, 8])
def test_same_as_single_calls(n, level):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2605_20565_gb300 as ot
    tree = ot.ot_octree_build(np.array([[0.5, 0.5, 0.5, 0.2, 0.05]]), 3, 6)
    ot.ot_octree_build_mates(tree)
    rng = np.random.default_rng(n)
    field = torch.as_tensor(rng.normal(size=(ot.ot_octree_info(tree)[0], 4)).astype(np.float32), device="cuda")
    groups, want = [], []
    for with_host in (False, True, True, False, True):
        x = [torch.as_tensor(rng.random(n), device="cuda") for _ in range(3)]
        h = torch.empty(n, dtype=torch.int32, device="cuda")
        want.append((ot.ot_interpolate(tree, ot.OT_TRILINEAR, *x, field, host_out=h), h))
        groups.append(dict(kernel=ot.OT_TRILINEAR, x=x[0], y=x[1], z=x[2],
                           u=torch.zeros((3, n), dtype=torch.float32, device="cuda"),
                           host=torch.full((n,), -9, dtype=torch.int32, device="cuda") if with_host else None))
    b = ot.ot_batch_create(tree, groups, field, launch=dict(order_level=level))
    for _ in range(2):
        for g in groups:
            g["u"].zero_()
        ot.ot_batch_run(b)
        for g, (u, h) in zip(groups, want):
            assert torch.equal(g["u"], u)
            assert g["host"] is None or torch.equal(g["host"], h)
