"""Trilinear calls with few points against the leaves compute only the cell means they read; they must
give the bits of a call that computes all of them (the same points among enough others to pass the
limit of 8 n + 2.4 million leaves), in FP32 and FP64, with hosts searched and given, and for
points outside the cube."""
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
    # about 6M leaves of levels 3 to 10: refined level-mates in the dense pyramid and on two node levels
    tree = ot.ot_octree_build(np.array([[0.42, 0.55, 0.5, 0.2, 0.0035], [0.8, 0.2, 0.7, 0.02, 0.004]]), 3, 10)
    assert ot.ot_octree_info(tree)[0] > 3_000_000
    return torch, ot, tree


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("given", [False, True])
@pytest.mark.parametrize("n", [1, 33, 20_000])
def test_same_bits_as_all_means(env, n, given, fp64):
    torch, ot, tree = env
    N = ot.ot_octree_info(tree)[0]
    rng = np.random.default_rng(n)
    c = np.array([[0.42], [0.55], [0.5]])
    d = rng.normal(size=(3, n))
    P = c + d / np.linalg.norm(d, axis=0) * 0.2 * (1.0 + rng.normal(size=n) * 0.1)  # across the shell's steps
    P[:, ::5] = rng.random((3, P[:, ::5].shape[1]))
    P[0, 7::50] = 1.5
    more = rng.random((3, N // 8))
    dtype = torch.float64 if fp64 else torch.float32
    field = torch.as_tensor(rng.normal(size=(N, 4)), device="cuda").to(dtype)
    interpolate = ot.ot_interpolate_f64 if fp64 else ot.ot_interpolate

    def run(Q):
        x = [torch.as_tensor(np.ascontiguousarray(Q[k]), device="cuda") for k in range(3)]
        h = ot.ot_locate(tree, *x) if given else None
        return interpolate(tree, ot.OT_TRILINEAR, *x, field, host_in=h)[:, :n].contiguous()

    few, all_ = run(P), run(np.concatenate([P, more], axis=1))
    assert torch.equal(few.isnan(), all_.isnan())
    assert torch.equal(torch.nan_to_num(few), torch.nan_to_num(all_))
