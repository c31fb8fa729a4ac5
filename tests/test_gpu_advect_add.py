"""The position update of the particle step: x + d must be the FP64 sum, bit for bit, over every kind
of operand -- displacements that cancel most of the position, ties, positions next to powers of
two, displacements far below or above the position, zeros, subnormals, negatives, infinities and
NaN -- in the scalar and in the 4-particle kernel.  With first != 0, drag off and dt = 1 the
displacement is the particle's velocity itself."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 511, 513, 400_001, 400_000])
def test_positions_add_as_fp64(n):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2605_20565_gb300 as ot
    rng = np.random.default_rng(n)
    X = rng.random((3, n))
    D = (rng.normal(size=(3, n)) * 10.0 ** rng.uniform(-9, 0, (3, n))).astype(np.float32)
    kind = rng.integers(0, 12, (3, n))
    X = np.where(kind == 0, -X, X)
    X = np.where(kind == 1, 2.0 ** rng.integers(-20, 2, (3, n)) * (1.0 + rng.integers(-2, 3, (3, n)) * 2.0 ** -52), X)
    D = np.where(kind == 2, (-X * (1.0 + 1e-6 * rng.normal(size=(3, n)))).astype(np.float32), D)   # cancels
    D = np.where(kind == 3, (rng.integers(-5, 6, (3, n)) * 2.0 ** -54).astype(np.float32), D)        # ties
    D = np.where(kind == 4, 0.0, D).astype(np.float32)
    X = np.where(kind == 5, X * 10.0 ** rng.uniform(-320, 300, (3, n)), X)
    D = np.where(kind == 6, D * np.float32(1e-38), D)                                                # subnormal
    with np.errstate(over="ignore"):
        D = np.where(kind == 7, D * np.float32(1e38) * np.float32(10.0), D).astype(np.float32)       # huge, infinite
    X.ravel()[::97] = np.resize([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, 1.7976931348623157e308], X.ravel()[::97].size)
    x = torch.as_tensor(X, device="cuda")
    v = torch.as_tensor(D, device="cuda")
    z = torch.zeros_like(v)
    ot.ot_advect_ab2(x, v, z.clone(), z.clone(), v.clone(), 1.0, 0.0, 1.0, first=True)
    # the kernel's displacement is dt (3/2 v - 1/2 v) in FP32
    with np.errstate(all="ignore"):
        d = np.float32(1.5) * D
        finite = np.isfinite(d) & (np.abs(D) > 1e-37)   # 3/2 v - v/2 is v there, with or without a fused product
        ref = X + (D + np.float32(0.0)).astype(np.float64)  # (3/2 v - 1/2 v of v = -0 is +0)
    got = x.cpu().numpy()
    use = finite | (D == 0)
    assert use.mean() > 0.7 or n < 10
    assert np.array_equal(got[use].view(np.int64)[~np.isnan(ref[use])], ref[use].view(np.int64)[~np.isnan(ref[use])])
    assert np.all(np.isnan(got[use][np.isnan(ref[use])]))


@pytest.mark.parametrize("n", [400, 401])
@pytest.mark.parametrize("tau", [1e-39, 2.0 ** -40, 1e-12, 1.0, 2.0 ** 60, 1e19, 1e38])
def test_relaxation_times(tau, n):
    """One division per particle where f_p / tau is a normal number, else one per component: rel / tau
    to two roundings (2^-22), and 0 where rel is 0."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_20565_gb300 as ot
    rng = np.random.default_rng(n)
    U = (rng.normal(size=(3, n)) * (1e-6 if tau < 1e-20 else 1e6)).astype(np.float32)
    U[:, ::3] = 0.0
    x = torch.zeros((3, n), dtype=torch.float64, device="cuda")
    v = torch.zeros((3, n), device="cuda")
    ap = torch.zeros_like(v)
    ot.ot_advect_ab2(x, v, ap, torch.zeros_like(v), torch.as_tensor(U, device="cuda"), tau, 0.0, 0.0, first=True)
    ref = U.astype(np.float64) / float(np.float32(tau))
    assert np.all(np.abs(ap.cpu().numpy() - ref) <= np.abs(ref) * 2.0 ** -22)
