"""Per-body sums where their split over a body's blocks can go wrong: empty bodies, one marker, sizes
around a block and a cluster, many bodies (one block each) and one large body (eight); and where
the sums in three floats hand over to FP64: coordinates outside (-1, 1) or within 1e-9 of the body's
centre at the origin, values too small, too large or not exactly multiplied in FP32, in some
of the markers or all.  Against numpy's FP64 sums of the
same terms: 1e-12 of the sum of the terms' magnitudes (n 2^-53 is 4e-11 of it at worst and about
1e-13 here)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("values", ["unit", "wide", "tiny", "huge", "mixed", "origin"])
@pytest.mark.parametrize("with_dv", [False, True])
@pytest.mark.parametrize("sizes", [[1], [0, 1, 0, 2, 255, 256, 257, 0], [2047, 2048, 2049], [300_001], [37] * 5000, [0, 0]])
def test_sums(sizes, with_dv, values):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2605_20565_gb300 as ot
    rng = np.random.default_rng(len(sizes) + sizes[0])
    start = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n, nb = int(start[-1]), len(sizes)
    X = rng.random((3, n))
    v = rng.normal(size=(3, n)).astype(np.float32)
    dV = (rng.uniform(0.5, 2.0, n) * (1e-20 if values == "tiny" else 1.0)).astype(np.float32)
    xb = rng.random((nb, 3))
    if values == "wide":
        X = 40.0 * X - 20.0
    elif values == "origin":
        X, xb = 1e-9 * X, 1e-9 * xb
    elif values in ("tiny", "huge"):
        v = v * np.float32(1e-25 if values == "tiny" else 1e25)
    elif values == "mixed":
        v = (v * 10.0 ** rng.choice([0, 0, 0, -20, 23, -30], n)).astype(np.float32)
        X = np.where(rng.random((3, n)) < 0.1, 1e-5 * X, np.where(rng.random((3, n)) < 0.05, 1.0 + X, X))
        v[:, ::7] = 0.0
    x = [torch.as_tensor(np.ascontiguousarray(X[d]), device="cuda") for d in range(3)]
    args = (*x, torch.as_tensor(v, device="cuda"), torch.as_tensor(start, device="cuda"),
            torch.as_tensor(xb, device="cuda"), 1.5)
    kw = dict(dV=torch.as_tensor(dV, device="cuda")) if with_dv else dict(w=0.25)
    lin, ang = (a.cpu().numpy() for a in ot.ot_body_sums(*args, **kw))
    again = [a.cpu().numpy() for a in ot.ot_body_sums(*args, **kw)]
    assert np.array_equal(lin, again[0]) and np.array_equal(ang, again[1])
    vw = v.astype(np.float64) * (dV.astype(np.float64) if with_dv else 0.25)
    body = np.repeat(np.arange(nb), sizes)
    cr = np.cross((X - xb[body].T).T, vw.T)
    for got, terms in ((lin, vw.T), (ang, cr)):
        ref, mag = np.zeros((nb, 3)), np.zeros((nb, 3))
        np.add.at(ref, body, terms)
        np.add.at(mag, body, np.abs(terms))
        assert np.all(np.abs(got - 1.5 * ref) <= 1e-12 * mag + 1e-300)
