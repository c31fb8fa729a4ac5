"""The volume-weighted mean where its sums in three floats hand over to FP64: values too small or too large
for them in some leaves or all, zeros, infinities and NaN, trees from one leaf to more than one
round of every thread.  Against numpy's sums in long double: 1e-12 of the sum of the terms' magnitudes (one
block adds at most some tens of terms in a row); the subtraction is that of the mean it reports, in FP32."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("values", ["unit", "tiny", "huge", "mixed", "zeros"])
@pytest.mark.parametrize("lmin,lmax", [(0, 0), (1, 4), (3, 7), (7, 8)])
def test_mean(lmin, lmax, values):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2605_20565_gb300 as ot
    tree = ot.ot_octree_build(np.array([[0.4, 0.5, 0.6, 0.25, 0.02]])[:lmax], lmin, lmax)
    lev = ot.ot_octree_copy_leaves(tree)[1].cpu().numpy()
    n = lev.size
    rng = np.random.default_rng(n)
    f = (0.3 + rng.normal(size=(n, 4))).astype(np.float32)
    if values in ("tiny", "huge"):
        f *= np.float32(1e-30 if values == "tiny" else 1e25)
    elif values == "mixed":
        f = (f * 10.0 ** rng.choice([0, 0, 0, -20, 24, -38], (n, 1))).astype(np.float32)
    elif values == "zeros":
        f[rng.random(n) < 0.9] = 0.0
    vol = np.longdouble(8.0) ** -lev.astype(np.longdouble)
    terms = vol[:, None] * f[:, :3].astype(np.longdouble)
    want, mag = terms.sum(0), np.abs(terms).sum(0)
    d = torch.as_tensor(f, device="cuda")
    m = ot.ot_field_subtract_mean(tree, d)
    again = ot.ot_field_subtract_mean(tree, torch.as_tensor(f, device="cuda"))
    assert torch.equal(m, again)
    m = m.cpu().numpy()
    assert np.all(np.abs(m - want) <= 1e-12 * mag)
    assert np.array_equal(d.cpu().numpy()[:, 3], f[:, 3])
    sub = f[:, :3] - m.astype(np.float32)
    # the difference of the FP32 value and the mean rounded to FP32, or rounded once from FP64
    once = (f[:, :3].astype(np.float64) - m).astype(np.float32)
    got = d.cpu().numpy()[:, :3]
    assert np.all((got == sub) | (got == once))
    # not finite: the components that hold one, not the others
    if n > 8:
        g = f.copy()
        g[n // 2, 0], g[1, 1] = np.inf, np.nan
        m2 = ot.ot_field_subtract_mean(tree, torch.as_tensor(g, device="cuda")).cpu().numpy()
        assert np.isposinf(m2[0]) and np.isnan(m2[1])
        terms2 = vol * g[:, 2].astype(np.longdouble)
        assert abs(m2[2] - terms2.sum()) <= 1e-12 * np.abs(terms2).sum()
