"""Reference lists (round filter, Lloyd) where the screened values leave their usual range:
the rounds and Lloyd's iterations equal those of the FP32 path, which compares every row
with every center."""
import numpy as np
import pytest

from paper_1203_6402_gb300 import datagen

torch = pytest.importorskip("torch")


def _same_rounds(Xd, k, ell, rounds, prec, sampling):
    from paper_1203_6402_gb300 import kmpar as km
    out = []
    for p in ("fp32", prec):
        g = km.KMeansPar(Xd, k, ell, rounds, 5, precision=p, sampling=sampling)
        per = []
        for r in range(1, rounds + 1):
            na, _ = g.round(r, sync=True)
            D2, idx = g.state()
            per.append((na, D2.cpu().numpy(), idx.cpu().numpy()))
        out.append(per)
        g.close()
    for r, (a, b) in enumerate(zip(*out)):
        assert a[0] == b[0], r + 1
        assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2]), r + 1
    return out[1]


def _same_lloyd(Xd, C0, iters, prec, ell=300.0):
    from paper_1203_6402_gb300 import kmpar as km
    k = len(C0)
    out = []
    for p in ("fp32", prec):
        g = km.KMeansPar(Xd, k, ell, 1, 9, precision=p)
        g.round(1)
        C = C0.clone()
        o = g.lloyd(C, iters, hist=True)
        out.append((o["labels"].cpu().numpy(), C.cpu().numpy(), o["iters"], np.array(o["cost_hist"])))
        g.close()
    a, b = out
    assert b[0].min() >= 0 and b[0].max() < k
    assert np.array_equal(a[0], b[0])
    assert np.array_equal(a[1], b[1], equal_nan=True)
    assert a[2] == b[2]
    np.testing.assert_allclose(a[3], b[3], rtol=1e-12)   # FP64 sums of the same FP32 distances


def _large(n, d, clusters, seed):
    """A mixture around one cluster at the mean, in units of 1e16: there a list reaches past
    the squared norm (1e30) that stands in for the columns beyond the last center."""
    X = datagen.gauss_mixture(n, d, clusters, 100.0, seed)
    at = np.arange(0, n, clusters)
    X[at] = datagen.gauss_mixture(len(at), d, 1, 0.0, seed + 1)
    return np.ascontiguousarray(X * np.float32(1e16))


# three columns short of the last tile: few enough beyond the centers for a list to hold them
@pytest.mark.gpu
@pytest.mark.parametrize("d,prec", [(64, "bf16"), (20, "fp8"), (96, "fp8")])
def test_columns_beyond_the_centers_stay_off_the_lists(d, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    X = torch.from_numpy(_large(60_000, d, 300, 1)).cuda()
    per = _same_rounds(X, 300, 1021.0, 3, prec, "exact")
    assert [p[0] for p in per] == [1021] * 3 and per[-1][2].max() <= 3 * 1021
    X = torch.from_numpy(_large(250_007, d, 4093, 2)).cuda()
    C0 = X[torch.randperm(len(X), generator=torch.Generator().manual_seed(3))[:4093].cuda()].contiguous()
    C0[7] = X[0]   # a center at the mean, whatever the draw
    _same_lloyd(X, C0, 5, prec)


# rows whose norm, or whose share of the mean, is beyond FP32: no screened value of theirs
# says anything, and no list may take that for "no center is near"
@pytest.mark.gpu
@pytest.mark.parametrize("value", [1e20, 1e30, float("inf"), float("nan")])
@pytest.mark.parametrize("d,prec", [(64, "bf16"), (128, "bf16"), (20, "fp8"), (96, "fp8")])
def test_lists_without_finite_thresholds_cover_no_row(d, prec, value):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    X = datagen.gauss_mixture(250_007, d, 4093, 10.0, 4)
    X[1234] = value
    Xd = torch.from_numpy(np.ascontiguousarray(X)).cuda()
    _same_rounds(Xd, 300, 1000.0, 4, prec, "bernoulli")
    C0 = Xd[torch.randperm(len(X), generator=torch.Generator().manual_seed(5))[:4093].cuda()].contiguous()
    if np.isfinite(value):
        C0[11] = Xd[1234]   # the row is a center, as step 8 makes it
    _same_lloyd(Xd, C0, 5, prec)
