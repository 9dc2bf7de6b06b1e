"""The FP32 scan against few centers (more than 40,000 rows): costs, labels and rounds against
FP64.  An FP32 sum of d squared differences is within (d + 4) 2^-24 of the exact one, and so is
a minimum of such sums; labels are decided in FP64 where FP32 cannot tell."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("d", [33, 48, 49, 64, 65, 96, 97, 128, 129])
@pytest.mark.parametrize("k", [1, 2, 8, 9])
def test_few_centers(d, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    n = 40_129
    rng = np.random.default_rng(1000 * d + k)
    X = torch.from_numpy(rng.standard_normal((n, d), dtype=np.float32)).cuda()
    C = torch.from_numpy(rng.standard_normal((k, d), dtype=np.float32)).cuda()
    X[n // 2] = C[k - 1]
    rel = (d + 4) * 2.0 ** -24
    D = torch.cdist(X.double(), C.double(), compute_mode="donot_use_mm_for_euclid_dist") ** 2
    want = D.min(1).values
    assert km.kmpar_cost(X.data_ptr(), n, d, C.data_ptr(), k) == pytest.approx(float(want.sum()), rel=rel)
    g = km.KMeansPar(X, k, 2.0 * k, 2, 7)
    for r in (1, 2):
        g.round(r)
    D2, _ = g.state()
    cand, _ = g.candidates()
    low = (torch.cdist(X.double(), X[cand.long()].double(), compute_mode="donot_use_mm_for_euclid_dist") ** 2).min(1).values
    assert bool(((D2.double() - low).abs() <= rel * low).all())
    o = g.lloyd(C.clone(), 0)
    got = D.gather(1, o["labels"].long()[:, None])[:, 0]
    assert bool((got <= want * (1 + 1e-12)).all())
    g.close()
