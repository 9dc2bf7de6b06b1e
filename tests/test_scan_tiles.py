"""The FP32 scan against FP64 at the edges of its row and center tiles, its chunks of
coordinates and its two block shapes (up to 40,000 rows, more): costs, labels and a round's
D^2.  An FP32 sum of d squared differences is within (d + 4) 2^-24 of the exact one (each
difference and each of the d additions rounds once, all terms >= 0), and so is a minimum of
such sums; labels are decided in FP64 where FP32 cannot tell."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

SHAPES = [  # rows, coordinates, centers
    (1, 33, 1), (31, 300, 2), (32, 96, 31), (33, 97, 33), (127, 128, 64), (129, 40, 65), (4001, 33, 130),
    (40_000, 42, 32), (40_001, 42, 33), (40_001, 100, 70), (50_003, 64, 129),
    (130, 32, 5), (4001, 7, 67),
]


@pytest.mark.gpu
@pytest.mark.parametrize("n,d,k", SHAPES)
def test_scan_at_tile_edges(n, d, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    rng = np.random.default_rng(1000 * d + k)
    X = torch.from_numpy(rng.standard_normal((n, d), dtype=np.float32)).cuda()
    C = torch.from_numpy(rng.standard_normal((k, d), dtype=np.float32)).cuda()
    X[n // 2] = C[k - 1]
    rel = (d + 4) * 2.0 ** -24
    D = torch.cdist(X.double(), C.double(), compute_mode="donot_use_mm_for_euclid_dist") ** 2
    want = D.min(1).values
    assert km.kmpar_cost(X.data_ptr(), n, d, C.data_ptr(), k) == pytest.approx(float(want.sum()), rel=rel)
    if n < 2 * k:
        return
    g = km.KMeansPar(X, k, 2.0 * k, 1, 7)
    g.round(1)
    D2, idx = g.state()
    cand, _ = g.candidates()
    R = torch.cdist(X.double(), X[cand.long()].double(), compute_mode="donot_use_mm_for_euclid_dist") ** 2
    low = R.min(1).values
    assert bool(((D2.double() - low).abs() <= rel * low).all())
    got = R.gather(1, idx.long()[:, None])[:, 0]
    assert bool((got <= low * (1 + 1e-12)).all())
    o = g.lloyd(C.clone(), 0)
    got = D.gather(1, o["labels"].long()[:, None])[:, 0]
    assert bool((got <= want * (1 + 1e-12)).all())
    assert o["final_cost"] == pytest.approx(float(want.sum()), rel=rel)
    g.close()
