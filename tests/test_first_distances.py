"""D^2 to the first center (Alg. 2 step 2) at the edges of its blocks of rows and of its
pieces of coordinates.  An FP32 sum of d squared differences is within (d + 4) 2^-24 of the
exact one (each difference and each addition rounds once, all terms >= 0)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

SHAPES = [(1, 1), (2, 64), (127, 3), (128, 63), (129, 64), (1000, 65), (257, 127), (130, 128), (4001, 129), (300, 300),
          (70_001, 42)]


@pytest.mark.gpu
@pytest.mark.parametrize("offset", [0, 1])   # rows that start at any float
@pytest.mark.parametrize("n,d", SHAPES)
def test_first_distances(n, d, offset):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    rng = np.random.default_rng(100 * d + n)
    flat = torch.from_numpy(rng.standard_normal(n * d + offset, dtype=np.float32)).cuda()
    X = flat[offset:].view(n, d)
    g = km.KMeansPar(X, 1, 2.0, 0, 7)
    D2, idx = g.state()
    cand, w = g.candidates()
    psi = g.stats()["phi"][0]
    g.close()
    want = ((X.double() - X[cand.long()].double()) ** 2).sum(1)
    assert int(w.sum()) == n and not idx.any()
    assert bool(((D2.double() - want).abs() <= (d + 4) * 2.0 ** -24 * want).all())
    assert psi == pytest.approx(float(D2.double().sum()), rel=1e-12)
