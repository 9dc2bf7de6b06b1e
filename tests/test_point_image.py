"""The tensor formats' image of the points at the edges of its row blocks and of its
16-byte pieces: every format's rounds and labels equal those of the FP32 path."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["bf16", "bf16x3", "fp8"])
@pytest.mark.parametrize("n,d", [(129, 1), (1000, 7), (1023, 16), (2049, 33), (777, 63), (1281, 65), (640, 130), (1500, 256)])
def test_image_edges_equal_fp32_path(prec, n, d):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    rng = np.random.default_rng(n + d)
    Xh = rng.standard_normal((n, d), dtype=np.float32) * 3 + 50
    Xh[::7] *= np.float32(1e-3)   # rows of very different scales
    Xh[n // 3] = 0
    X = torch.from_numpy(Xh).cuda()
    k = 40
    out = []
    for p in ("fp32", prec):
        try:
            g = km.KMeansPar(X, k, 2.0 * k, 2, 11, precision=p)
        except km.KmparError:
            assert p != "fp32"
            pytest.skip("a format that does not take this dimension")
        for r in (1, 2):
            g.round(r)
        D2, idx = g.state()
        cand, w = g.candidates()
        o = g.lloyd(X[:k].clone(), 1)
        out.append([t.cpu().numpy() for t in (D2, idx, cand, w, o["labels"])])
        g.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
