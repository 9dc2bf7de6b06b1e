"""The points image at the largest dimensions that each tensor format takes, and at the
number of rows from which a warp's last block is partly or wholly empty."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

CASES = [  # format, largest d (K atoms of 128 bytes, three at most; d at most 190)
    ("bf16x3", 63), ("bf16x3", 62), ("bf16x3", 21), ("bf16x3", 42), ("bf16", 190), ("bf16", 128), ("bf16", 126),
    ("fp8", 190), ("fp8", 128),
]


@pytest.mark.gpu
@pytest.mark.parametrize("prec,d", CASES)
@pytest.mark.parametrize("n", [1, 7, 136, 1025])
def test_image_limits_equal_fp32_path(prec, d, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    rng = np.random.default_rng(n + d)
    Xh = rng.standard_normal((n, d), dtype=np.float32) * 3 + 50
    Xh[::5] *= np.float32(1e-3)   # rows of very different scales
    X = torch.from_numpy(Xh).cuda()
    k = min(n, 40)
    out = []
    for p in ("fp32", prec):
        g = km.KMeansPar(X, k, 2.0 * k, 2, 11, precision=p)
        for r in (1, 2):
            g.round(r)
        D2, idx = g.state()
        cand, w = g.candidates()
        o = g.lloyd(X[:k].clone(), 1)
        out.append([t.cpu().numpy() for t in (D2, idx, cand, w, o["labels"])])
        g.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.gpu
@pytest.mark.parametrize("prec,d", [("bf16x3", 64), ("bf16", 191), ("fp8", 191)])
def test_one_more_coordinate_is_refused(prec, d):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    X = torch.zeros(200, d, device="cuda")
    with pytest.raises(km.KmparError) as e:
        km.KMeansPar(X, 2, 4.0, 1, 1, precision=prec)
    assert e.value.status == km.KMPAR_ERR_UNSUPPORTED
