"""Round passes that filter rows by their candidate (Alg. 2 step 5 in the tensor modes):
every round's D^2 and idx, the candidates and the weights equal those of the FP32 path,
which compares every row with every candidate.  Dimensions cover each copy width of the
list refine; the data cover lists that hold, lists that overflow (no separation, one
far cluster, copies), a round in several parts, and rounds that draw nothing."""
import numpy as np
import pytest

from paper_1203_6402_gb300 import datagen

torch = pytest.importorskip("torch")


def _far(n, d, seed):
    """Close clusters, one cluster 1,000 times farther out, and 10% copies."""
    X = datagen.gauss_mixture(n, d, 12, 10.0, seed)
    X[: n // 50] += 3000.0
    X[n // 2: n // 2 + n // 10] = X[: n // 10]
    return X


CASES = [
    # name, rows, k, l, rounds, precision (rows x draws a round are enough for the filter)
    ("d4", lambda: datagen.gauss_mixture(60011, 4, 40, 100.0, seed=1), 300, 600.0, 4, "fp8"),
    ("d16_no_separation", lambda: datagen.uniform_box(60001, 16, seed=2), 300, 600.0, 4, "fp8"),
    ("d20", lambda: datagen.gauss_mixture(80000, 20, 100, 4.0, seed=3), 100, 450.0, 5, "fp8"),
    ("d64_bf16", lambda: datagen.gauss_mixture(60000, 64, 300, 10.0, seed=4), 300, 700.0, 5, "bf16"),
    ("d96_far_and_copies", lambda: _far(90000, 96, 5), 60, 300.0, 5, "fp8"),
    ("d132", lambda: datagen.gauss_mixture(50033, 132, 50, 100.0, seed=6), 250, 600.0, 4, "fp8"),
    ("d188", lambda: datagen.gauss_mixture(50000, 188, 30, 100.0, seed=7), 200, 600.0, 3, "fp8"),
    ("d128_parts", lambda: datagen.gauss_mixture(400_001, 128, 5000, 100.0, seed=8), 5000, 15000.0, 3, "bf16"),
    ("d64_all_drawn", lambda: np.repeat(datagen.uniform_box(40, 64, seed=9), 2000, 0), 20, 300.0, 4, "bf16"),
]


@pytest.mark.gpu
@pytest.mark.parametrize("name,mk,k,ell,rounds,prec", CASES, ids=[c[0] for c in CASES])
def test_filtered_rounds_equal_fp32_path(name, mk, k, ell, rounds, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    Xd = torch.from_numpy(np.ascontiguousarray(mk())).cuda()
    n = len(Xd)
    out = {}
    for p in ("fp32", prec):
        g = km.KMeansPar(Xd, k, ell, rounds, 5, precision=p)
        per = []
        for r in range(1, rounds + 1):
            na, _ = g.round(r, sync=True)
            D2, idx = g.state()
            per.append((na, D2.cpu().numpy(), idx.cpu().numpy()))
        cand, w = g.candidates()
        out[p] = (per, cand.cpu().numpy(), w.cpu().numpy(), g.stats())
        g.close()
    for r, (a, b) in enumerate(zip(out["fp32"][0], out[prec][0])):
        assert a[0] == b[0], r + 1
        assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2]), r + 1
    assert np.array_equal(out["fp32"][1], out[prec][1]) and np.array_equal(out["fp32"][2], out[prec][2])
    # every row is counted once a round, whichever pass settles it
    assert out[prec][3]["screen_rows"] == rounds * n
