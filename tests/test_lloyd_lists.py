"""Lloyd's iteration by reference lists (tensor modes, rows x centers large enough): the
labels, centers, costs and iteration counts equal those of the FP32 path, which compares
every row with every center.  The data cover lists that hold and lists that overflow
(no separation, one far cluster, copies); the starting centers are the reclustering's,
and others that the candidates know nothing of."""
import numpy as np
import pytest

from paper_1203_6402_gb300 import datagen

torch = pytest.importorskip("torch")


def _far(n, d, seed):
    X = datagen.gauss_mixture(n, d, 12, 10.0, seed)
    X[: n // 50] += 3000.0
    X[n // 2: n // 2 + n // 10] = X[: n // 10]
    return X


CASES = [
    # name, rows, k, rounds, Lloyd updates, precision
    ("d64_bf16", lambda: datagen.gauss_mixture(250_007, 64, 4100, 10.0, seed=1), 4100, 1, 9, "bf16"),
    ("d20_far_and_copies", lambda: _far(500_000, 20, 2), 2048, 3, 6, "fp8"),
    ("d8_no_separation", lambda: datagen.uniform_box(400_003, 8, seed=3), 2600, 3, 5, "fp8"),
    ("d132_few_true_clusters", lambda: datagen.gauss_mixture(300_000, 132, 900, 100.0, seed=4), 3400, 2, 5, "fp8"),
]


@pytest.mark.gpu
@pytest.mark.parametrize("name,mk,k,rounds,iters,prec", CASES, ids=[c[0] for c in CASES])
def test_lloyd_lists_equal_fp32_path(name, mk, k, rounds, iters, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    Xd = torch.from_numpy(np.ascontiguousarray(mk())).cuda()
    n = len(Xd)
    other = Xd[torch.randperm(n, generator=torch.Generator().manual_seed(5))[:k].cuda()].contiguous()
    out = {}
    for p in ("fp32", prec):
        g = km.KMeansPar(Xd, k, 1.0 * k, rounds, 9, precision=p)
        for r in range(1, rounds + 1):
            g.round(r)
        g.weight()
        C, _ = g.recluster()
        res = []
        for c0 in (C, other):
            c = c0.clone()
            o = g.lloyd(c, iters, hist=True)
            res.append((o["labels"].cpu().numpy(), c.cpu().numpy(), o["iters"], o["final_cost"], o["cost_hist"]))
        out[p] = res, g.stats()
        g.close()
    for a, b in zip(out["fp32"][0], out[prec][0]):
        assert np.array_equal(a[0], b[0])
        assert np.array_equal(a[1], b[1])
        assert a[2] == b[2]
        np.testing.assert_allclose(a[4], b[4], rtol=1e-12)   # FP64 sums of the same FP32 distances
    if name in ("d64_bf16", "d132_few_true_clusters"):   # elsewhere every row may go through the dense pass
        assert out[prec][1]["lloyd_settled"] > 0
