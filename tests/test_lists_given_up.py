"""Data that do not separate: rounds that go on without lists after a pass that left most rows
open (and try again with six times as many candidates), and Lloyd's iteration that drops them
after its first assignments.  Rounds, labels, centers and costs equal those of the FP32 path."""
import numpy as np
import pytest

from paper_1203_6402_gb300 import datagen

torch = pytest.importorskip("torch")


def _late(n, d, seed):
    """A box in which tight clusters hold two rows of three."""
    X = datagen.uniform_box(n, d, seed=seed, lo=-40.0, hi=40.0)
    X[n // 3:] = datagen.gauss_mixture(n - n // 3, d, 60, 100.0, seed + 1)
    return X


CASES = [  # rows, l, rounds, k for Lloyd, precision
    (lambda: datagen.uniform_box(60_001, 64, seed=1), 700.0, 8, 0, "bf16"),
    (lambda: datagen.uniform_box(60_000, 16, seed=2), 40.0, 9, 0, "fp8"),       # 6 times the candidates: lists again
    (lambda: _late(90_000, 96, 3), 300.0, 7, 0, "fp8"),
    (lambda: datagen.uniform_box(400_001, 128, seed=4), 12_000.0, 2, 0, "bf16"),   # a round in parts
    (lambda: datagen.uniform_box(250_007, 64, seed=5), 1000.0, 3, 4100, "bf16"),
    (lambda: _late(250_007, 20, 6), 1000.0, 1, 4100, "fp8"),
]


@pytest.mark.gpu
@pytest.mark.parametrize("mk,ell,rounds,k,prec", CASES)
def test_given_up_lists_equal_fp32_path(mk, ell, rounds, k, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    Xd = torch.from_numpy(np.ascontiguousarray(mk())).cuda()
    out = []
    for p in ("fp32", prec):
        g = km.KMeansPar(Xd, k or 20, ell, rounds, 5, precision=p)
        per = []
        for r in range(1, rounds + 1):
            na, _ = g.round(r, sync=True)
            per += [np.array(na)] + [t.cpu().numpy() for t in g.state()]
        per += [t.cpu().numpy() for t in g.candidates()]
        if k:
            C = Xd[torch.randperm(len(Xd), generator=torch.Generator().manual_seed(7))[:k].cuda()].contiguous()
            o = g.lloyd(C, 7, hist=True)
            per += [o["labels"].cpu().numpy(), C.cpu().numpy(), np.array(o["iters"])]
            cost = o["cost_hist"]
            out.append((per, cost, g.stats()))
        else:
            out.append((per, [0.0], g.stats()))
        g.close()
    for a, b in zip(out[0][0], out[1][0]):
        assert np.array_equal(a, b)
    np.testing.assert_allclose(out[0][1], out[1][1], rtol=1e-12)   # FP64 sums of the same FP32 distances
    assert out[1][2]["screen_rows"] >= rounds * len(Xd)   # every row is counted once a round (and by Lloyd's passes)
