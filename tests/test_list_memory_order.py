"""The buffers of the round filter and of Lloyd's lists make room for what a later call of
the context cannot do without: in whichever order the calls come, a limit under which they
all run has no higher one under which one of them is refused."""
import numpy as np
import pytest

from paper_1203_6402_gb300 import datagen

torch = pytest.importorskip("torch")

MB = 1 << 20


def _clocks(km, X, k):
    """Clocks of exactly-l rounds, after the filter's buffers."""
    g = km.KMeansPar(X, k, 1.0 * k, 2, 3, precision="bf16", sampling="exact")
    yield g
    for r in (1, 2):
        g.round(r)
    cand, w = g.candidates()
    yield cand.cpu().numpy(), w.cpu().numpy()


def _lloyd_first(km, X, k):
    """Lloyd before step 8: the candidates' labels and their transposed copy after the lists."""
    g = km.KMeansPar(X, k, 1.0 * k, 2, 3, precision="bf16")
    yield g
    for r in (1, 2):
        g.round(r)
    g.weight()
    C = X[:k].clone()
    labels = g.lloyd(C, 2)["labels"]
    km.kmpar_weighted_lloyd(g.ctx, C.data_ptr(), 1)
    seeds, _ = g.recluster()
    yield labels.cpu().numpy(), C.cpu().numpy(), seeds.cpu().numpy(), g.lloyd(seeds, 9)["labels"].cpu().numpy()


@pytest.mark.gpu
@pytest.mark.parametrize("calls", [_clocks, _lloyd_first])
def test_more_memory_refuses_no_call(monkeypatch, calls):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    monkeypatch.setenv("KMPAR_RECLUSTER_GRID", "1")   # the form that needs its transposed copy
    n, d, k = 250_007, 64, 4100
    X = torch.from_numpy(np.ascontiguousarray(datagen.gauss_mixture(n, d, k, 10.0, seed=1))).cuda()

    def run(limit):
        monkeypatch.setenv("KMPAR_CTX_LIMIT_BYTES", str(limit))
        g, out = None, None
        try:
            for out in calls(km, X, k):
                g = g or out
            return out
        except km.KmparError as e:
            assert e.status == km.KMPAR_ERR_OOM
            return None
        finally:
            if g is not None:
                g.close()

    want = run(4096 * MB)
    low = next(m for m in range(400, 40, -4) if run(m * MB) is None)
    refused = 0
    for limit in range((low + 24) * MB, (low - 16) * MB, -MB // 4):
        got = run(limit)
        if got is None:
            refused = refused or limit
            continue
        assert not refused, (limit, refused)
        assert all(np.array_equal(a, b) for a, b in zip(got, want))
    assert refused
