"""The round filter and Lloyd's lists take memory only where there is some: under a falling
limit on a context's memory the path first goes without them (same results), then refuses."""
import numpy as np
import pytest

from paper_1203_6402_gb300 import datagen

torch = pytest.importorskip("torch")


@pytest.mark.gpu
def test_lists_are_optional_under_a_memory_limit(monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    n, d, k = 250_007, 64, 4100
    X = torch.from_numpy(np.ascontiguousarray(datagen.gauss_mixture(n, d, k, 10.0, seed=1))).cuda()

    def run(limit):
        if limit:
            monkeypatch.setenv("KMPAR_CTX_LIMIT_BYTES", str(limit))
        else:
            monkeypatch.delenv("KMPAR_CTX_LIMIT_BYTES", raising=False)
        g = None
        try:
            g = km.KMeansPar(X, k, 1.0 * k, 2, 3, precision="bf16")
            for r in (1, 2):
                g.round(r)
            g.weight()
            C, _ = g.recluster()
            o = g.lloyd(C, 4)
            return o["labels"].cpu().numpy(), C.cpu().numpy(), o["final_cost"], g.stats()["lloyd_settled"]
        except km.KmparError as e:
            assert e.status == km.KMPAR_ERR_OOM
            return None
        finally:
            if g is not None:
                g.close()

    want = run(None)
    settled, refused = set(), False
    for limit in range(400 << 20, 60 << 20, -(2 << 20)):
        got = run(limit)
        if got is None:
            refused = True
            continue
        assert not refused   # what runs with less runs with more
        assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
        assert got[2] == pytest.approx(want[2], rel=1e-12)
        settled.add(got[3])
    assert refused and len(settled) > 1   # with the lists, with the bounds alone, not at all
