"""Step 8 one draw at a time where the cluster form's plan changes: CTAs that hold fewer than
512 candidates, and more of them where that brings all coordinates into shared memory."""
import numpy as np
import pytest

from paper_1203_6402_gb300 import datagen

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("n,d,k,ell,rounds", [(200, 600, 12, 20.0, 3), (900, 300, 40, 100.0, 3), (600, 1500, 10, 20.0, 3),
                                              (2500, 109, 50, 250.0, 2), (4000, 128, 60, 600.0, 3), (40, 108, 5, 1.0, 1)])
def test_small_candidate_sets_of_many_coordinates(orc, n, d, k, ell, rounds):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    X = datagen.gauss_mixture(n, d, 8, 10.0, seed=n + d)
    g = km.KMeansPar(torch.from_numpy(X).cuda(), k, ell, rounds, 11)
    for r in range(1, rounds + 1):
        g.round(r)
    cand, w = g.candidates()
    C, status = g.recluster()
    near = g.stats()["recluster_near"]
    g.close()
    rows = cand.cpu().numpy()
    chosen, rnear, warn = orc.recluster(X[rows].astype(np.float64), w.cpu().numpy(), k, 11)
    assert (status == km.KMPAR_WARN_FEW_CANDIDATES) == warn
    same = np.all(C.cpu().numpy() == X[rows[chosen]], axis=1)
    # the trajectories may part only at a draw that either side reports as a near tie
    assert same.all() or near > 0 or rnear.any(), int(np.argmin(same))
