"""Batched problems whose squared distances partly exceed FP32: a row that has no finite
distance but one (or none) still changes its center when another comes within reach.  The
labels are those that the single-problem FP32 path, which compares every row with every
center, gives for the final centers."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")


def _steps(seed):
    """Uneven groups of rows 1.3e19 apart: a center among them comes out of reach of some."""
    rng = np.random.default_rng(1000 + seed)
    d = int(rng.integers(1, 3))
    n = int(rng.integers(4096, 6000))
    k = int(rng.integers(2, 5))
    places = rng.integers(k + 1, k + 5)
    at = np.zeros((places, d))
    at[:, 0] = 1.3 * rng.permutation(2 * places)[:places]
    X = at[rng.choice(places, size=n, p=rng.dirichlet(np.full(places, 0.4)))] + rng.normal(0.0, 0.02, size=(n, d))
    return (X * 1e19).astype(np.float32), k


def _line(seed):
    """Clusters along a line of some 1e19 (FP32 squares end at 1.84e19), a few rows wide each."""
    rng = np.random.default_rng(seed)
    d = int(rng.integers(1, 4))
    n = int(rng.integers(4096, 6000))
    k = int(rng.integers(2, 9))
    places = rng.integers(k + 1, 3 * k + 3)
    at = rng.uniform(-4.0, 4.0, size=(places, d)) * np.where(np.arange(d) == 0, 1.0, 0.1)
    share = rng.dirichlet(np.full(places, 0.5))
    X = at[rng.choice(places, size=n, p=share)] + rng.normal(0.0, 0.02, size=(n, d))
    return (X * 1e19).astype(np.float32), k


@pytest.mark.gpu
@pytest.mark.parametrize("rows", [_line, _steps])
@pytest.mark.parametrize("split", [0, 3000])
def test_far_rows_follow_the_centers(split, rows):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    Xs, probs, off = [], [], dict(x=0, c=0, l=0)
    for seed in range(160):
        X, k = rows(seed)
        n, d = X.shape
        Xs.append(X)
        probs.append(dict(n=n, d=d, k=k, ell=1.0, rounds=seed % 4, max_iter=1 + seed % 7, seed=seed,
                          x_offset=off["x"], c_offset=off["c"], l_offset=off["l"], cand_offset=0))
        off["x"] += (n * d + 3) // 4 * 4 if seed % 3 else n * d
        off["c"] += k * d
        off["l"] += n
    flat = np.zeros(off["x"], dtype=np.float32)
    for p, X in zip(probs, Xs):
        flat[p["x_offset"]: p["x_offset"] + X.size] = X.ravel()
    Xd = torch.from_numpy(flat).cuda()
    C = torch.zeros(off["c"], dtype=torch.float32, device="cuda")
    L = torch.full((off["l"],), -1, dtype=torch.int32, device="cuda")
    km.kmpar_batch_set_split(split)
    try:
        res = km.kmpar_batch_run(Xd.data_ptr(), probs, C.data_ptr(), L.data_ptr())[1]
    finally:
        km.kmpar_batch_set_split(25000)
    bad, costs = [], []
    for i, (p, r, X) in enumerate(zip(probs, res, Xs)):
        if r["status"] == km.KMPAR_ERR_CAPACITY:
            continue
        n, d, k = p["n"], p["d"], p["k"]
        g = km.KMeansPar(torch.from_numpy(X).cuda(), k, 1.0, 0, 1)
        o = g.lloyd(C[p["c_offset"]: p["c_offset"] + k * d].reshape(k, d).clone(), 0)
        g.close()
        if not torch.equal(o["labels"], L[p["l_offset"]: p["l_offset"] + n]):
            bad.append((i, int((o["labels"] != L[p["l_offset"]: p["l_offset"] + n]).sum())))
        if not r["final_cost"] == pytest.approx(o["final_cost"], rel=1e-12):   # FP64 sums of the same FP32 distances
            costs.append((i, r["final_cost"], o["final_cost"]))
    assert not bad and not costs, (bad, costs)
