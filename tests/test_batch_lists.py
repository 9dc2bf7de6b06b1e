"""Batched problems by reference lists, a row per thread and tiles of rows (which of them:
rows, dimension, centers; one block or a cluster): candidates and weights equal those of
the single-problem FP32 path, and the labels and the cost are those which that path, which
compares every row with every center, gives for the final centers."""
import numpy as np
import pytest

from paper_1203_6402_gb300 import datagen

torch = pytest.importorskip("torch")


def _copies(n, d, seed):
    X = datagen.gauss_mixture(n, d, 9, 5.0, seed)
    X[n // 2:] = X[: n - n // 2]
    X[:50] += 500.0
    return X


PROBLEMS = [  # points, clusters, rounds, Lloyd updates
    (lambda: datagen.gauss_mixture(4095, 17, 30, 10.0, 1), 30, 3, 5),      # dense passes
    (lambda: datagen.gauss_mixture(4096, 17, 30, 10.0, 2), 30, 3, 5),      # lists, 4-byte copies
    (lambda: datagen.gauss_mixture(20_011, 64, 40, 30.0, 3), 40, 4, 9),    # lists, 16-byte copies
    (lambda: datagen.gauss_mixture(9_001, 128, 20, 100.0, 4), 24, 3, 0),
    (lambda: datagen.gauss_mixture(30_001, 127, 64, 10.0, 5), 64, 3, 7),
    (lambda: datagen.uniform_box(12_345, 5, seed=6), 50, 3, 6),            # lists overflow
    (lambda: _copies(16_000, 33, 7), 65, 2, 8),
    (lambda: datagen.gauss_mixture(40_000, 32, 256, 10.0, 8), 256, 1, 3),
    (lambda: datagen.gauss_mixture(300, 100, 4, 10.0, 9), 3, 2, 4),
    (lambda: datagen.gauss_mixture(33, 3, 2, 10.0, 10), 1, 5, 10),
]


@pytest.mark.gpu
@pytest.mark.parametrize("split", [0, 3000, 25000])   # rows per block before a problem is cut (0: never)
def test_batch_lists_equal_single_problem(split):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    Xs = [np.ascontiguousarray(mk(), dtype=np.float32) for mk, *_ in PROBLEMS]
    probs, off = [], dict(x=0, c=0, l=0, a=0)
    for (_, k, rounds, iters), X in zip(PROBLEMS, Xs):
        n, d = X.shape
        probs.append(dict(n=n, d=d, k=k, ell=2.0 * k, rounds=rounds, max_iter=iters, seed=77, x_offset=off["x"],
                          c_offset=off["c"], l_offset=off["l"], cand_offset=off["a"]))
        off["x"] += n * d
        off["c"] += k * d
        off["l"] += n
        off["a"] += km.kmpar_batch_cand_capacity(2.0 * k, rounds)
    Xd = torch.from_numpy(np.concatenate([X.ravel() for X in Xs])).cuda()
    C = torch.zeros(off["c"], dtype=torch.float32, device="cuda")
    L = torch.zeros(off["l"], dtype=torch.int32, device="cuda")
    cand = torch.full((off["a"],), -1, dtype=torch.int32, device="cuda")
    w = torch.zeros(off["a"], dtype=torch.int64, device="cuda")
    km.kmpar_batch_set_split(split)
    try:
        km.kmpar_batch_run(Xd.data_ptr(), probs, C.data_ptr(), L.data_ptr(), cand.data_ptr(), w.data_ptr())
        res = km.kmpar_batch_run(Xd.data_ptr(), probs, C.data_ptr(), L.data_ptr(), cand.data_ptr(), w.data_ptr())[1]
    finally:
        km.kmpar_batch_set_split(25000)
    for p, r, X in zip(probs, res, Xs):
        n, d, k = p["n"], p["d"], p["k"]
        g = km.KMeansPar(torch.from_numpy(X).cuda(), k, p["ell"], p["rounds"], p["seed"])
        for i in range(1, p["rounds"] + 1):
            g.round(i)
        gc, gw = g.candidates()
        m = r["m"]
        if r["sample_near"] == 0:
            assert m == len(gc), p
            assert torch.equal(cand[p["cand_offset"]: p["cand_offset"] + m], gc), p
            assert torch.equal(w[p["cand_offset"]: p["cand_offset"] + m], gw), p
        seeds, _ = g.recluster()
        final = C[p["c_offset"]: p["c_offset"] + k * d].reshape(k, d)
        if r["sample_near"] == 0 and r["recluster_near"] == 0:
            # FP64 sums of the same FP32 distances
            assert g.lloyd(seeds.clone(), 0)["final_cost"] == pytest.approx(r["seed_cost"], rel=1e-12)
        o = g.lloyd(final.clone(), 0)
        assert torch.equal(o["labels"], L[p["l_offset"]: p["l_offset"] + n]), p
        assert o["final_cost"] == pytest.approx(r["final_cost"], rel=1e-12)
        g.close()
