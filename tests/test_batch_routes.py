"""Batched problems at the lines of the rules that choose their passes: lists or not (rows,
centers x coordinates, 16-byte rows), lists that are given up because the data do not
separate, tiles or a row per thread, launches with and without the tiles' shared memory, and
blocks of little work.  Candidates and weights equal those of the single-problem FP32 path;
labels and costs are those it gives for the final centers."""
import numpy as np
import pytest

from paper_1203_6402_gb300 import datagen

torch = pytest.importorskip("torch")

GROUPS = {
    # no problem of the call has a use for tiles or lists
    "lean": [(4095, 64, 30, 3, 3), (5000, 3, 40, 3, 4), (300, 128, 40, 2, 4), (12_000, 15, 60, 2, 3), (4096, 21, 5, 3, 3)],
    # the same kinds beside problems that have
    "mixed": [(4095, 64, 30, 3, 3), (4096, 64, 16, 3, 5), (9000, 128, 63, 2, 3), (9000, 128, 64, 3, 3),
              (6000, 30, 512, 1, 2), (8200, 101, 90, 3, 4), (700, 40, 200, 2, 3), (20_000, 3, 256, 3, 3)],
    "few": [(30_001, 4, 3, 3, 6)],
}


@pytest.mark.gpu
@pytest.mark.parametrize("group", GROUPS)
@pytest.mark.parametrize("kind", ["mixture", "box"])   # lists that hold, lists given up
def test_batch_routes_equal_single_problem(kind, group):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1203_6402_gb300 import kmpar as km
    Xs, probs, off = [], [], dict(x=0, c=0, l=0, a=0)
    for i, (n, d, k, rounds, iters) in enumerate(GROUPS[group]):
        X = datagen.gauss_mixture(n, d, k, 50.0, 10 + i) if kind == "mixture" else datagen.uniform_box(n, d, seed=10 + i)
        Xs.append(np.ascontiguousarray(X))
        probs.append(dict(n=n, d=d, k=k, ell=2.0 * k, rounds=rounds, max_iter=iters, seed=5 + i, x_offset=off["x"],
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
    res = km.kmpar_batch_run(Xd.data_ptr(), probs, C.data_ptr(), L.data_ptr(), cand.data_ptr(), w.data_ptr())[1]
    for p, r, X in zip(probs, res, Xs):
        n, d, k, a0, m = p["n"], p["d"], p["k"], p["cand_offset"], r["m"]
        g = km.KMeansPar(torch.from_numpy(X).cuda(), k, p["ell"], p["rounds"], p["seed"])
        for i in range(1, p["rounds"] + 1):
            g.round(i)
        gc, gw = g.candidates()
        if r["sample_near"] == 0:
            assert m == len(gc) and torch.equal(cand[a0: a0 + m], gc) and torch.equal(w[a0: a0 + m], gw), p
        o = g.lloyd(C[p["c_offset"]: p["c_offset"] + k * d].reshape(k, d).clone(), 0)
        assert torch.equal(o["labels"], L[p["l_offset"]: p["l_offset"] + n]), p
        assert o["final_cost"] == pytest.approx(r["final_cost"], rel=1e-12)   # FP64 sums of the same FP32 distances
        g.close()
