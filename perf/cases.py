"""The work that users of this framework have it do, as cases that can be timed.

Every case goes through the public entry points of ``paper_1203_6402_gb300.kmpar``:
a whole fit (``kmpar_fit``), the seeding alone (``KMeansPar``: init, rounds,
weights, reclustering), Lloyd's iteration on a kept context, a batch of
independent problems (``kmpar_batch_run``) and the cost of given centers
(``kmpar_cost``).  Sizes are those of ``datagen.WORKLOADS``, of the benchmark's
batched recipe and of the tests, and generic ones between them.

Inputs are drawn on the GPU with the recipes of ``datagen``: a mixture of unit
Gaussians around centers ~ N(0, R I) ("gmm"), and heavy-tailed rows with integer
columns and exact copies ("kdd").

``exact`` gives the same outputs in 64 bits from plain torch, where that is quick.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1203_6402_gb300 import datagen
from paper_1203_6402_gb300 import kmpar as km


def _case(name, op, data, n, d, k, **more):
    c = dict(name=name, op=op, data=data, n=n, d=d, k=k, R=10.0, ell_factor=2.0, rounds=5, max_iter=10,
             precision="fp32", sampling="bernoulli", recluster_batch=0, weighted_iters=0, host=False)
    c.update(more)
    return c


def listed():
    return [
        # the smallest call: the cost of a few centers on a small sample (launch latency)
        _case("cost_gmm_n2k_d15_k10", "cost", "gmm", 2_000, 15, 10),
        # scoring a trained model on a data set: the FP32 nearest-center scan alone
        _case("cost_kdd_n1M_d42_k500", "cost", "kdd", 1_000_000, 42, 500),
        # the GAUSSMIXTURE configuration: a whole fit that is all launches and waits
        _case("fit_gmm_n10k_d15_k50_fp32", "fit", "gmm", 10_000, 15, 50, max_iter=100),
        # a ragged fit on CUDA cores with the options of step 4 and step 8: exactly-l
        # rounds and Lloyd's iteration on the weighted candidates
        _case("fit_gmm_n200k_d50_k300_fp32", "fit", "gmm", 200_003, 50, 300, sampling="exact", weighted_iters=5),
        # the 1e6 x 42 configuration: a whole fit of 100 Lloyd updates, split BF16
        _case("fit_kdd_n1M_d42_k500_bf16x3", "fit", "kdd", 1_000_000, 42, 500, max_iter=100, precision="bf16x3"),
        # the 4.8e6 x 42 configuration in its two halves
        _case("seed_kdd_n4.8M_d42_k1000_bf16x3", "seed", "kdd", 4_800_000, 42, 1_000, precision="bf16x3"),
        _case("lloyd_kdd_n4.8M_d42_k1000_bf16x3", "lloyd", "kdd", 4_800_000, 42, 1_000, precision="bf16x3"),
        # rows in pinned host memory, copied in and out by the call, as the end-to-end
        # measurement of the benchmark does
        _case("fit_gmm_n300k_d128_k1000_bf16_host", "fit", "gmm", 300_000, 128, 1_000, R=100.0, precision="bf16",
              host=True),
        # FP8 screening, a dimension between the tuned ones
        _case("fit_gmm_n1M_d96_k2000_fp8", "fit", "gmm", 1_000_000, 96, 2_000, R=100.0, precision="fp8"),
        # the 1e7 x 128 configuration in its two halves (step 8 in batches, as the
        # benchmark runs it): the largest work of the framework
        _case("seed_gmm_n10M_d128_k10000_bf16", "seed", "gmm", 10_000_000, 128, 10_000, R=100.0, precision="bf16",
              recluster_batch=64),
        _case("lloyd_gmm_n10M_d128_k10000_bf16", "lloyd", "gmm", 10_000_000, 128, 10_000, R=100.0, precision="bf16",
              recluster_batch=64),
        # many independent problems in one call: an eighth of the benchmark's batch
        dict(name="batch_512", op="batch", count=512, sizes=1000, n_lo=1_000, n_hi=200_000, k_lo=16, k_hi=256,
             dims="32,64,128", R=10.0, ell_factor=2.0, rounds=5, max_iter=10),
    ]


# ------------------------------------------------------------------ drawn cases
def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _evals(c) -> float:
    """Distance evaluations of the definition (Lloyd at its cap)."""
    n, k = c["n"], c["k"]
    seeding = n * (1.0 + c["rounds"] * c["ell_factor"] * k) + k * (1.0 + c["rounds"] * c["ell_factor"] * k)
    lloyd = (c["max_iter"] + 1.0) * n * k
    return {"cost": n * float(k), "fit": seeding + lloyd, "seed": seeding, "lloyd": lloyd}[c["op"]]


def draw(rng: random.Random):
    op = rng.choice(["cost", "fit", "fit", "fit", "seed", "seed", "lloyd", "lloyd", "batch"])
    if op == "batch":
        n_lo = _log_int(rng, 500, 5_000)
        k_lo = rng.randint(2, 32)
        return dict(op="batch", count=_log_int(rng, 4, 256), sizes=rng.randint(1, 10_000), n_lo=n_lo,
                    n_hi=_log_int(rng, 2 * n_lo, 100_000), k_lo=k_lo, k_hi=rng.randint(k_lo + 1, 256),
                    dims=rng.choice(["32,64,128", "15,42", "20,96,101"]),
                    R=rng.choice([4.0, 10.0, 100.0]), ell_factor=rng.choice([1.0, 2.0]), rounds=rng.randint(2, 8),
                    max_iter=rng.randint(3, 20))
    # FP32 on CUDA cores, or the benchmark's choice of the screening type for d, or FP8
    kind = "fp32" if op == "cost" else rng.choice(["fp32", "tensor", "tensor", "tensor", "fp8"])
    data = rng.choice(["gmm", "kdd"]) if kind != "fp8" else "gmm"
    for _ in range(200):
        d = _log_int(rng, 2, 160)
        if kind == "fp32":
            n, k, most = _log_int(rng, 300, 1_000_000), _log_int(rng, 2, 1_000), 1.5e11
        else:
            n, k, most = _log_int(rng, 20_000, 4_000_000), _log_int(rng, 8, 4_000), 4e12
        if data == "kdd":
            d = max(10, min(d, 60))
        c = _case("", op, data, n, min(d, 160), min(k, n // 20), R=rng.choice([4.0, 10.0, 100.0]),
                  ell_factor=rng.choice([0.5, 1.0, 2.0, 2.0, 3.0]), rounds=rng.randint(2, 8),
                  max_iter=rng.randint(3, 40))
        if c["k"] >= 2 and _evals(c) * (c["d"] + 16) <= most * 40:
            break
    c["precision"] = {"fp32": "fp32", "fp8": "fp8"}.get(kind) or ("bf16x3" if 3 * c["d"] + 2 <= 192 else "bf16")
    c["sampling"] = rng.choice(["bernoulli", "bernoulli", "bernoulli", "exact"]) if c["ell_factor"] * c["k"] >= 1 else \
        "bernoulli"
    if c["op"] != "cost":
        c["recluster_batch"] = rng.choice([0, 0, 16, 64])
    if c["op"] == "fit":
        c["weighted_iters"] = rng.choice([0, 0, 0, 3])
        c["host"] = rng.random() < 0.2
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs
def _points(c, seed: int) -> torch.Tensor:
    """The rows of a case on the GPU: the recipes of datagen with a device generator."""
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * int(seed) + 17)
    n, d = c["n"], c["d"]
    X = torch.empty(n, d, dtype=torch.float32, device="cuda")
    block = max(1, (1 << 27) // d)
    if c["data"] == "gmm":
        cen = torch.randn(c["k"], d, generator=g, device="cuda") * math.sqrt(c["R"])
        for i in range(0, n, block):
            x = X[i: i + block]
            comp = torch.randint(0, c["k"], (x.shape[0],), generator=g, device="cuda")
            torch.add(torch.randn(x.shape, generator=g, device="cuda"), cen[comp], out=x)
        return X
    d_int = min(8, d // 5)
    d_log = d - d_int
    for i in range(0, n, block):
        x = X[i: i + block]
        x[:, :d_log] = torch.exp(2.0 * torch.randn(x.shape[0], d_log, generator=g, device="cuda"))
        x[:, d_log:] = torch.randint(0, 256, (x.shape[0], d_int), generator=g, device="cuda").float()
    perm = torch.randperm(n, generator=g, device="cuda")
    dst, src = perm[: n // 5], perm[n // 5:]   # a fifth of the rows are copies of other rows
    X[dst] = X[src[torch.randint(0, src.numel(), (dst.numel(),), generator=g, device="cuda")]]
    return X


def _run_seed(seed: int) -> int:
    return 7 + 13 * int(seed)


def _seeding(c, X, seed):
    """Algorithm 2 on a new context; its candidates, weights and seed centers."""
    g = km.KMeansPar(X, c["k"], c["ell_factor"] * c["k"], c["rounds"], _run_seed(seed), precision=c["precision"],
                     sampling=c["sampling"], recluster_batch=c["recluster_batch"])
    for i in range(1, c["rounds"] + 1):
        g.round(i)
    cand, w = g.candidates()
    C, status = g.recluster()
    return g, cand, w, C, status


def _batch_sizes(c):
    """The problems of a batch: their sizes are the case's, their rows the seed's."""
    return datagen.batched_problems(c["count"], seed=c["sizes"], n_lo=c["n_lo"], n_hi=c["n_hi"], k_lo=c["k_lo"],
                                    k_hi=c["k_hi"], dims=tuple(int(v) for v in c["dims"].split(",")), R=c["R"],
                                    rounds=c["rounds"], max_iter=c["max_iter"])


def _batch_problems(c, seed):
    probs = _batch_sizes(c)
    off = 0
    for i, p in enumerate(probs):
        p["seed"], p["data_seed"] = 100_003 * int(seed) + i, 7_919 * int(seed) + i
        p["ell"] = c["ell_factor"] * p["k"]
        p["cand_offset"] = off
        off += km.kmpar_batch_cand_capacity(p["ell"], p["rounds"])
    return probs, off


def prepare(case, seed):
    c = dict(case)
    if c["op"] == "batch":
        probs, slots = _batch_problems(c, seed)
        X = torch.empty(sum(p["n"] * p["d"] for p in probs), dtype=torch.float32, device="cuda")
        g = torch.Generator(device="cuda")
        for p in probs:
            g.manual_seed(p["data_seed"])
            n, d, k = p["n"], p["d"], p["k"]
            cen = torch.randn(k, d, generator=g, device="cuda") * math.sqrt(c["R"])
            comp = torch.randint(0, k, (n,), generator=g, device="cuda")
            x = X[p["x_offset"]: p["x_offset"] + n * d].view(n, d)
            torch.add(torch.randn(n, d, generator=g, device="cuda"), cen[comp], out=x)
        return dict(case=c, X=X, probs=probs,
                    C=torch.zeros(sum(p["k"] * p["d"] for p in probs), device="cuda"),
                    labels=torch.zeros(sum(p["n"] for p in probs), dtype=torch.int32, device="cuda"),
                    cand=torch.full((slots,), -1, dtype=torch.int32, device="cuda"),
                    w=torch.zeros(slots, dtype=torch.int64, device="cuda"))
    X = _points(c, seed)
    s = dict(case=c, X=X, seed=int(seed))
    if c["op"] == "cost":
        # a model to score: rows of the data moved a little, as centroids of a few points are
        g = torch.Generator(device="cuda")
        g.manual_seed(int(seed) + 29)
        rows = torch.randperm(c["n"], generator=g, device="cuda")[: 4 * c["k"]]
        s["C"] = X[rows].view(c["k"], 4, c["d"]).mean(1).contiguous()
    elif c["op"] == "lloyd":
        # the context and the seed centers that a program has in hand before Lloyd
        s["ctx"], _, _, s["C0"], _ = _seeding(c, X, seed)
    elif c["op"] == "fit" and c["host"]:
        s["X"] = torch.empty(X.shape, dtype=torch.float32, pin_memory=True)
        s["X"].copy_(X)
    if c["op"] == "fit":
        where = dict(pin_memory=True) if c["host"] else dict(device="cuda")
        s["C"] = torch.zeros(c["k"], c["d"], dtype=torch.float32, **where)
        s["labels"] = torch.zeros(c["n"], dtype=torch.int32, **where)
    return s


# ------------------------------------------------------------------ one pass
def run(state):
    c = state["case"]
    stream = torch.cuda.current_stream()
    X = state["X"]
    if c["op"] == "cost":
        return {"cost": km.kmpar_cost(X.data_ptr(), c["n"], c["d"], state["C"].data_ptr(), c["k"],
                                      km.PRECISIONS[c["precision"]], stream.cuda_stream)}
    if c["op"] == "fit":
        flags = ((km.KMPAR_HOST_BUFFERS if c["host"] else 0) |
                 (km.KMPAR_EXACT_SAMPLING if c["sampling"] == "exact" else 0) |
                 (c["weighted_iters"] << 8) | (c["recluster_batch"] << 16))
        r = km.kmpar_fit(X.data_ptr(), c["n"], c["d"], c["k"], c["ell_factor"] * c["k"], c["rounds"],
                         _run_seed(state["seed"]), km.PRECISIONS[c["precision"]], c["max_iter"],
                         state["C"].data_ptr(), state["labels"].data_ptr(), flags, stream.cuda_stream)
        return {"centers": state["C"], "labels": state["labels"], "seed_cost": r["seed_cost"],
                "final_cost": r["final_cost"], "iters": r["iters"], "status": r["status"]}
    if c["op"] == "seed":
        g, cand, w, C, status = _seeding(c, X, state["seed"])
        D2, idx = g.state()
        g.close()
        # in buffers of a size that does not depend on the draws
        slots = km.kmpar_batch_cand_capacity(c["ell_factor"] * c["k"], c["rounds"])
        cand, w = (torch.nn.functional.pad(v, (0, slots - v.numel()), value=-1) for v in (cand, w))
        return {"D2": D2, "idx": idx, "candidates": cand, "weights": w, "centers": C, "status": status}
    if c["op"] == "lloyd":
        C = state["C0"].clone()
        r = state["ctx"].lloyd(C, c["max_iter"])
        return {"centers": C, "labels": r["labels"], "iters": r["iters"], "final_cost": r["final_cost"]}
    status, res = km.kmpar_batch_run(X.data_ptr(), state["probs"], state["C"].data_ptr(),
                                     state["labels"].data_ptr(), state["cand"].data_ptr(), state["w"].data_ptr(),
                                     stream.cuda_stream)
    return {"centers": state["C"], "labels": state["labels"], "candidates": state["cand"], "weights": state["w"],
            "m": np.array([r["m"] for r in res]), "iters": np.array([r["iters"] for r in res]),
            "seed_cost": np.array([r["seed_cost"] for r in res]),
            "final_cost": np.array([r["final_cost"] for r in res]), "status": status}


# ------------------------------------------------------------------ least work
def work(case):
    """Bytes: rows read once, outputs written once.  Flops: 2 d per distance
    evaluation of the definition (Lloyd: its first assignment only, since how many
    iterations follow depends on the data)."""
    c = dict(case)
    if c["op"] == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for p in _batch_sizes(c):
            w = work(dict(c, op="fit", n=p["n"], d=p["d"], k=p["k"]))
            total = {q: total[q] + w[q] for q in total}
        return total
    n, d, k = c["n"], c["d"], c["k"]
    out = {"cost": 8.0, "fit": 4.0 * n + 4.0 * k * d, "lloyd": 4.0 * n + 4.0 * k * d,
           "seed": 8.0 * n + 4.0 * k * d}[c["op"]]
    return {"bytes": 4.0 * n * d + (4.0 * k * d if c["op"] in ("cost", "lloyd") else 0.0) + out,
            "flops": 2.0 * d * _evals(dict(c, max_iter=0))}


# ------------------------------------------------------------------ 64 bits
_MASK = 0xFFFFFFFF


def _uniforms(count: int, rnd: int, tag: int, seed: int) -> torch.Tensor:
    """Uniforms of the counters (i, 0, rnd, tag) under key seed: Philox4x32-10."""
    c0 = torch.arange(count, dtype=torch.int64, device="cuda")
    c1 = torch.zeros_like(c0)
    c2 = torch.full_like(c0, rnd)
    c3 = torch.full_like(c0, tag)
    k0, k1 = seed & _MASK, (seed >> 32) & _MASK
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57   # the low 64 bits of each product
        n0 = ((p1 >> 32) & _MASK) ^ c1 ^ k0
        n2 = ((p0 >> 32) & _MASK) ^ c3 ^ k1
        c0, c1, c2, c3 = n0, p1 & _MASK, n2, p0 & _MASK
        k0, k1 = (k0 + 0x9E3779B9) & _MASK, (k1 + 0xBB67AE85) & _MASK
    return ((c0 >> 5).double() * 67108864.0 + (c1 >> 6).double()) / 9007199254740992.0


def _nearest(X, C):
    """Index of and squared distance to the nearest row of C for every row of X."""
    n, d = X.shape
    lab = torch.empty(n, dtype=torch.int64, device="cuda")
    d2 = torch.empty(n, dtype=torch.float64, device="cuda")
    mean = X.mean(0)
    Cm = C - mean
    cn = (Cm * Cm).sum(1)
    block = max(1, (1 << 27) // max(d, C.shape[0]))
    for i in range(0, n, block):
        x = X[i: i + block]
        lab[i: i + block] = torch.addmm(cn, x - mean, Cm.T, alpha=-2.0).argmin(1)
        t = x - C[lab[i: i + block]]
        d2[i: i + block] = (t * t).sum(1)
    return lab, d2


def _exact_seeding(c, X, seed):
    n, k, ell, key = c["n"], c["k"], c["ell_factor"] * c["k"], _run_seed(seed)
    first = min(n - 1, int(math.floor(float(_uniforms(1, 0, 1, key)[0]) * n)))
    cand = torch.tensor([first], device="cuda")
    idx = torch.zeros(n, dtype=torch.int64, device="cuda")
    D2 = ((X - X[first]) ** 2).sum(1)
    for r in range(1, c["rounds"] + 1):
        if c["sampling"] == "exact":
            t = -torch.log(_uniforms(n, r, 4, key)) / D2
            t[D2 <= 0] = math.inf
            new = torch.topk(t, min(int(ell), int((D2 > 0).sum())), largest=False).indices.sort().values
        else:
            phi = D2.sum()
            p = torch.clamp(ell * D2 / phi, max=1.0) if phi > 0 else torch.zeros_like(D2)
            new = torch.nonzero(_uniforms(n, r, 2, key) < p).flatten()
        if new.numel():
            lab, d2 = _nearest(X, X[new])
            better = d2 < D2
            idx = torch.where(better, lab + cand.numel(), idx)
            D2 = torch.where(better, d2, D2)
            cand = torch.cat([cand, new])
    w = torch.bincount(idx, minlength=cand.numel()).double()
    Y = X[cand]
    u = _uniforms(k, 0, 3, key)
    mass, near, chosen = w.clone(), torch.full_like(w, math.inf), []
    for t in range(k):
        pre = torch.cumsum(mass, 0)
        chosen.append(torch.searchsorted(pre, (u[t] * pre[-1]).reshape(1), right=True).clamp(max=len(w) - 1))
        near = torch.minimum(near, ((Y - Y[chosen[-1]]) ** 2).sum(1))
        mass = w * near
    return D2, Y, w, Y[torch.cat(chosen)]


def _exact_lloyd(X, C, max_iter, w=None):
    """Centers and the cost of each assignment (w: row weights)."""
    C, prev, costs = C.clone(), None, []
    for t in range(max_iter + 1):
        lab, d2 = _nearest(X, C)
        costs.append(float(d2.sum()))
        if t == max_iter or (prev is not None and torch.equal(lab, prev)):
            break
        prev = lab
        ww = torch.ones(len(X), dtype=torch.float64, device="cuda") if w is None else w
        tot = torch.zeros(len(C), dtype=torch.float64, device="cuda").index_add_(0, lab, ww)
        s = torch.zeros_like(C).index_add_(0, lab, X * ww[:, None])
        C = torch.where(tot[:, None] > 0, s / tot.clamp(min=1e-300)[:, None], C)
    return C, costs


def exact(case, seed):
    c = dict(case)
    # batches draw their own sequences per problem, one after another in Python; step
    # 8 in batches of draws is a sampler of its own
    if c["op"] == "batch" or c["recluster_batch"] > 0 or _evals(c) * c["d"] > 6e12:
        return None
    if c["op"] == "cost":
        s = prepare(c, seed)
        return {"cost": float(_nearest(s["X"].double(), s["C"].double())[1].sum())}
    X = _points(c, seed).double()
    D2, Y, w, C = _exact_seeding(c, X, seed)
    if c["op"] == "seed":
        return {"D2": D2, "idx": None, "candidates": None, "weights": None, "centers": C, "status": None}
    if c["op"] == "fit" and c["weighted_iters"]:
        C, _ = _exact_lloyd(Y, C, c["weighted_iters"], w)
    C, costs = _exact_lloyd(X, C, c["max_iter"])
    if c["op"] == "lloyd":
        return {"centers": C, "labels": None, "iters": None, "final_cost": costs[-1]}
    return {"centers": C, "labels": None, "seed_cost": costs[0], "final_cost": costs[-1], "iters": None,
            "status": None}
