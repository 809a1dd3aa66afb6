"""Workloads for timing the library through its public entry points.

listed() names them, draw() gives more from the same ranges, prepare() makes what a
user's program holds before the call (device inputs, a handle with its options),
run() is one pass, work() what a pass cannot do without, exact() the numeric outputs
in 64 bits by plain torch.

Five kinds:

  search   the whole PC algorithm on one data set: correlation, skeleton search,
           orientation (Phase II) -- pc_corr, pc_skeleton, pc_orient
  batch    many independent skeleton searches in one batched handle --
           pc_corr_blocks, pc_skeleton
  tests    raw CI tests given as index matrices -- pc_ci_batch
  corr64   the FP64 correlation matrix into the caller's buffer -- pc_corr_noalloc
  mlp      the proposal network's scores ("forward") or loss gradient ("grad")

The data are linear-Gaussian SEMs, X_j = sum_i a_ij X_i + eps_j, eps ~ N(0, 1): "er"
(a random order, edges Bernoulli(prob), weights +-U[0.1, 1]), "powerlaw" (in-degrees
from pmf ~ (k+1)^-gamma on 0..40, mean total degree 6) and "hub" (edges
Bernoulli(5/(p-1)) along a fixed order, then two nodes whose neighbours are replaced by
ten random others, weights +-U[0.2, 0.8]).  Graph and weights are drawn on the host, the
samples on the device.
"""
import math
import random

import numpy as np
import torch

from paper_2109_04626_gb300 import fastpc as fp

CONVENTIONAL, REVERSED = 0, 1


def listed():
    return [
        # the smallest search: a 20-variable FP64 data set; launches and latency
        dict(name="search_er20_f64", kind="search", graph="er", prob=0.2, p=20, n=1000, f64=True, alpha=0.01,
             order=REVERSED, cap=-1),
        # the simulation's sparse hub graphs: a middle size in the conventional order ...
        dict(name="search_hub55", kind="search", graph="hub", prob=0.0, p=55, n=5000, f64=False, alpha=1e-3,
             order=CONVENTIONAL, cap=-1),
        # ... and its 95-variable size in the reversed order
        dict(name="search_hub95_rev", kind="search", graph="hub", prob=0.0, p=95, n=5000, f64=False, alpha=1e-3,
             order=REVERSED, cap=-1),
        # a dense 95-variable graph, the reversed order's own ground: many high stages
        dict(name="search_dense95_rev", kind="search", graph="er", prob=0.3, p=95, n=5000, f64=False, alpha=0.01,
             order=REVERSED, cap=-1),
        # gene-network shape: 500 variables, heavy-tailed degrees, a level cap
        dict(name="search_powerlaw500", kind="search", graph="powerlaw", prob=0.0, p=500, n=10000, f64=False,
             alpha=0.01, order=CONVENTIONAL, cap=8),
        # the largest single problem: 1000 variables, 20000 samples, every level
        dict(name="search_er1000", kind="search", graph="er", prob=10.0 / 999.0, p=1000, n=20000, f64=False,
             alpha=0.01, order=CONVENTIONAL, cap=-1),
        # many independent data sets of mixed sizes at once
        dict(name="batch_64", kind="batch", count=64, p_lo=50, p_hi=400, n_lo=2000, n_hi=20000, alpha=0.01),
        # a large batch of small tests, as a caller with its own search issues them
        dict(name="tests_l3", kind="tests", p=500, n=10000, l=3, b=1 << 20, alpha=0.01),
        # fewer tests with large conditioning sets
        dict(name="tests_l14", kind="tests", p=200, n=5000, l=14, b=50001, alpha=0.01),
        # FP64 correlations of a middle-sized data set
        dict(name="corr64_p300", kind="corr64", p=300, n=8000, f64=False),
        # scoring the candidate rows of a large stage
        dict(name="mlp_forward_1m", kind="mlp", what="forward", rows=1 << 20),
        # the gradient of a large batch of training rows
        dict(name="mlp_grad_100k", kind="mlp", what="grad", rows=100003),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sparse", "sparse", "powerlaw", "hub", "hub", "dense", "batch", "tests", "tests", "corr64",
                       "mlp"])
    n = _log_int(rng, 2000, 20000)
    if kind == "sparse":
        p = _log_int(rng, 20, 950)
        return dict(kind="search", graph="er", prob=round(min(0.2, rng.uniform(5, 10) / (p - 1)), 5), p=p, n=n,
                    f64=p <= 200 and rng.random() < 0.3, alpha=0.01, order=CONVENTIONAL, cap=-1)
    if kind == "powerlaw":
        return dict(kind="search", graph="powerlaw", prob=0.0, p=_log_int(rng, 100, 500), n=_log_int(rng, 2000, 10000),
                    f64=False, alpha=0.01, order=CONVENTIONAL, cap=rng.randint(3, 8))
    if kind == "hub":
        return dict(kind="search", graph="hub", prob=0.0, p=rng.randint(15, 100), n=_log_int(rng, 2000, 10000),
                    f64=rng.random() < 0.3, alpha=1e-3, order=rng.choice([CONVENTIONAL, REVERSED]), cap=-1)
    if kind == "dense":
        return dict(kind="search", graph="er", prob=round(rng.uniform(0.2, 0.3), 3), p=rng.randint(20, 95),
                    n=_log_int(rng, 1000, 5000), f64=rng.random() < 0.3, alpha=0.01, order=REVERSED, cap=-1)
    if kind == "batch":
        p_lo = rng.randint(30, 60)
        return dict(kind="batch", count=_log_int(rng, 4, 48), p_lo=p_lo, p_hi=p_lo + rng.randint(20, 300), n_lo=2000,
                    n_hi=_log_int(rng, 4000, 16000), alpha=0.01)
    if kind == "tests":
        l = rng.randint(0, 16)
        return dict(kind="tests", p=_log_int(rng, 50, 500), n=n, l=l,
                    b=_log_int(rng, 1000, 1000000 if l <= 4 else 60000), alpha=0.01)
    if kind == "corr64":
        return dict(kind="corr64", p=_log_int(rng, 30, 500), n=_log_int(rng, 1000, 8000), f64=rng.random() < 0.5)
    return dict(kind="mlp", what=rng.choice(["forward", "grad"]), rows=_log_int(rng, 8000, 400000))


# ---- inputs -------------------------------------------------------------------

def _weights(rng, k, lo, hi):
    return rng.uniform(lo, hi, k) * np.where(rng.random(k) < 0.5, -1.0, 1.0)


def _powerlaw_gamma(p, mean_in, max_in):
    k = np.arange(max_in + 1.0)
    t = np.minimum(np.arange(p), max_in)

    def mean(gamma):
        w = (k + 1.0) ** -gamma
        return ((k * w).cumsum() / w.cumsum())[t].mean()
    lo, hi = 0.01, 6.0
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if mean(mid) > mean_in else (lo, mid)
    return 0.5 * (lo + hi)


def _sem(graph, prob, p, rng):
    """(weights p x p, strictly upper triangular along the order; order)"""
    if graph == "er":
        A = np.triu(rng.random((p, p)) < prob, 1)
        order = rng.permutation(p)
    elif graph == "powerlaw":
        k = np.arange(41)
        w = (k + 1.0) ** -_powerlaw_gamma(p, 3.0, 40)
        A = np.zeros((p, p), dtype=bool)
        order = rng.permutation(p)
        for t in range(1, p):
            pm = w[:min(40, t) + 1]
            A[rng.choice(t, size=int(rng.choice(pm.size, p=pm / pm.sum())), replace=False), t] = True
    else:
        A = np.triu(rng.random((p, p)) < 5.0 / (p - 1), 1)
        hubs = rng.choice(p, size=2, replace=False)
        A[hubs, :] = False
        A[:, hubs] = False
        for h in hubs:
            for x in rng.choice(np.delete(np.arange(p), h), size=min(10, p - 1), replace=False):
                A[min(h, x), max(h, x)] = True
        order = np.arange(p)
    W = np.zeros((p, p))
    W[A] = _weights(rng, int(A.sum()), *((0.2, 0.8) if graph == "hub" else (0.1, 1.0)))
    return W, order


def _sample(W, order, n, gen, f64):
    """n samples (device, row-major) of X = eps (I - W)^-1 along the order."""
    p = W.shape[0]
    eps = torch.randn((n, p), generator=gen, device="cuda", dtype=torch.float64)
    T = torch.eye(p, device="cuda", dtype=torch.float64) - torch.from_numpy(W).cuda()
    X = torch.empty_like(eps)
    X[:, torch.from_numpy(order).cuda()] = torch.linalg.solve_triangular(T, eps, upper=True, left=False,
                                                                         unitriangular=True)
    return X if f64 else X.float()


def _data(graph, prob, p, n, f64, seed):
    W, order = _sem(graph, prob, p, np.random.default_rng(seed))
    return _sample(W, order, n, torch.Generator(device="cuda").manual_seed(seed), f64)


def _batch_sizes(case):
    r = random.Random(case["count"])
    return [(r.randint(case["p_lo"], case["p_hi"]), r.randint(case["n_lo"], case["n_hi"]), r.uniform(0.05, 0.3))
            for _ in range(case["count"])]


def _test_indices(case, seed):
    """b random tests: distinct nodes u, v and a set of l others."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    b, p, k = case["b"], case["p"], case["l"] + 2
    # a partial shuffle of 0..p-1 per test
    ids = torch.arange(p, dtype=torch.int16, device="cuda").repeat(b, 1)
    for t in range(k):
        at = torch.randint(t, p, (b, 1), generator=gen, device="cuda")
        x, y = ids[:, t:t + 1].clone(), ids.gather(1, at)
        ids.scatter_(1, at, x)
        ids[:, t:t + 1] = y
    ids = ids[:, :k].int()
    return ids[:, :2].contiguous(), ids[:, 2:].contiguous()


def _mlp_rows(rows, seed):
    """Feature rows as the search forms them for a candidate k of a pair (u, v) --
    marginal correlations, first-order partial correlations, the test statistic
    relative to the threshold, the stage's shape -- and 0/1 labels."""
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def rand(*s):
        return torch.rand(s, generator=gen, device="cuda", dtype=torch.float64)
    c = (rand(rows, 3) * 2 - 1) ** 3 * 0.57                       # mostly weak, always jointly valid
    uv, uk, vk = c[:, 0], c[:, 1], c[:, 2]

    def first(ab, ac, bc):
        return (ab - ac * bc) / torch.sqrt((1 - ac * ac) * (1 - bc * bc))
    uv_k, uk_v, vk_u = first(uv, uk, vk), first(uk, uv, vk), first(vk, uv, uk)
    s = 40.0                                                       # sqrt(n) / q
    l = torch.randint(1, 9, (rows,), generator=gen, device="cuda").double()
    d = l + torch.randint(1, 60, (rows,), generator=gen, device="cuda").double()
    one = torch.ones_like(uv)
    f = [uv.abs(), uk.abs(), vk.abs(), (uk * vk).abs(), uv_k.abs(), uk_v.abs(), vk_u.abs(),
         (s * uv_k.abs()).clamp(max=4), (s * uv.abs()).clamp(max=4), (s * (uv.abs() - uv_k.abs())).clamp(-4, 4),
         l / d, torch.log2(d + 1) / 8, l / 16, (uv * uk * vk > 0).double(), one, 0 * one]
    y = (rand(rows) < torch.sigmoid(4 * (uk.abs() + vk.abs()) - 2)).float()
    return torch.stack(f, 1).float().contiguous(), y


def _mlp_params(seed):
    rng = np.random.default_rng(seed)
    parts = [rng.uniform(-1, 1, 128 * 16) * math.sqrt(6.0 / 16), rng.uniform(-0.1, 0.1, 128),
             rng.uniform(-1, 1, 128 * 128) * math.sqrt(6.0 / 128), rng.uniform(-0.1, 0.1, 128),
             rng.uniform(-1, 1, 128) * math.sqrt(6.0 / 128), rng.uniform(-0.1, 0.1, 1)]
    return np.concatenate(parts).astype(np.float32)


# ---- a state, a pass ----------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "search":
        p, n = case["p"], case["n"]
        X = _data(case["graph"], case["prob"], p, n, case["f64"], seed)
        pc = fp.PC(n, p, case["alpha"], case["cap"], order=case["order"])
        return dict(kind=kind, pc=pc, X=X, adj=torch.empty((p, p), dtype=torch.uint8, device="cuda"),
                    codes=torch.empty((p, p), dtype=torch.int8, device="cuda"))
    if kind == "batch":
        sizes = _batch_sizes(case)
        Xs = [_data("er", prob, p, n, False, seed * 1009 + i) for i, (p, n, prob) in enumerate(sizes)]
        pb = fp.PCBatch([n for _, n, _ in sizes], [p for p, _, _ in sizes], case["alpha"], -1, order=CONVENTIONAL)
        return dict(kind=kind, pc=pb, X=Xs, adj=torch.empty((pb.p, pb.p), dtype=torch.uint8, device="cuda"))
    if kind == "tests":
        X = _data("er", min(0.3, 8.0 / (case["p"] - 1)), case["p"], case["n"], False, seed)
        pc = fp.PC(case["n"], case["p"], case["alpha"])
        pc.corr(X)
        ij, S = _test_indices(case, seed)
        return dict(kind=kind, pc=pc, ij=ij, S=S, l=case["l"], X=X)
    if kind == "corr64":
        X = _data("er", min(0.3, 8.0 / (case["p"] - 1)), case["p"], case["n"], case["f64"], seed)
        return dict(kind=kind, X=X, C=torch.empty((case["p"], case["p"]), dtype=torch.float64, device="cuda"))
    feats, labels = _mlp_rows(case["rows"], seed)
    pc = fp.PC(1000, 20, 0.01)
    fp.pc_mlp_set_params(pc.h, _mlp_params(seed))
    return dict(kind=case["what"], pc=pc, feats=feats, labels=labels)


def run(s):
    kind = s["kind"]
    if kind == "search":
        s["pc"].corr(s["X"])
        adj, st = s["pc"].skeleton(s["adj"])
        codes, _ = s["pc"].orient(s["codes"])
        return {"adj": adj, "codes": codes, "tests": st["tests_canonical"]}
    if kind == "batch":
        s["pc"].corr_blocks(s["X"])
        adj, st = s["pc"].skeleton(s["adj"])
        return {"adj": adj, "tests": st["tests_canonical"]}
    if kind == "tests":
        r, indep, z = s["pc"].ci_batch(s["ij"], s["S"], s["l"])
        return {"r": r, "indep": indep, "z": z}
    if kind == "corr64":
        fp.pc_corr_noalloc(s["X"], s["C"])
        return {"C": s["C"]}
    if kind == "forward":
        return {"scores": fp.pc_mlp_forward(s["pc"].h, s["feats"])}
    grad, loss = fp.pc_mlp_grad(s["pc"].h, s["feats"], s["labels"])
    return {"grad": grad, "loss": loss}


def work(case):
    """Bytes and flops of one pass.  A search's CI tests depend on the data (from a few
    thousand to some 3e8 of about 40 flops) and are not counted here: its flops are the
    correlation product's."""
    kind = case["kind"]
    if kind == "search":
        p, n = case["p"], case["n"]
        return {"bytes": n * p * (8 if case["f64"] else 4) + 2 * p * p, "flops": float(n) * p * (p + 1)}
    if kind == "batch":
        sizes = _batch_sizes(case)
        total = sum(p for p, _, _ in sizes)
        return {"bytes": sum(4 * n * p for p, n, _ in sizes) + total * total,
                "flops": float(sum(n * p * (p + 1) for p, n, _ in sizes))}
    if kind == "tests":
        l, b = case["l"], case["b"]
        return {"bytes": b * (4 * (l + 2) + 8 + 1 + 4) + 4 * case["p"] ** 2,
                "flops": b * (l ** 3 / 3.0 + 2 * l * l + 6 * l + 10)}
    if kind == "corr64":
        p, n = case["p"], case["n"]
        return {"bytes": n * p * (8 if case["f64"] else 4) + 8 * p * p, "flops": float(n) * p * (p + 1)}
    macs = case["rows"] * (16 * 128 + 128 * 128 + 128)
    if case["what"] == "forward":
        return {"bytes": case["rows"] * (64 + 4), "flops": 2.0 * macs}
    return {"bytes": case["rows"] * (64 + 4), "flops": 2.0 * 3 * macs}


# ---- the same in 64 bits ------------------------------------------------------

def _corr64(X):
    X = X.double()
    X = X - X.mean(0)
    X = X / X.square().sum(0).sqrt()
    C = X.T @ X
    C.fill_diagonal_(1.0)
    return C


def _ci64(C, ij, S, n, l):
    r = []
    idx = torch.cat([S, ij], 1).long()
    for part in idx.split(1 << 16):
        M = C[part[:, :, None], part[:, None, :]]
        H = M[:, l:, l:]
        if l:
            A = M[:, :l, l:]
            H = H - A.transpose(1, 2) @ torch.linalg.solve(M[:, :l, :l], A)
        r.append(H[:, 0, 1] / torch.sqrt(H[:, 0, 0] * H[:, 1, 1]))
    r = torch.cat(r)
    return r, math.sqrt(n - l - 3) * torch.atanh(r).abs()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("search", "batch"):
        return None                                   # graphs and counts: whole numbers only
    if kind == "tests":
        X = _data("er", min(0.3, 8.0 / (case["p"] - 1)), case["p"], case["n"], False, seed)
        ij, S = _test_indices(case, seed)
        r, z = _ci64(_corr64(X), ij, S, case["n"], case["l"])
        return {"r": r, "indep": None, "z": z}
    if kind == "corr64":
        return {"C": _corr64(_data("er", min(0.3, 8.0 / (case["p"] - 1)), case["p"], case["n"], case["f64"], seed))}
    feats, labels = _mlp_rows(case["rows"], seed)
    theta = torch.from_numpy(_mlp_params(seed)).double().cuda().requires_grad_(True)
    w1, b1, w2, b2, w3, b3 = theta.split([128 * 16, 128, 128 * 128, 128, 128, 1])
    h = torch.relu(feats.double() @ w1.view(128, 16).T + b1)
    h = torch.relu(h @ w2.view(128, 128).T + b2)
    s = h @ w3 + b3
    if case["what"] == "forward":
        return {"scores": s.detach()}
    loss = torch.nn.functional.binary_cross_entropy_with_logits(s, labels.double())
    loss.backward()
    return {"grad": theta.grad, "loss": float(loss)}
