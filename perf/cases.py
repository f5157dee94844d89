"""The work that this library's users have it do, as measurable cases.

A case is a dict of plain values; ``op`` names the public entry point:

  eval        ``deoct_eval_population``: class counts and errors of P trees
  encode      ``deoct_encode`` (uint16 ranks) or, with width 0, ``encode_dataset``
              (the width picked from the data)
  fit         ``deoct_fit_subtree``: one DEOCT run
  fit_mh      ``deoct_fit_moving_horizon`` (batched level solves) on a resident set
  request     what the server does with one fit request: encode, then the batched fit
  classifier  ``MHDEOCTClassifier.fit``: the paper's Normal preset, both warm starts
  predict     ``deoct_predict`` on raw values, with the count of correct ones

Features are i.i.d. Uniform(0,1) on a grid ("grid", ``levels`` distinct values), half
uniform and half log-normal ("mixed"), or a Gaussian mixture ("gmm"); labels follow a
planted axis-aligned tree (a mixture's labels: its component) with some flipped.
"""
import math

import numpy as np
import torch

from paper_2311_06952_gb300 import deoct
from paper_2311_06952_gb300.estimator import MHDEOCTClassifier

DEV = "cuda"


def listed():
    return [
        # scoring a small population on a small set: one launch, latency alone
        dict(name="eval_tiny", op="eval", n=1000, F=8, K=2, data="grid", levels=1000, flips=0.05,
             width=2, P=64, depth=2, subset=False),
        # the population-evaluation workload: a few hundred candidate trees on 1e5 samples
        dict(name="eval_population", op="eval", n=100_000, F=20, K=3, data="gmm", levels=0, flips=0.10,
             width=4, P=256, depth=3, subset=False),
        # counts of one fitted tree over a large resident set (reporting, leaf statistics)
        dict(name="eval_one_tree", op="eval", n=10_000_000, F=10, K=2, data="grid", levels=60_000,
             flips=0.02, width=2, P=1, depth=4, subset=False),
        # one generation of a deep-tree DEOCT (a depth-8 warm start) on wide continuous data
        dict(name="eval_deep", op="eval", n=1_000_003, F=28, K=2, data="gmm", levels=0, flips=0.05,
             width=4, P=100, depth=8, subset=False),
        # encoding a large set with ties (the large-scale workload)
        dict(name="encode_large", op="encode", n=10_000_000, F=10, K=2, data="grid", levels=60_000,
             flips=0.02, width=2),
        # encoding a serving request: continuous values, width picked by the library
        dict(name="encode_request", op="encode", n=200_003, F=33, K=5, data="gmm", levels=0, flips=0.05,
             width=0),
        # the smallest fit: launches and host work
        dict(name="fit_tiny", op="fit", n=1000, F=8, K=2, data="grid", levels=1000, flips=0.05, width=2,
             P=64, G=100, depth=2, dither=False, cr=0.9),
        # the large-scale DEOCT workload
        dict(name="fit_large", op="fit", n=10_000_000, F=10, K=2, data="grid", levels=60_000, flips=0.02,
             width=2, P=1024, G=50, depth=4, dither=False, cr=0.9),
        # the batched moving-horizon workload
        dict(name="fit_mh", op="fit_mh", n=1_000_000, F=30, K=4, data="mixed", levels=0, flips=0.05,
             width=4, P=128, G=200, depth=8, horizon=3),
        # an ordinary serving request from features to tree
        dict(name="request", op="request", n=60_001, F=24, K=5, data="gmm", levels=0, flips=0.05, width=0,
             P=128, G=200, depth=5, horizon=3),
        # the estimator as a user calls it, warm starts included
        dict(name="classifier", op="classifier", n=150_001, F=18, K=2, data="gmm", levels=0, flips=0.05,
             depth=4, warm=True),
        # prediction and score on unseen rows with a deep tree
        dict(name="predict", op="predict", n=2_750_000, F=28, K=2, data="gmm", levels=0, flips=0.05, depth=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["eval"] * 5 + ["encode"] * 3 + ["fit"] * 3 + ["fit_mh"] * 2
                    + ["request", "request", "classifier", "predict", "predict"])
    n, F, K = _log(rng, 1_000, 8_000_000), _log(rng, 4, 60), rng.randint(2, 10)
    data = rng.choice(["grid", "gmm", "mixed"])
    if op in ("request", "classifier", "fit_mh"):
        n = _log(rng, 1_000, 600_000)
    if n * F > 200_000_000:
        n = 200_000_000 // F
    levels = min(n, _log(rng, 100, 65_536)) if data == "grid" else 0
    c = dict(op=op, n=n, F=F, K=K, data=data, levels=levels, flips=rng.choice([0.02, 0.05, 0.1]))
    width = 2 if (data == "grid" or n <= 65_536) and rng.random() < 0.8 else 4
    if op == "eval":
        depth = rng.choice([1, 2, 3, 3, 4, 4, 5, 6, 8])
        P = _log(rng, 1, min(1024, max(2.0, 4e9 / (n * depth))))
        c.update(width=width, P=P, depth=depth, subset=rng.random() < 0.2)
    elif op == "encode":
        c.update(width=2 if width == 2 and data == "grid" else 0)
    elif op == "fit":
        depth = rng.choice([2, 3, 4, 5])
        P = _log(rng, 32, 1024)
        n = c["n"] = min(n, max(1_000, int(1e11 / (P * depth * 50))))
        c["levels"] = min(c["levels"], n)
        c.update(width=2 if data == "grid" or n <= 65_536 else 4, P=P, depth=depth,
                 G=max(5, min(200, int(1e11 / (n * P * depth)))), dither=rng.random() < 0.5,
                 cr=rng.choice([0.1, 0.9]))
    elif op == "fit_mh":
        c.update(width=2 if data == "grid" or n <= 65_536 else 4, P=rng.choice([64, 100, 128]),
                 G=rng.choice([100, 200]), depth=rng.randint(2, 7), horizon=rng.choice([2, 3]))
    elif op == "request":
        c.update(width=0, P=128, G=200, depth=rng.randint(2, 6), horizon=rng.choice([2, 3]))
    elif op == "classifier":
        c["n"] = min(c["n"], 200_000)
        c["levels"] = min(c["levels"], c["n"])
        c.update(depth=rng.choice([2, 3, 4]), warm=rng.random() < 0.7)
    else:
        c.update(depth=rng.randint(2, 8))
    return c


# ---------------------------------------------------------------------------
# inputs (the seed alone decides them)
# ---------------------------------------------------------------------------

def _gen(seed, salt):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 1009 + salt)


def _features(case, seed):
    """X [n][F] float32 and each row's mixture component (None: no mixture)."""
    n, F, K = case["n"], case["F"], case["K"]
    g = _gen(seed, 1)
    if case["data"] == "gmm":
        comp = torch.randint(0, K, (n,), generator=g, device=DEV)
        means = torch.randn(K, F, generator=g, device=DEV) * 2.0
        return torch.randn(n, F, generator=g, device=DEV).add_(means[comp]), comp
    X = torch.rand(n, F, generator=g, device=DEV)
    if case["data"] == "grid":
        q = float(case["levels"])
        return X.mul_(q).floor_().div_(q), None
    h = F // 2
    X[:, h:] = torch.randn(n, F - h, generator=g, device=DEV).exp_()
    return X, None


def _labels(case, seed, X, comp):
    n, F, K = case["n"], case["F"], case["K"]
    g = _gen(seed, 2)
    if comp is not None:
        y = comp.clone()
    else:  # a planted depth-4 tree: random features, thresholds at medians of a sample of rows
        depth = 4
        node = torch.ones(n, dtype=torch.int64, device=DEV)
        feats = torch.randint(0, F, (1 << depth,), generator=g, device=DEV)
        part = X[:: max(1, n // 8192)]
        thr = torch.zeros(1 << depth, device=DEV)
        pn = torch.ones(part.shape[0], dtype=torch.int64, device=DEV)
        for d in range(depth):
            for t in range(1 << d, 2 << d):
                v = part[pn == t, feats[t]]
                thr[t] = v.median() if v.numel() else 0.5
            pn = 2 * pn + (part.gather(1, feats[pn][:, None])[:, 0] >= thr[pn]).long()
            node = 2 * node + (X.gather(1, feats[node][:, None])[:, 0] >= thr[node]).long()
        leaf = torch.randperm(1 << depth, generator=g, device=DEV) % K
        y = leaf[node - (1 << depth)]
    hit = torch.rand(n, generator=g, device=DEV) < case["flips"]
    shift = torch.randint(1, K, (n,), generator=g, device=DEV)
    return torch.where(hit, (y + shift) % K, y).to(torch.uint8)


def _trees(case, seed, n_unique):
    """P random trees: features 0 (no split) .. F, threshold ranks uniform over the values."""
    P, B, F = case["P"], (1 << case["depth"]) - 1, case["F"]
    g = _gen(seed, 3)
    a = torch.randint(0, F + 1, (P, B), generator=g, device=DEV)
    u = torch.rand(P, B, generator=g, device=DEV, dtype=torch.float64)
    th = (u * n_unique.long()[(a - 1).clamp(min=0)].double()).long()
    th = torch.where(a > 0, th, torch.zeros_like(th))
    return a.to(torch.int16), th.to(torch.int32)


def _subset(case, seed):
    """A sorted random half of the samples (a node's subset), or None."""
    if not case.get("subset"):
        return None
    keep = torch.rand(case["n"], generator=_gen(seed, 4), device=DEV) < 0.5
    keep[0] = True
    return keep.nonzero()[:, 0].to(torch.int32)


def _raw_tree(case, seed, X):
    """One tree in raw units: features, float64 thresholds between data values, leaf classes."""
    B, n, F = (1 << case["depth"]) - 1, case["n"], case["F"]
    g = _gen(seed, 5)
    a = torch.randint(0, F + 1, (B,), generator=g, device=DEV)
    r = torch.randint(0, n, (2, B), generator=g, device=DEV)
    col = (a - 1).clamp(min=0)
    b = (X[r[0], col].double() + X[r[1], col].double()) * 0.5
    b = torch.where(a > 0, b, torch.zeros_like(b))
    leaf = torch.randint(0, case["K"], (B + 1,), generator=g, device=DEV).to(torch.uint8)
    return a.to(torch.int16), b, leaf


def _params(case):
    flags = deoct.DEOCT_BATCHED if case["op"] != "fit" else 0
    if case.get("dither"):
        flags |= deoct.DEOCT_DITHER_M
    return deoct.make_params(case["depth"], case["P"], case["G"], cr=case.get("cr", 0.9), seed=0,
                             horizon=case.get("horizon", 0), flags=flags)


def prepare(case, seed):
    op = case["op"]
    st = dict(op=op)
    X, comp = _features(case, seed)
    y = _labels(case, seed, X, comp)
    if op == "classifier":
        warm = ("cart", "deoct") if case["warm"] else ()
        st.update(X=X, y=y, K=case["K"], clf=MHDEOCTClassifier(depth=case["depth"], preset="normal",
                                                               warm_starts=warm))
        return st
    st["ctx"] = ctx = deoct.Context(torch.cuda.current_device())
    if op == "predict":
        a, b, leaf = _raw_tree(case, seed, X)
        st.update(X=X, y=y, a=a, b=b, leaf=leaf, depth=case["depth"])
    elif op in ("encode", "request"):
        st.update(X=X, y=y, K=case["K"], n=case["n"], width=case["width"])
        if op == "request":
            st["params"] = _params(case)
    else:
        st["ds"] = ds = deoct.encode_dataset(ctx, X, y, case["K"], case["width"])
        if op == "eval":
            st["a"], st["theta"] = _trees(case, seed, ds.n_unique)
            st.update(depth=case["depth"], idx=_subset(case, seed))
        else:
            st["params"] = _params(case)
            if op == "fit":
                st["pop"] = torch.empty(case["P"], 2 * ((1 << case["depth"]) - 1), dtype=torch.float32,
                                        device=DEV)
        ctx.release_scratch()  # the encoder's: the set is encoded once
    return st


def run(st):
    op = st["op"]
    if op == "eval":
        return deoct.deoct_eval_population(st["ctx"], st["ds"], st["a"], st["theta"], st["depth"],
                                           sample_idx=st["idx"])
    if op == "encode":
        if st["width"] == 2:
            ranks, nu = deoct.deoct_encode(st["ctx"], st["X"], 2)
            width = 2
        else:
            ds = deoct.encode_dataset(st["ctx"], st["X"], st["y"], st["K"], 0)
            ranks, nu, width = ds.ranks, ds.n_unique, ds.rank_bytes
        return ranks[:, : st["n"]], nu, width  # (a row's columns past n are padding)
    if op == "fit":
        a, theta, fit = deoct.deoct_fit_subtree(st["ctx"], st["ds"], st["params"], pop_out=st["pop"])
        return a, theta, fit, st["pop"]
    if op == "fit_mh":
        return deoct.deoct_fit_moving_horizon(st["ctx"], st["ds"], st["params"])
    if op == "request":
        ds = deoct.encode_dataset(st["ctx"], st["X"], st["y"], st["K"], 0)
        return deoct.deoct_fit_moving_horizon(st["ctx"], ds, st["params"])
    if op == "classifier":
        return st["clf"].fit(st["X"], st["y"], K=st["K"]).tree_
    return deoct.deoct_predict(st["ctx"], st["X"], st["a"], st["b"], st["depth"], st["leaf"], y=st["y"])


# ---------------------------------------------------------------------------
# the work of one pass, and what it has to return
# ---------------------------------------------------------------------------

def _ops(depth):
    """Integer operations of one (tree, sample) evaluation: per level the node's feature and
    threshold, the rank, the comparison and the step down; then one count."""
    return 4 * depth + 2


def work(case):
    n, F, K, op = case["n"], case["F"], case["K"], case["op"]
    if op == "encode":
        w = 2 if case["width"] == 2 or case["data"] == "grid" or n <= 65_536 else 4
        return dict(bytes=n * F * (4 + w) + 4 * F, flops=n * F * max(1, math.ceil(math.log2(n))))
    if op == "predict":
        return dict(bytes=n * (4 * F + 2), flops=n * _ops(case["depth"]))
    D = case["depth"]
    L, B = 1 << D, (1 << D) - 1
    if op == "eval":
        m = (n + 1) // 2 if case["subset"] else n
        return dict(bytes=m * (F * case["width"] + 1 + (4 if case["subset"] else 0))
                    + case["P"] * (B * 6 + L * K * 4 + 4), flops=m * case["P"] * _ops(D))
    if op == "fit":
        return dict(bytes=n * (F * case["width"] + 1) + case["P"] * B * 8,
                    flops=n * case["P"] * (case["G"] + 1) * _ops(D))
    raw = op in ("request", "classifier")
    P, G, H = (100, 600, 2 if D == 2 else 3) if op == "classifier" else (case["P"], case["G"], case["horizon"])
    levels = [min(H, D - d) for d in range(D)]
    flops = sum(n * P * (G + 1) * _ops(t) if t >= 2 else n * F * K for t in levels)
    if op == "classifier" and case["warm"]:
        flops += n * P * (G + 1) * _ops(D)
    return dict(bytes=n * (F * (4 if raw else case["width"]) + 1), flops=flops)


def _exact_ranks(X):
    """Dense ranks [F][n] (int64) and the distinct counts [F]."""
    ranks, nu = [], []
    for f in range(X.shape[1]):
        v, inv = torch.unique(X[:, f].double(), sorted=True, return_inverse=True)
        ranks.append(inv)
        nu.append(v.numel())
    return ranks, nu


def exact(case, seed):
    op, n, K = case["op"], case["n"], case["K"]
    if op not in ("eval", "encode", "predict"):
        return None  # a trajectory of random draws and selections
    if op == "eval" and n * case["P"] * case["depth"] > 4_000_000_000:
        return None
    X, comp = _features(case, seed)
    if op == "predict":
        y = _labels(case, seed, X, comp)
        a, b, leaf = _raw_tree(case, seed, X)
        a = a.long()
        t = torch.ones(n, dtype=torch.int64, device=DEV)
        for _ in range(case["depth"]):
            p = a[t - 1]
            v = X.gather(1, (p - 1).clamp(min=0)[:, None])[:, 0].double()
            t = 2 * t + 1 - ((p > 0) & (v < b[t - 1])).long()
        pred = leaf[t - len(leaf)]
        return pred, (pred == y).sum().reshape(1)
    ranks, nu = _exact_ranks(X)
    if op == "encode":
        width = 2 if case["width"] == 2 or max(nu) <= 65_536 else 4
        rows = torch.stack([r.to(torch.int32) for r in ranks])
        return (rows.to(torch.int16) if width == 2 else rows), torch.tensor(nu, dtype=torch.int32), width
    y = _labels(case, seed, X, comp).long()
    a, th = _trees(case, seed, torch.tensor(nu, device=DEV))
    idx = _subset(case, seed)
    R = torch.stack([r.to(torch.int32) for r in ranks])
    if idx is not None:
        R, y = R[:, idx.long()], y[idx.long()]
    m, L = R.shape[1], 1 << case["depth"]
    cols = torch.arange(m, device=DEV)
    counts = torch.zeros(case["P"], L, K, dtype=torch.int64)
    for i in range(case["P"]):
        ai, ti = a[i].long(), th[i].long()
        t = torch.ones(m, dtype=torch.int64, device=DEV)
        for _ in range(case["depth"]):
            p = ai[t - 1]
            v = R[(p - 1).clamp(min=0), cols]
            t = 2 * t + 1 - ((p > 0) & (v < ti[t - 1])).long()
        counts[i] = torch.bincount((t - L) * K + y, minlength=L * K).reshape(L, K).cpu()
    errors = m - counts.max(dim=2).values.sum(dim=1)
    return counts.to(torch.int32), errors.to(torch.int32)
