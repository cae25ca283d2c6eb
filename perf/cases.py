"""What the speed of this framework is measured on: calls that its users
make through paper_2407_12208_gb300.Context, from the smallest query to the
largest Lloyd step.

Sizes are those of the benchmark's workloads, of the served job mix
(n 10^3..10^6, d in {2, 8, 32, 128, 256}, k 4..1024) and of the paper's
Tables 6.1-6.7, with odd and ragged ones among them.  Inputs are made on the
GPU from the seed alone, with the distributions of workloads.py.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2407_12208_gb300 as mpkm

DEV = "cuda:0"


def listed():
    return [
        # a query against few centres: the smallest job of the served mix, where latency counts
        dict(name="query-small", call="assign", low="bf16", data="mixture", n=1000, d=32, k=64),
        # a whole small clustering: Gaussian blobs 10^4 x 16, k = 8, 20 iterations
        dict(name="run-blobs-small", call="run", low="bf16", data="blobs", n=10000, d=16, k=8, iters=20),
        # a whole clustering of Table 6.6's size
        dict(name="run-blobs-d128", call="run", low="fp16", data="blobs", n=100000, d=128, k=500, iters=10),
        # one iteration at Table 6.3's size: d is no multiple of a vector load
        dict(name="step-blobs-d10", call="step", low="bf16", data="blobs", n=100000, d=10, k=100),
        # the benchmark's step: uniform data, every centre about equally far
        dict(name="step-uniform", call="step", low="bf16", data="uniform", n=1000000, d=128, k=1024),
        # a large mixture at d = 64: the step that memory traffic weighs on most
        dict(name="step-mixture", call="step", low="bf16", data="mixture", n=4000000, d=64, k=256),
        # image segmentation, (r, g, b, x, y) per pixel, plain fp32: the largest n
        dict(name="step-image", call="step", low="fp32", data="image", n=4096 * 4096, d=5, k=16),
        # the cancellation regime of Section 4: every pair fails the reliability test
        dict(name="assign-cancellation", call="assign", low="bf16", data="cancellation", n=1000000, d=128, k=1024),
        # a first iteration on wide data in eight bits: rows of clusters that got no initial
        # centre stay open after the screen; ragged n and k
        dict(name="step-wide-e4m3", call="step", low="e4m3", data="mixture", n=150001, d=256, k=389),
        # the fp32 direct formula at an odd shape
        dict(name="assign-ragged-fp32", call="assign", low="fp32", data="mixture", n=60013, d=50, k=203),
        # Tables 6.1 / 6.2: the full distance matrix, half of the rows next to a centre
        dict(name="distances-half-near", call="distances", low="fp16", test="tc", data="near", n=5000, d=128, k=5000),
        # k-means++ seeds for a clustering of Table 6.6's size
        dict(name="seeding", call="seed", data="blobs", n=100000, d=128, k=64),
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, uniform in its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _dim(rng, lo=2, hi=256):
    """Half the time a dimension of the served mix, else any."""
    usual = [d for d in (2, 8, 16, 32, 64, 128, 256) if lo <= d <= hi]
    return rng.choice(usual) if rng.random() < 0.5 else _log(rng, lo, hi)


def draw(rng):
    call = rng.choice(["assign", "assign", "step", "step", "step", "run", "run", "distances", "seed"])
    if call == "distances":
        # every tested precision; Alg. 2's own test with bf16 sends all pairs to the fallback
        low, test = rng.choice([("fp16", "tc"), ("bf16", "tc"), ("fp16", "paper"), ("bf16", "paper")])
        n, d = _log(rng, 300, 3000), _dim(rng, 16, 200)
        return dict(call=call, low=low, test=test, data="near", n=n, d=d, k=min(n, _log(rng, 300, 3000)))
    if call == "seed":
        n = _log(rng, 1000, 200000)
        return dict(call=call, data="blobs", n=n, d=_dim(rng), k=_log(rng, 4, 64))
    if call == "run":
        n = _log(rng, 1000, 200000)
        low = rng.choice(["bf16", "fp16", "fp32"])
        d = _dim(rng, 2 if low == "fp32" else 8, 16 if low == "fp32" else 256)
        return dict(call=call, low=low, data="blobs", n=n, d=d, k=min(_log(rng, 4, 512), n // 8),
                    iters=rng.choice([5, 10, 20]))
    if call == "step" and rng.random() < 0.25:
        n, k = _log(rng, 65536, 1 << 23), _log(rng, 4, 32)
        return dict(call=call, low="fp32", data="image", n=n, d=5, k=k)
    low = rng.choice(["bf16", "bf16", "fp16", "fp32", "e4m3"])
    if low == "e4m3":  # eight bits are for wide data
        n, d = _log(rng, 1000, 500000), _dim(rng, 128, 256)
        return dict(call=call, low=low, data="mixture", n=n, d=d, k=min(n // 8, _log(rng, 4, 1024)))
    data = rng.choice(["uniform", "mixture", "blobs", "cancellation"])
    d = _dim(rng)
    # all pairs in fp32 (the direct format, the cancellation regime): up to a tenth of the largest
    slow = low == "fp32" or data == "cancellation"
    n, k = _log(rng, 1000, 100000 if slow else 1000000), _log(rng, 4, 1024)
    return dict(call=call, low=low, data=data, n=n, d=d, k=min(k, n // 8))


# --------------------------------------------------------------------- inputs
def _distinct_rows(X, k, g):
    return X[torch.randperm(X.shape[0], generator=g, device=DEV)[:k].sort().values].clone()


def _inputs(case, seed):
    """(X, C): points and centres, float32 on the GPU."""
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * seed + 17)
    n, d, k, data = case["n"], case["d"], case["k"], case["data"]
    rand = lambda *s: torch.rand(*s, generator=g, device=DEV)  # noqa: E731
    randn = lambda *s: torch.randn(*s, generator=g, device=DEV)  # noqa: E731
    if data == "near":  # C = X + 1e-4 N(0, I) on half of the rows
        X = randn(n, d)
        C = randn(k, d)
        m = k // 2
        C[:m] = X[:m] + 1e-4 * C[:m]
        return X, C
    if data == "uniform":
        X = rand(n, d)
    elif data == "cancellation":
        X = randn(n, d).mul_(1e-2).add_(1e3)
    elif data == "image":
        w = int(math.isqrt(n))
        rows = -(-n // w)
        sites = 16
        at, colour = rand(sites, 2) * torch.tensor([w, rows], device=DEV), rand(sites, 3)
        X = torch.empty(n, 5, device=DEV)
        step = 1 << 21
        for s in range(0, n, step):
            i = torch.arange(s, min(n, s + step), device=DEV)
            x, y = (i % w).float(), torch.div(i, w, rounding_mode="floor").float()
            region = ((x[:, None] - at[:, 0]) ** 2 + (y[:, None] - at[:, 1]) ** 2).argmin(1)
            X[s : s + step, :3] = (colour[region] + 0.02 * randn(len(i), 3)).clamp_(0, 1)
            X[s : s + step, 3] = x / max(w - 1, 1)
            X[s : s + step, 4] = y / max(rows - 1, 1)
    else:
        if data == "blobs":
            centres, std = 20 * rand(k, d) - 10, torch.ones(k, device=DEV)
        else:
            centres, std = 5 * randn(k, d), torch.exp(rand(k) * math.log(20.0) + math.log(0.1))
        X = randn(n, d)
        step = 1 << 20
        for s in range(0, n, step):
            lab = torch.randint(0, k, (min(n, s + step) - s,), generator=g, device=DEV)
            X[s : s + step] = X[s : s + step] * std[lab, None] + centres[lab]
    return X, _distinct_rows(X, k, g)


def _draws(case, seed):
    return np.random.Generator(np.random.PCG64(seed + 5)).random(case["k"])


def prepare(case, seed):
    X, C = _inputs(case, seed)
    st = dict(call=case["call"], X=X, C=C, ctx=mpkm.Context(0))
    if case["call"] == "seed":
        st["u"] = _draws(case, seed)
    else:
        st["p"] = mpkm.params(case["low"], test=case.get("test", "tc"), max_iter=case.get("iters", 20))
    return st


def run(st):
    ctx, X, call = st["ctx"], st["X"], st["call"]
    if call == "seed":
        return dict(zip(("C", "idx"), ctx.seed_pp(X, st["u"])))
    C, p = st["C"], st["p"]
    if call == "assign":
        return dict(zip(("labels", "min_dist", "flagged"), ctx.assign(X, C, p)))
    if call == "step":  # as in a loop of a fixed number of iterations: nobody asks for the shift
        return dict(zip(("labels", "min_dist", "C", "counts"), ctx.lloyd_step(X, C, p, want_shift=False)))
    if call == "run":
        return dict(zip(("C", "labels", "sse", "eta", "iters"), ctx.lloyd_run(X, C, p)))
    return dict(zip(("D", "flags", "flagged"), ctx.distances(X, C, p)))


def work(case):
    """Inputs read once, outputs written once; two operations per pair and coordinate."""
    n, d, k, call = case["n"], case["d"], case["k"], case["call"]
    pairs = float(n) * k
    io = 4 * n * d + 4 * k * d
    if call == "seed":
        return {"bytes": io + 16 * k, "flops": 2 * pairs * d}
    if call == "distances":
        return {"bytes": io + 4 * pairs + pairs / 8, "flops": 2 * pairs * d}
    if call == "assign":
        return {"bytes": io + 12 * n, "flops": 2 * pairs * d}
    if call == "step":
        return {"bytes": io + 12 * n + 4 * k * d + 8 * k, "flops": 2 * pairs * d}
    return {"bytes": io + 4 * n + 4 * k * d + 16 * case["iters"], "flops": 2 * pairs * d * (case["iters"] + 1)}


# ------------------------------------------------------------ 64-bit results
def _nearest(X, C):
    """(labels, squared distances) in binary64: the two nearest centres by the
    expanded formula about the mean, decided by the direct formula."""
    mu = C.double().mean(0)
    Cd = C.double() - mu
    q = (Cd * Cd).sum(1)
    lab = torch.empty(X.shape[0], dtype=torch.int64, device=X.device)
    md = torch.empty(X.shape[0], dtype=torch.float64, device=X.device)
    step = max(1, min(1 << 18, (1 << 27) // max(C.shape[0], C.shape[1])))
    for s in range(0, X.shape[0], step):
        x = X[s : s + step].double() - mu
        e = torch.addmm(q, x, Cd.T, alpha=-2.0)
        two = e.topk(min(2, C.shape[0]), dim=1, largest=False).indices.sort(1).values
        x = X[s : s + step].double()
        best = None
        for c in two.unbind(1):
            t = x - C[c].double()
            v = (t * t).sum(1)
            if best is None:
                best, arg = v, c
            else:
                arg = torch.where(v < best, c, arg)
                best = torch.minimum(best, v)
        lab[s : s + step], md[s : s + step] = arg, best
    return lab, md


def _means(X, lab, md, C):
    """(new centres in float32, counts); empty clusters take the farthest rows."""
    k, d = C.shape
    s = torch.zeros(k, d, dtype=torch.float64, device=X.device)
    step = 1 << 20
    for i in range(0, X.shape[0], step):
        s.index_add_(0, lab[i : i + step], X[i : i + step].double())
    cnt = torch.bincount(lab, minlength=k)
    new = s / cnt.clamp(min=1)[:, None]
    empty = (cnt == 0).nonzero().flatten()
    if len(empty):
        far = torch.sort(md, descending=True, stable=True).indices[: len(empty)]
        new[empty] = X[far].double()
    return new, cnt


def exact(case, seed):
    X, C = _inputs(case, seed)
    call = case["call"]
    if call == "distances":
        D = torch.empty(X.shape[0], C.shape[0], dtype=torch.float64, device=X.device)
        step = max(1, (1 << 27) // C.numel())
        for s in range(0, X.shape[0], step):
            t = X[s : s + step, None].double() - C.double()
            D[s : s + step] = (t * t).sum(2)
        return dict(D=D, flags=None, flagged=None)
    if call == "seed":
        u, n = _draws(case, seed), case["n"]
        x = X.double()
        i = min(int(u[0] * n), n - 1)
        idx, d2 = [i], None
        for t in range(1, case["k"]):
            v = ((x - x[i]) ** 2).sum(1)
            d2 = v if d2 is None else torch.minimum(d2, v)
            c = d2.cumsum(0)
            i = min(int(torch.searchsorted(c, float(u[t]) * c[-1:], right=True)), n - 1)
            idx.append(i)
        return dict(C=x[idx], idx=None)
    if call in ("assign", "step"):
        lab, md = _nearest(X, C)
        if call == "assign":
            return dict(labels=None, min_dist=md, flagged=None)
        return dict(labels=None, min_dist=md, C=_means(X, lab, md, C)[0], counts=None)
    sse = []
    for it in range(case["iters"] + 1):
        lab, md = _nearest(X, C)
        sse.append(float(md.sum()))
        if it < case["iters"]:
            new = _means(X, lab, md, C)[0]
            C = new.float()  # the centres are kept in float32 from one iteration to the next
    return dict(C=new, labels=None, sse=np.array(sse), eta=None, iters=None)
