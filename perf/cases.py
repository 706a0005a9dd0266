"""The work whose speed matters: what programs have this library do.

Every case goes through the public Python binding
(``paper_2507_14261_gb300.famst``) on one library context, as a program
keeps it for all its clouds. The clouds are the recipes of ``workloads/``
drawn on the device: isotropic Gaussian mixtures, mixtures on the unit sphere
and two embedded moons, with the rows in random order.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare`` makes a case's inputs from a seed, ``run`` is one pass, ``work``
what a pass cannot do without, ``exact`` its result in 64 bits where plain
torch can give one.
"""
from __future__ import annotations

import math

import torch

from paper_2507_14261_gb300 import famst

ALG3_SEED = 1   # the seed of Algorithm 3's draws; a program keeps its own


def listed():
    return [
        # a small cloud in a notebook or an inner loop, at the binding's
        # default precision: launches and round trips count
        dict(name="build_2k_fp32", op="build", recipe="blobs", n=2000, d=16, centres=10,
             sigma_lo=1.0, sigma_hi=1.0, k=10, lam=5, prec="fp32"),
        # the ordinary build: one mixture of separated clusters
        dict(name="build_100k", op="build", recipe="blobs", n=100_000, d=128, centres=50,
             sigma_lo=0.5, sigma_hi=2.0, k=16, lam=5, prec="bf16x3"),
        # the largest build: a million unit vectors in a thousand clusters
        dict(name="build_sphere_1m", op="build", recipe="sphere", n=1_000_000, d=128,
             centres=1000, k=32, lam=10, prec="bf16x3"),
        # a training step with the tree weight as topological loss: forward
        # (a build) and backward (the gradient with respect to the points)
        dict(name="train_moons_50k", op="train", recipe="moons", n=50_000, d=64, k=16, lam=5,
             prec="bf16x3"),
        # many clouds of uneven sizes and mixed dimensions in one call
        dict(name="batch_256", op="batch", clouds=256, n_lo=500, n_hi=20_000, shape_seed=1000,
             k=16, lam=5, prec="bf16x3"),
        # the kNN graph alone at the default precision, a width that is no
        # multiple of a warp and a size that is no multiple of a tile
        dict(name="knn_fp32_50k", op="knn", recipe="blobs", n=50_021, d=100, centres=20,
             sigma_lo=1.0, sigma_hi=1.0, k=16, prec="fp32"),
        # the kNN graph of a cloud without gaps between its clusters (most
        # pairs of tiles have to be looked at), tensor-core tiles
        dict(name="knn_overlap_65k", op="knn", recipe="overlap", n=65_537, d=96, centres=200,
             sigma_lo=1.0, sigma_hi=1.0, k=32, prec="bf16x3"),
        # the approximate kNN graph, as the paper runs its first phase
        dict(name="nndescent_100k", op="nndescent", recipe="blobs", n=100_000, d=128,
             centres=50, sigma_lo=0.5, sigma_hi=2.0, k=16),
        # the exact tree that an approximate one is compared with
        dict(name="emst_10k", op="emst", recipe="blobs", n=10_000, d=128, centres=20,
             sigma_lo=0.5, sigma_hi=2.0, prec="bf16x3"),
        # a program that has its own kNN graph and runs the later phases one
        # by one: components, connect, refine, tree
        dict(name="phases_sphere_200k", op="phases", recipe="sphere", n=200_000, d=128,
             centres=500, k=32, lam=10),
        # components joined by their nearest pairs, found over all pairs
        dict(name="nearest_100k", op="nearest", recipe="blobs", n=100_000, d=128, centres=50,
             sigma_lo=0.5, sigma_hi=2.0, k=16, lam=5),
        # the gradient of the tree weight alone, for a tree in hand
        dict(name="backward_1m", op="backward", recipe="sphere", n=1_000_000, d=128,
             centres=1000, k=16, lam=1),
    ]


def _between(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["build", "build", "build", "train", "batch", "knn", "knn", "nndescent",
                     "emst", "phases", "nearest", "backward"])
    d = rng.choice([3, 16, 31, 32, 64, 77, 96, 100, 128])
    c = dict(op=op)
    if op == "batch":
        c.update(clouds=_between(rng, 16, 256), n_lo=500, n_hi=_between(rng, 2000, 20_000),
                 shape_seed=rng.randrange(1 << 20), k=rng.choice([8, 10, 16]),
                 lam=rng.randint(2, 6), prec="bf16x3")
        return c
    mix = dict(sigma_lo=0.5, sigma_hi=rng.choice([1.0, 2.0]))
    if op == "build":
        recipe = rng.choice(["blobs", "blobs", "sphere"])
        if recipe == "sphere":
            n = _between(rng, 5000, 500_000)
            c.update(recipe="sphere", n=n, d=rng.choice([32, 64, 100, 128]),
                     centres=max(5, min(500, n // rng.randint(300, 1000))),
                     k=rng.randint(8, 32), lam=rng.randint(2, 10), prec="bf16x3")
        else:
            prec = rng.choice(["fp32", "bf16x3", "bf16x3"])
            n = _between(rng, 1000, 20_000 if prec == "fp32" else 150_000)
            c.update(recipe="blobs", n=n, d=d, centres=rng.randint(5, 50), k=rng.randint(5, 24),
                     lam=rng.randint(1, 8), prec=prec, **mix)
    elif op == "train":
        recipe = rng.choice(["moons", "blobs"])
        c.update(recipe=recipe, n=_between(rng, 2000, 80_000), d=rng.choice([16, 32, 64, 77, 128]),
                 k=rng.randint(8, 20), lam=rng.randint(2, 6), prec="bf16x3")
        if recipe == "blobs":
            c.update(centres=rng.randint(5, 30), **mix)
    elif op == "knn":
        prec = rng.choice(["fp32", "bf16x3"])
        recipe = rng.choice(["blobs", "overlap"])
        c.update(recipe=recipe, n=_between(rng, 1000, 50_000), d=d, k=rng.randint(4, 32),
                 centres=rng.randint(5, 50) if recipe == "blobs" else rng.randint(20, 200),
                 prec=prec, **mix)
    elif op == "nndescent":
        c.update(recipe="blobs", n=_between(rng, 2000, 100_000), d=rng.choice([16, 32, 64, 77, 128]),
                 centres=rng.randint(5, 50), k=rng.randint(8, 24), **mix)
    elif op == "emst":
        c.update(recipe="blobs", n=_between(rng, 500, 10_000), d=d, centres=rng.randint(5, 20),
                 prec=rng.choice(["fp32", "bf16x3", "bf16x3"]), **mix)
    elif op == "phases":
        n = _between(rng, 10_000, 200_000)
        c.update(recipe="sphere", n=n, d=rng.choice([32, 64, 77, 100, 128]),
                 centres=max(5, min(400, n // rng.randint(300, 1000))), k=rng.randint(8, 32),
                 lam=rng.randint(2, 10))
    elif op == "nearest":
        c.update(recipe="blobs", n=_between(rng, 5000, 100_000), d=rng.choice([32, 64, 77, 128]),
                 centres=rng.randint(5, 50), k=rng.randint(8, 16), lam=rng.randint(1, 8), **mix)
    else:   # backward
        n = _between(rng, 5000, 1_000_000)
        c.update(recipe="sphere", n=n, d=rng.choice([32, 64, 100, 128]),
                 centres=max(5, min(1000, n // 1000)), k=rng.randint(8, 16), lam=1)
    return c


# ----------------------------------------------------------------- inputs

def _mixture(g, n, d, centres, lo, hi, box):
    dev = g.device
    c = (torch.rand((centres, d), generator=g, device=dev) * 2 - 1) * box
    s = torch.rand(centres, generator=g, device=dev) * (hi - lo) + lo
    lab = torch.randperm(n, generator=g, device=dev) % centres
    x = torch.randn((n, d), generator=g, device=dev)
    return x.mul_(s[lab, None]).add_(c[lab])


def _points(case, seed):
    """The cloud of a case, n x d float32 on the device."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 7919 + 17)
    n, d, recipe = case["n"], case["d"], case["recipe"]
    if recipe in ("blobs", "overlap"):
        return _mixture(g, n, d, case["centres"], case["sigma_lo"], case["sigma_hi"],
                        10.0 if recipe == "blobs" else 1.0)
    if recipe == "sphere":
        c = torch.randn((case["centres"], d), generator=g, device=g.device)
        c /= c.norm(dim=1, keepdim=True)
        lab = torch.randperm(n, generator=g, device=g.device) % case["centres"]
        x = torch.randn((n, d), generator=g, device=g.device).mul_(0.02).add_(c[lab])
        return x.div_(x.norm(dim=1, keepdim=True))
    # two interleaved half circles in a random plane of d dimensions
    t = torch.rand(n, generator=g, device=g.device) * math.pi
    up = torch.randperm(n, generator=g, device=g.device) < n // 2
    p = torch.stack([torch.where(up, t.cos(), 1 - t.cos()),
                     torch.where(up, t.sin(), 0.5 - t.sin())], dim=1)
    q, _ = torch.linalg.qr(torch.randn((d, 2), generator=g, device=g.device))
    return (torch.randn((n, d), generator=g, device=g.device) * 0.05 + p @ q.T).contiguous()


def _batch_shape(case):
    """Point offsets and dimensions of a batch: one shape for a program's
    whole run, so it hangs on the case and not on the inputs' seed."""
    g = torch.Generator()
    g.manual_seed(case["shape_seed"])
    B = case["clouds"]
    n = torch.randint(case["n_lo"], case["n_hi"] + 1, (B,), generator=g)
    dims = torch.tensor([3, 32, 128])[torch.randint(0, 3, (B,), generator=g)]
    centres = torch.randint(5, 21, (B,), generator=g)
    off = torch.zeros(B + 1, dtype=torch.int64)
    off[1:] = n.cumsum(0)
    return off.numpy(), dims.to(torch.int32).numpy(), n.tolist(), dims.tolist(), centres.tolist()


def prepare(case, seed):
    ctx = famst.default_context()
    s = dict(case=case, ctx=ctx)
    if case["op"] == "batch":
        off, dims, ns, ds, cs = _batch_shape(case)
        g = torch.Generator(device="cuda")
        g.manual_seed(seed * 7919 + 17)
        X = torch.empty(sum(n * d for n, d in zip(ns, ds)), device="cuda")
        at = 0
        for n, d, c in zip(ns, ds, cs):
            X[at:at + n * d] = _mixture(g, n, d, c, 1.0, 1.0, 10.0).reshape(-1)
            at += n * d
        m = sum(ns) - len(ns)
        out = (torch.empty(m, dtype=torch.int32, device="cuda"),
               torch.empty(m, dtype=torch.int32, device="cuda"),
               torch.empty(m, dtype=torch.float32, device="cuda"))
        s.update(X=X, off=off, dims=dims, out=out)
        return s
    X = s["X"] = _points(case, seed)
    if case["op"] == "train":
        X.requires_grad_(True)
    elif case["op"] == "phases":
        s["nbr"], s["dist"] = ctx.knn_graph(X, case["k"], "bf16x3")
    elif case["op"] == "nearest":
        nbr, _ = ctx.knn_graph(X, case["k"], "bf16x3")
        s["comp"], s["t"] = ctx.components(nbr)
    elif case["op"] == "backward":
        tree, _ = ctx.build(X, case["k"], case["lam"], ALG3_SEED, "bf16x3")
        s.update(tu=tree.u, tv=tree.v)
    return s


# ------------------------------------------------------------- one pass

def _edges(E):
    return dict(u=E.u, v=E.v, w=E.w, ci=E.ci, cj=E.cj)


def _counts(c, length):
    """Counts of as many iterations as the inputs took, in one length."""
    return torch.tensor([int(x) for x in c[:length]] + [0] * (length - len(c)))


def run(s):
    case, ctx = s["case"], s["ctx"]
    op = case["op"]
    if op == "build":
        T, _ = ctx.build(s["X"], case["k"], case["lam"], ALG3_SEED, case["prec"])
        return dict(u=T.u, v=T.v, w=T.w, W=T.W)
    if op == "train":
        W = famst.mst_weight(s["X"], case["k"], case["lam"], ALG3_SEED, case["prec"])
        (gX,) = torch.autograd.grad(W, s["X"])
        return dict(W=W.detach(), gX=gX)
    if op == "batch":
        _, W, t, _ = ctx.build_batched(s["X"], s["off"], s["dims"], case["k"], case["lam"],
                                       ALG3_SEED, case["prec"], out=s["out"])
        u, v, w = s["out"]
        return dict(u=u, v=v, w=w, W=W, t=t)
    if op == "knn":
        nbr, dist = ctx.knn_graph(s["X"], case["k"], case["prec"])
        return dict(nbr=nbr, dist=dist)
    if op == "nndescent":
        nbr, dist, iters, updates, pairs = ctx.knn_nndescent(s["X"], case["k"], seed=ALG3_SEED)
        return dict(nbr=nbr, dist=dist, iters=iters, updates=_counts(updates, 10),
                    pairs=_counts(pairs, 10))
    if op == "emst":
        T, rounds = ctx.emst_exact(s["X"], case["prec"])
        return dict(u=T.u, v=T.v, w=T.w, W=T.W, rounds=rounds)
    if op == "phases":
        X, n = s["X"], case["n"]
        comp, t = ctx.components(s["nbr"])
        E = ctx.connect(X, comp, t, case["lam"], ALG3_SEED)
        sweeps, delta = ctx.refine(X, s["nbr"], comp, E)
        u, v, w, W = ctx.mst(n, s["nbr"], s["dist"], E)
        return dict(comp=comp, E=_edges(E), sweeps=sweeps, delta=_counts(delta, 64), u=u, v=v,
                    w=w, W=W)
    if op == "nearest":
        return _edges(ctx.connect_nearest(s["X"], s["comp"], s["t"], case["lam"]))
    return dict(gX=ctx.mst_backward(s["X"], s["tu"], s["tv"]))


# ------------------------------------------------ what a pass has to do

def _knn_work(n, d, k, own):
    """Points in, lists out; every row against the rows of its own cluster
    (`own` of them): fewer cannot tell its nearest ones."""
    return 4 * n * d + 8 * n * k, 2 * d * n * max(own, k)


def work(case):
    op = case["op"]
    if op == "batch":
        _, _, ns, ds, cs = _batch_shape(case)
        b = f = 0
        for n, d, c in zip(ns, ds, cs):
            b += 4 * n * d + 12 * (n - 1)
            f += 2 * d * n * max(n // c, case["k"]) + case["lam"] ** 2 * c * (c - 1) * d
        return dict(bytes=b, flops=f)
    n, d, k = case["n"], case["d"], case.get("k", 1)
    t = case.get("centres", 2)
    own = n if case["recipe"] == "overlap" else n // t
    lam = case.get("lam", 0)
    pairs = t * (t - 1) // 2
    tree = 12 * (n - 1)
    # Algorithm 3's draws, and one scan of each end of each kept edge
    later = pairs * (lam * lam * 2 * d + lam * 2 * k * 2 * d)
    if op in ("build", "train"):
        f = 2 * d * n * max(own, k) + later
        b = 4 * n * d + (tree if op == "build" else 4 * n * d)
    elif op == "knn":
        b, f = _knn_work(n, d, k, own)
    elif op == "nndescent":
        # one join of every list with itself
        b, f = 4 * n * d + 8 * n * k, n * k * (k - 1) // 2 * 2 * d
    elif op == "emst":
        b, f = 4 * n * d + tree, n * (n - 1) // 2 * 2 * d
    elif op == "phases":
        b = 4 * n * d + 8 * n * k + 4 * n + 20 * lam * pairs + tree
        f = later
    elif op == "nearest":
        b, f = 4 * n * d + 4 * n + 20 * lam * pairs, int((1 - 1 / t) * n * n / 2 * 2 * d)
    else:
        b, f = 8 * n * d + 8 * (n - 1), 6 * d * n
    return dict(bytes=b, flops=f)


# ------------------------------------------------------ in 64 bits

def _sq(a, b, bb):
    return (a.square().sum(1)[:, None] + bb[None, :]).addmm_(a, b.T, alpha=-2).clamp_(min=0)


def exact(case, seed):
    op = case["op"]
    if op not in ("knn", "emst", "nearest", "backward"):
        return None   # their distances belong to edges that the draws choose
    s = prepare(case, seed)
    X = s["X"].double()
    n = case["n"]
    if op == "knn":
        xx, k = X.square().sum(1), case["k"]
        dist = torch.empty((n, k), dtype=torch.float64, device=X.device)
        step = max(1, (1 << 27) // n)
        for a in range(0, n, step):
            b = min(n, a + step)
            D = _sq(X[a:b], X, xx)
            D[torch.arange(b - a, device=X.device), torch.arange(a, b, device=X.device)] = math.inf
            ids = D.topk(k, dim=1, largest=False).indices
            near = (X[a:b, None, :] - X[ids]).square().sum(2).sqrt() if k * case["d"] * (b - a) < (1 << 28) \
                else torch.stack([(X[a:b] - X[ids[:, r]]).square().sum(1).sqrt() for r in range(k)], 1)
            dist[a:b] = near.sort(dim=1).values
        return dict(nbr=None, dist=dist)
    if op == "emst":   # Prim on the complete graph
        best = (X - X[0]).square().sum(1)
        best[0] = math.inf
        out = torch.zeros(n, dtype=torch.bool, device=X.device)
        out[0] = True
        W = torch.zeros((), dtype=torch.float64, device=X.device)
        for _ in range(n - 1):
            v = best.argmin()
            W += best[v].sqrt()
            out[v] = True
            best = torch.minimum(best, (X - X[v]).square().sum(1)).masked_fill_(out, math.inf)
        return dict(u=None, v=None, w=None, W=float(W), rounds=None)
    if op == "nearest":
        t, lam = s["t"], case["lam"]
        order = s["comp"].long().argsort(stable=True)
        sizes = torch.bincount(s["comp"].long(), minlength=t).tolist()
        if t < 2 or t > 200 or min(sizes) < lam:
            return None
        P = [p for p in X[order].split(sizes)]
        w = []
        for i in range(t):
            for j in range(i + 1, t):
                D = _sq(P[i], P[j], P[j].square().sum(1))
                at = D.reshape(-1).topk(lam, largest=False).indices
                near = (P[i][at // sizes[j]] - P[j][at % sizes[j]]).square().sum(1).sqrt()
                w.append(near.sort().values)
        return dict(u=None, v=None, w=torch.cat(w), ci=None, cj=None)
    # gradient: unit vectors along the tree's edges
    u, v = s["tu"].long(), s["tv"].long()
    g = X[u] - X[v]
    ln = g.norm(dim=1, keepdim=True)
    g = torch.where(ln > 0, g / ln, torch.zeros_like(g))
    return dict(gX=torch.zeros_like(X).index_add_(0, u, g).index_add_(0, v, -g))
