"""The work that users of libflashgmm have it do, as timed cases: EM iterations and fits from ten thousand points to ten
million, the k-means warm start, the IVF assignment and its posting lists, densities, Fisher vectors and data streamed
from the host.

A case is a dict: ``op`` names the entry point, ``N``, ``D``, ``K`` the shape, and a few ops have one more number.  All
inputs are draws from a diagonal mixture as in ``paper_2606_10896_b200/synth.py`` (see ``_data``).  Parameters are what
the entry point meets in use, as the warm start leaves them: a few k-means iterations from data rows, then the clusters'
moments, so that some clusters hold several components, some components cover several clusters, and a few hold a point
or two and sit at the variance floor.  Whole fits and the codebook of the Fisher vectors get them with the smallest
clusters replaced by halves of the largest, as a careful user starts them (a component of one point in a fit follows
rounding errors from the second iteration on).
"""
import math

import numpy as np
import torch

from paper_2606_10896_b200 import flashgmm as fg

VAR_FLOOR = 1e-6
SPLIT = 48                    # points that a cluster has to hold to start a component of a fit

_contexts = {}


def _context():
    """One context for the whole program, on the stream current when it is first needed (as a user's program keeps it)."""
    dev = torch.cuda.current_device()
    if dev not in _contexts:
        _contexts[dev] = fg.Context(dev)
    return _contexts[dev]


def listed():
    return [
        # Clustering of a small table: a whole fit of ten iterations, nothing but launches and waits.
        {"name": "fit 10K x 16, K=8", "op": "fit", "N": 10_000, "D": 16, "K": 8, "iters": 10},
        # The paper's table at 100K points: the first iterations of a fit, about 100 points per component.
        {"name": "fit 100K x 128, K=1024", "op": "fit", "N": 100_000, "D": 128, "K": 1024, "iters": 5},
        # One iteration of a fit at a word-embedding size: D is no multiple of 16, N no multiple of a tile.
        {"name": "em 1.2M x 100, K=1000", "op": "em", "N": 1_183_514, "D": 100, "K": 1000},
        # One iteration of a large fit, the shape of the paper's table and of the benchmark.
        {"name": "em 10M x 128, K=1024", "op": "em", "N": 10_000_000, "D": 128, "K": 1024},
        # One iteration at the IVF coarse-quantizer shape: wide unit-norm embeddings, many components.
        {"name": "em 1M x 768, K=4096", "op": "em", "N": 1_000_000, "D": 768, "K": 4096},
        # One iteration over data that stays in (pinned) host memory.
        {"name": "host 1M x 128, K=1024", "op": "em_host", "N": 1_000_000, "D": 128, "K": 1024},
        # IVF multi-assignment: the two best components of every vector and their responsibilities.
        {"name": "top2 1M x 128, K=1024", "op": "assign", "N": 1_000_000, "D": 128, "K": 1024, "m": 2},
        # The assignment that follows the fit at the coarse-quantizer shape.
        {"name": "top4 500K x 768, K=4096", "op": "assign", "N": 500_000, "D": 768, "K": 4096, "m": 4},
        # Posting lists of an index over ten million vectors, at most two lists per vector.
        {"name": "lists 10M, K=1024", "op": "lists", "N": 10_000_000, "D": 1, "K": 1024},
        # One Lloyd iteration of the warm start.
        {"name": "kmeans 1M x 128, K=1024", "op": "kmeans", "N": 1_000_000, "D": 128, "K": 1024},
        # Log-densities of a batch of queries.
        {"name": "score 50K x 96, K=512", "op": "score", "N": 50_021, "D": 96, "K": 512},
        # Fisher vectors of 500 images of about 2000 local descriptors each.
        {"name": "fisher 500 x 2000 x 64, K=256", "op": "fisher", "N": 1_000_000, "D": 64, "K": 256, "groups": 500},
    ]


_MOST_FLOPS = 2.4e13          # about what the largest listed case takes


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["fit", "fit", "em", "em", "em", "em_host", "assign", "assign", "lists", "kmeans", "score", "fisher"])
    if op == "lists":
        return {"op": op, "N": _log_int(rng, 10_000, 10_000_000), "D": 1, "K": _log_int(rng, 8, 4096)}
    wide = op in ("em", "assign", "kmeans") and rng.random() < 0.3
    if wide:
        # embeddings: 64 components and more, at least about a hundred points for each
        D, K = _log_int(rng, 129, 1024), _log_int(rng, 64, 4096)
        N = _log_int(rng, max(20_000, 100 * K), 1_000_000)
    elif op == "fit":
        D, K = _log_int(rng, 2, 128), _log_int(rng, 2, 1024)
        N = _log_int(rng, max(2_000, 60 * K), 200_000)
    elif op == "fisher":
        D, K = _log_int(rng, 16, 128), _log_int(rng, 16, 512)
        groups = _log_int(rng, 4, 500)
        N = groups * _log_int(rng, 500, 4_000)
    else:
        D, K = _log_int(rng, 8, 128), _log_int(rng, 16, 4096)
        N = _log_int(rng, max(10_000, 60 * K), 1_000_000 if op in ("em_host", "score") else 10_000_000)
    case = {"op": op, "N": N, "D": D, "K": K}
    if op == "fit":
        case["iters"] = rng.randint(3, 8)
    if op == "fisher":
        case["groups"] = groups
    if op == "assign":
        case["m"] = rng.choice([1, 2, 4])
    if op == "score":
        case["N"] = min(N, int(2e12 / (4.0 * D * K)))
    # (a case stays within the largest listed one's arithmetic, and within 6 GB of data)
    most = min(_MOST_FLOPS / (8.0 * D * K * case.get("iters", 1)), 1.5e9 / D)
    case["N"] = max(2_000, int(min(case["N"], most)))
    return case


# ---------------------------------------------------------------------------------------------------------------- inputs

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(1_000_003 * (int(seed) % (1 << 40)) + 17)
    return g


def _data(case, gen):
    """N draws from a diagonal mixture.  D <= 128: means ~ N(0, 3^2), standard deviations ~ U[0.5, 1.5]; wide data:
    unit-norm means, standard deviations ~ U[0.02, 0.08], points of unit norm.  Weights ~ Dirichlet(1)."""
    N, D, K = case["N"], case["D"], case["K"]
    wide = D > 128
    f = dict(device="cuda", generator=gen)
    means = torch.randn((K, D), **f) * (1.0 if wide else 3.0)
    stds = torch.rand((K, D), **f)
    if wide:
        means /= means.norm(dim=1, keepdim=True)
        stds = 0.02 + 0.06 * stds
    else:
        stds = 0.5 + stds
    w = torch.empty(K, dtype=torch.float64, device="cuda").exponential_(1.0, generator=gen)
    cdf = torch.cumsum(w / w.sum(), 0)
    X = torch.empty((N, D), dtype=torch.float32, device="cuda")
    step = max(1, (1 << 28) // D)
    for lo in range(0, N, step):
        hi = min(N, lo + step)
        c = torch.searchsorted(cdf, torch.rand(hi - lo, dtype=torch.float64, **f), right=True).clamp_(0, K - 1)
        x = X[lo:hi]
        x.normal_(generator=gen)
        x.mul_(stds[c]).add_(means[c])
        if wide:
            x.div_(x.norm(dim=1, keepdim=True))
    return X


def _rows(X, K, gen):
    """K distinct rows of X."""
    N = X.shape[0]
    n = min(N, 64 * K)
    return X[torch.randperm(n, device="cuda", generator=gen)[:K]].clone()


def _clusters(X, K, gen, iters=3):
    """K-means on the first rows of X, from data rows: (centroids, those rows, their clusters as a one-hot matrix)."""
    xs = X[: min(X.shape[0], max(128 * K, 16_384), (1 << 30) // K)]
    cen = _rows(X, K, gen)
    one = torch.empty((xs.shape[0], K), device="cuda")
    for it in range(iters + 1):
        a = torch.addmm((cen * cen).sum(1), xs, cen.t(), alpha=-2.0).argmin(1)
        one.zero_().scatter_(1, a[:, None], 1.0)
        n = one.sum(0)[:, None]
        if it < iters:
            cen = torch.where(n > 0, one.t() @ xs / n.clamp_min(1.0), cen)
    return cen, xs, one


def _warm_params(X, K, gen, split=0):
    """What EM gets from the k-means warm start: the clusters' shares, means and variances.  Clusters of fewer than
    ``split`` points take half of one of the largest each."""
    cen, xs, one = _clusters(X, K, gen)
    n = one.sum(0)
    shift = xs.mean(0)                                      # (moments about the data's mean: less to cancel)
    xc = xs - shift
    s1, s2 = one.t() @ xc, one.t() @ (xc * xc)
    nn = n[:, None].clamp_min(1.0)
    m = s1 / nn
    var = (s2 / nn - m * m).clamp_min(VAR_FLOOR)
    held = n[:, None] > 0
    glob = (xc * xc).mean(0).clamp_min(VAR_FLOOR)
    mu = torch.where(held, m + shift, cen).contiguous()
    var = torch.where(held, var, glob).contiguous()
    n = n + 1e-3
    if split:
        order = torch.argsort(n)
        few = min(int((n < split).sum()), K // 2)
        small, large = order[:few], order[K - few:].flip(0)
        off = 0.25 * var[large].sqrt() * torch.randn((few, X.shape[1]), device="cuda", generator=gen)
        mu[small], var[small] = mu[large] + off, var[large]
        mu[large] -= off
        n[large] *= 0.5
        n[small] = n[large]
    pi = n / n.sum()
    return pi.contiguous(), mu, var


def _stats(K, D):
    f = dict(dtype=torch.float64, device="cuda")
    return torch.empty(K, **f), torch.empty((K, D), **f), torch.empty((K, D), **f)


def prepare(case, seed):
    op, N, D, K = case["op"], case["N"], case["D"], case["K"]
    gen = _generator(seed)
    s = {"case": case, "ctx": _context()}
    if op == "lists":
        # what the top-2 assignment gives: sharp posteriors, the second one above the threshold for the same share of the
        # vectors in every draw
        a = torch.randint(0, K, (N,), device="cuda", generator=gen)
        b = (a + torch.randint(1, max(2, K), (N,), device="cuda", generator=gen)) % K
        r = ((torch.randperm(N, device="cuda", generator=gen).double() + 0.5) / N).pow_(12).float() * 0.5
        s["idx"] = torch.stack([a, b], 1).int().contiguous()
        s["resp"] = torch.stack([1.0 - r, r], 1).contiguous()
        s["out"] = (torch.empty(K + 1, dtype=torch.int64, device="cuda"), torch.empty(2 * N, dtype=torch.int32, device="cuda"))
        return s
    X = _data(case, gen)
    s["X"] = X
    if op == "fit":
        s["start"] = _warm_params(X, K, gen, split=SPLIT)
        s["params"] = tuple(t.clone() for t in s["start"])
        return s
    if op == "kmeans":
        s["cen"] = _clusters(X, K, gen, iters=2)[0].contiguous()
        s["out"] = (torch.empty(N, dtype=torch.int32, device="cuda"), torch.empty_like(s["cen"]),
                    torch.empty(K, dtype=torch.int64, device="cuda"))
        s["work"] = torch.empty(2 * N, dtype=torch.int32, device="cuda")
        return s
    s["params"] = _warm_params(X, K, gen, split=SPLIT if op == "fisher" else 0)
    if op == "em":
        s["out"] = _stats(K, D)
    elif op == "em_host":
        s["pinned"] = torch.empty((N, D), dtype=torch.float32, pin_memory=True)
        s["pinned"].copy_(X)
        del s["X"]
        s["Xh"] = s["pinned"].numpy()
        s["params"] = tuple(t.cpu().numpy() for t in s["params"])
        s["out"] = (np.empty(K), np.empty((K, D)), np.empty((K, D)))
    elif op == "assign":
        m = case["m"]
        s["out"] = (torch.empty((N, m), dtype=torch.int32, device="cuda"),
                    None if m == 1 else torch.empty((N, m), dtype=torch.float32, device="cuda"))
    elif op == "score":
        s["out"] = torch.empty(N, dtype=torch.float32, device="cuda")
    elif op == "fisher":
        # images differ in size by a factor of three
        G = case["groups"]
        size = 0.5 + torch.rand(G, device="cuda", generator=gen, dtype=torch.float64)
        cut = torch.round(torch.cumsum(size / size.sum(), 0) * N).long()
        cut[-1] = N
        s["offsets"] = np.concatenate([[0], cut.cpu().numpy()]).astype(np.int64)
        s["out"] = torch.empty((G, 2, K, D), dtype=torch.float32, device="cuda")
    return s


# ------------------------------------------------------------------------------------------------------------------ runs

def run(s):
    case, ctx, op = s["case"], s["ctx"], s["case"]["op"]
    if op == "fit":
        for t, t0 in zip(s["params"], s["start"]):
            t.copy_(t0)
        trace, done = ctx.gmm_fit(s["X"], *s["params"], case["iters"], var_floor=VAR_FLOOR)
        return [trace, done, *s["params"]]
    if op == "em":
        return list(ctx.gmm_em_step(s["X"], *s["params"], out=s["out"]))
    if op == "em_host":
        return list(ctx.gmm_em_step_host(s["Xh"], *s["params"], out=s["out"]))
    if op == "assign":
        return list(ctx.gmm_assign_topm(s["X"], *s["params"], case["m"], out=s["out"], indices_only=case["m"] == 1))
    if op == "lists":
        offsets, items, total, mean = ctx.gmm_build_posting_lists(s["idx"], s["resp"], case["K"], out=s["out"])
        return [offsets, items[:total], total, mean]
    if op == "kmeans":
        return list(ctx.gmm_kmeans_step(s["X"], s["cen"], out=s["out"], work=s["work"]))
    if op == "score":
        return list(ctx.gmm_score_samples(s["X"], *s["params"], out=s["out"]))
    return list(ctx.gmm_fisher_vectors(s["X"], s["offsets"], *s["params"], out=s["out"]))


def work(case):
    """Inputs read once, outputs written once; the contractions of the method (E-step: two, statistics: two; a
    nearest-centroid search: one)."""
    op, N, D, K = case["op"], float(case["N"]), float(case["D"]), float(case["K"])
    params = 4.0 * (K + 2 * K * D)
    stats = 8.0 * (K + 2 * K * D)
    x = 4.0 * N * D
    if op == "fit":
        return {"bytes": case["iters"] * (x + 2 * params), "flops": case["iters"] * 8.0 * N * K * D}
    if op in ("em", "em_host"):
        return {"bytes": x + params + stats, "flops": 8.0 * N * K * D}
    if op == "assign":
        m = case["m"]
        return {"bytes": x + params + N * m * (4.0 if m == 1 else 8.0), "flops": 4.0 * N * K * D}
    if op == "lists":
        return {"bytes": N * 2 * 8.0 + N * 1.5 * 4.0 + 8.0 * K, "flops": 0.0}
    if op == "kmeans":
        return {"bytes": x + 8.0 * K * D + 4.0 * N + 8.0 * K, "flops": 2.0 * N * K * D}
    if op == "score":
        return {"bytes": x + params + 4.0 * N, "flops": 4.0 * N * K * D}
    return {"bytes": x + params + case["groups"] * 8.0 * K * D, "flops": 8.0 * N * K * D}


def tolerance(case):
    """Sums over points of 22- to 24-bit terms, and ties between components that those cannot tell apart."""
    op = case["op"]
    if op == "lists":
        return "exact"
    if op == "assign":
        return {"rel": 3e-5, "max": 1e-2, "differ": 2e-3}       # (the order of components that carry no weight)
    if op == "kmeans":
        return {"rel": 1e-4, "max": 5e-2, "differ": 1e-2}       # (one near-tie decided the other way changes two counts)
    if op == "score":
        return {"rel": 1e-5, "max": 1e-4}
    if op == "fit":
        return {"rel": 1e-4, "max": 1e-2}                       # (differences of one iteration carried into the next)
    if op == "fisher":
        return {"rel": 1e-4, "max": 2e-2}                       # (differences of raw moments)
    return {"rel": 2e-5, "max": 2e-3}
