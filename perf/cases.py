"""The clustering, step and unrolled-gradient calls whose speed is watched.

Each case is one call (or forward and backward) through the package's public
entry points.  Point sets are Gaussian blobs of the sizes, spreads and
bandwidths that this repository's workloads and tests use; every input is made
on the GPU from the seed alone.  `exact` restates each result in 64 bits with
plain torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2112_13891_gb300 as fms

DEV = "cuda"
MODES = 256      # rows of a caller's modes buffer
SET_MODES = 64   # and, on average, of one set's share of the modes of a batch


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # one update of a few seeds on a small 2-D set: what a program that drives
        # its own iteration calls in a loop; latency and launches
        dict(name="step_2d_small", kind="step", n=2000, d=2, m=128, k=5, box=100.0, sigma=2.0,
             h=4.0),
        # one FP32 update of many seeds at an embedding's width, odd sizes
        dict(name="step_32d_ragged", kind="step", n=65_537, d=32, m=20_011, k=64, box=0.0,
             sigma=0.5, h=1.0),
        # one coarse (tensor-core) update, every point a seed
        dict(name="coarse_16d", kind="coarse", n=65_536, d=16, m=65_536, k=32, box=50.0,
             sigma=1.0, h=2.5),
        # plain mean shift of a small 2-D set, every point a seed (Alg. 1)
        dict(name="cluster_2d_all_seeds", kind="cluster", n=2000, d=2, k=5, box=100.0, sigma=2.0,
             h=4.0, noise=0.0, all_seeds=True, metric="euclidean", kernel="gaussian"),
        # the paper-scale clustering: Seed Selection and Early Stopping, 2 % noise
        dict(name="cluster_3d", kind="cluster", n=200_000, d=3, k=20, box=200.0, sigma=0.0,
             h=5.0, noise=0.02, all_seeds=False, metric="euclidean", kernel="gaussian"),
        # plain mean shift at that size (no noise: hundreds of one-point modes would tie
        # in density, and their order in the result with them)
        dict(name="cluster_3d_all_seeds", kind="cluster", n=200_000, d=3, k=20, box=200.0,
             sigma=0.0, h=5.0, noise=0.0, all_seeds=True, metric="euclidean", kernel="gaussian"),
        # image segmentation: RGB pixels in page-locked host memory, labels back there
        dict(name="host_rgb_512", kind="host", n=512 * 512, d=3, k=12, sigma=6.0, h=12.0),
        # embeddings in clusters, precision "auto" (coarse updates, FP32 finish)
        dict(name="cluster_32d", kind="cluster", n=65_536, d=32, k=64, box=0.0, sigma=0.5, h=1.0,
             noise=0.0, all_seeds=False, metric="euclidean", kernel="gaussian"),
        # directions of embeddings (cosine metric)
        dict(name="cosine_16d", kind="cluster", n=200_000, d=16, k=32, box=0.0, sigma=0.05,
             h=0.15, noise=0.0, all_seeds=False, metric="cosine", kernel="gaussian"),
        # many point sets of uneven size in one call
        dict(name="batched_16d", kind="batched", B=256, lo=1000, hi=50_000, d=16, sigma=1.0,
             h=2.5),
        # a training step through unrolled updates: small odd sizes, few seeds
        dict(name="unrolled_3d_small", kind="unrolled", B=3, n=1500, m=701, d=3, k=6, box=40.0,
             sigma=1.0, h=2.0, T=10, ckpt=4, own=False),
        # the large training step: every point a seed, forward and all gradients
        dict(name="unrolled_16d", kind="unrolled", B=8, n=16_384, m=16_384, d=16, k=32, box=50.0,
             sigma=1.0, h=2.0, T=20, ckpt=5, own=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges (every family, sizes over their logarithm)."""
    kind = rng.choice(["step", "step", "coarse", "cluster", "cluster", "cluster", "all", "host",
                       "batched", "unrolled", "unrolled"])
    if kind == "step":
        d = rng.choice([2, 3, 5, 8, 12, 16, 24, 32])
        n = _log(rng, 2000, 65_537)
        m = _log(rng, 64, min(n, 20_011))
        return dict(kind="step", n=n, d=d, m=m, **_shape(rng, d))
    if kind == "coarse":
        d = rng.choice([9, 12, 16, 20])
        n = _log(rng, 8000, 65_536)
        return dict(kind="coarse", n=n, d=d, m=_log(rng, 500, n), **_shape(rng, d))
    if kind == "cluster":
        d = rng.choice([2, 3, 4, 7, 9, 16, 24, 32])
        n = _log(rng, 2000, 200_000)
        # the flat kernel and the cosine metric are used with Seed Selection
        opt = rng.choice(["gaussian", "gaussian", "flat", "cosine"])
        c = dict(kind="cluster", n=n, d=d, noise=0.0, all_seeds=False, metric="euclidean",
                 kernel="gaussian", **_shape(rng, d))
        if opt == "cosine" and d > 2:
            c.update(metric="cosine", box=0.0, sigma=0.05, h=0.15, k=min(c["k"], 2 * d))
        elif opt == "flat" and d <= 4:
            # a window of several spreads: a small one leaves plateaus of the count
            c.update(kernel="flat", h=round(4.0 * c["sigma"], 3))
        return c
    if kind == "all":
        d = rng.choice([2, 3, 3, 6])
        return dict(kind="cluster", n=_log(rng, 2000, 120_000), d=d, noise=0.0, all_seeds=True,
                    metric="euclidean", kernel="gaussian", **_shape(rng, d))
    if kind == "host":
        n = _log(rng, 10_000, 512 * 512)
        return dict(kind="host", n=n, d=3, k=rng.randint(6, 16), sigma=6.0, h=12.0)
    if kind == "batched":
        return dict(kind="batched", B=_log(rng, 8, 200), lo=_log(rng, 500, 2000),
                    hi=_log(rng, 4000, 50_000), d=rng.choice([3, 8, 16]), sigma=1.0, h=2.5)
    d = rng.choice([2, 3, 6, 8, 12, 16])
    n = _log(rng, 500, 12_000)
    own = rng.random() < 0.5
    return dict(kind="unrolled", B=rng.randint(1, 8), n=n, d=d,
                m=n if own else _log(rng, 100, n), k=rng.randint(4, 32), box=50.0, sigma=1.0,
                h=2.0, T=rng.randint(5, 20), ckpt=rng.randint(2, 5), own=own)


def _shape(rng, d):
    """Blob count, centre box, spread and bandwidth, as the workloads of that width have them."""
    if d >= 24:      # embeddings on a sphere of radius 10
        return dict(k=rng.randint(16, 64), box=0.0, sigma=0.5, h=1.0)
    if d >= 8:
        return dict(k=rng.randint(4, 40), box=50.0, sigma=1.0, h=2.5)
    return dict(k=rng.randint(5, 20), box=200.0, sigma=2.0, h=5.0)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _blobs(g, n, d, k, box, sigma, noise=0.0):
    """n points of k Gaussian blobs in random order.  box > 0: centres uniform in [0, box]^d;
    box = 0: centres on the sphere of radius 10.  sigma = 0: each blob's spread uniform in
    [1, 3] and Dirichlet(2) proportions.  noise: that share uniform over the box."""
    if box > 0:
        centers = torch.rand((k, d), generator=g, device=DEV, dtype=torch.float64) * box
    else:
        u = torch.randn((k, d), generator=g, device=DEV, dtype=torch.float64)
        centers = 10.0 * u / u.norm(dim=1, keepdim=True)
    if sigma > 0:
        lab = torch.randint(k, (n,), generator=g, device=DEV)
        spread = torch.full((k,), float(sigma), device=DEV, dtype=torch.float64)
    else:
        e = -torch.log(torch.rand((k, 2), generator=g, device=DEV, dtype=torch.float64)).sum(1)
        lab = torch.multinomial(e / e.sum(), n, replacement=True, generator=g)
        spread = 1.0 + 2.0 * torch.rand((k,), generator=g, device=DEV, dtype=torch.float64)
    X = centers[lab] + spread[lab, None] * torch.randn((n, d), generator=g, device=DEV,
                                                       dtype=torch.float64)
    n_noise = int(round(noise * n))
    if n_noise:
        X[:n_noise] = torch.rand((n_noise, d), generator=g, device=DEV,
                                 dtype=torch.float64) * box
        X = X[torch.randperm(n, generator=g, device=DEV)]
    return X.float().contiguous()


def _directions(g, n, d, k, spread):
    """Directions spread around k axes-like unit vectors (at least 0.9 rad apart, by
    construction: signed axes), every point with a length of its own."""
    q = torch.randn((d, d), generator=g, device=DEV, dtype=torch.float64).cpu().numpy()
    q = np.linalg.qr(q)[0]
    q = torch.from_numpy(np.ascontiguousarray(q)).to(DEV)
    dirs = torch.cat([q, -q], 0)[:k]
    lab = torch.randint(dirs.shape[0], (n,), generator=g, device=DEV)
    P = dirs[lab] + spread * torch.randn((n, d), generator=g, device=DEV, dtype=torch.float64)
    P = P / P.norm(dim=1, keepdim=True)
    r = 0.5 + 19.5 * torch.rand((n, 1), generator=g, device=DEV, dtype=torch.float64)
    return (P * r).float().contiguous()


def _pixels(g, n, k, sigma):
    pal = 20.0 + 215.0 * torch.rand((k, 3), generator=g, device=DEV, dtype=torch.float64)
    e = -torch.log(torch.rand((k, 2), generator=g, device=DEV, dtype=torch.float64)).sum(1)
    lab = torch.multinomial(e / e.sum(), n, replacement=True, generator=g)
    X = pal[lab] + sigma * torch.randn((n, 3), generator=g, device=DEV, dtype=torch.float64)
    return X.clamp(0.0, 255.0).float().contiguous()


def _set_sizes(case):
    """Sizes (log-uniform) and blob counts of a batch's sets: the case's own, for every seed."""
    rng = np.random.default_rng(case["B"] * 31 + case["hi"])
    sizes = np.floor(np.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]),
                                        case["B"]))).astype(np.int64)
    return sizes, rng.integers(4, 41, case["B"])


def _inputs(case, seed):
    """The raw tensors of a case."""
    g = _gen(seed)
    kind = case["kind"]
    if kind in ("step", "coarse"):
        X = _blobs(g, case["n"], case["d"], case["k"], case["box"], case["sigma"])
        pick = torch.randperm(case["n"], generator=g, device=DEV)[: case["m"]]
        # positions on their way to a mode: points moved by a fraction of the spread
        Y = X[pick] + 0.3 * case["sigma"] * torch.randn((case["m"], case["d"]), generator=g,
                                                        device=DEV)
        return X, Y.contiguous()
    if kind == "cluster":
        if case["metric"] == "cosine":
            return _directions(g, case["n"], case["d"], case["k"], case["sigma"])
        return _blobs(g, case["n"], case["d"], case["k"], case["box"], case["sigma"],
                      case["noise"])
    if kind == "host":
        return _pixels(g, case["n"], case["k"], case["sigma"])
    if kind == "batched":
        sizes, ks = _set_sizes(case)
        X = torch.cat([_blobs(g, int(s), case["d"], int(k), 50.0, case["sigma"])
                       for s, k in zip(sizes, ks)], 0)
        return X, np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    X = torch.stack([_blobs(g, case["n"], case["d"], case["k"], case["box"], case["sigma"])
                     for _ in range(case["B"])])
    if case["own"]:
        Y0 = X.clone()
    else:
        Y0 = X[:, : case["m"]] + 0.3 * case["sigma"] * torch.randn(
            (case["B"], case["m"], case["d"]), generator=g, device=DEV)
    G = torch.randn((case["B"], case["m"], case["d"]), generator=g, device=DEV)
    return X, Y0.contiguous(), G


def prepare(case, seed):
    kind = case["kind"]
    data = _inputs(case, seed)
    s = dict(case=case, rng_seed=int(seed) % 1000)
    if kind == "step":
        s.update(X=data[0], Y=data[1], ws=fms.Workspace(
            int(fms._lib.fms_step_workspace_size(case["n"], case["d"], case["m"]))))
    elif kind == "coarse":
        s.update(X=data[0], Y=data[1], ws=fms.Workspace(
            int(fms._lib.fms_coarse_step_workspace_size(case["n"], case["d"], case["m"]))))
    elif kind == "cluster":
        opts = _options(case)
        s.update(X=data, opts=opts,
                 ws=fms.Workspace(fms.workspace_size(case["n"], case["d"], **opts)),
                 # (rows past the mode count stay zero)
                 out=(torch.zeros((MODES, case["d"]), device=DEV),
                      torch.empty(case["n"], dtype=torch.int32, device=DEV),
                      torch.empty(case["n"], device=DEV)))
    elif kind == "host":
        opts = fms.make_options()
        s.update(X=data.cpu().pin_memory(),
                 ws=fms.Workspace(int(fms._lib.fms_cluster_host_workspace_size(
                     case["n"], case["d"], MODES, fms.ctypes.byref(opts)))),
                 out=(torch.zeros((MODES, case["d"])).pin_memory(),
                      torch.empty(case["n"], dtype=torch.int32).pin_memory(), None))
    elif kind == "batched":
        X, offs = data
        opts = fms.make_options()
        s.update(X=X, offs=offs, ws=fms.Workspace(int(fms._lib.fms_batched_workspace_size(
            offs.ctypes.data, case["B"], case["d"], fms.ctypes.byref(opts)))))
    else:
        X, Y0, G = data
        s.update(X=X.requires_grad_(True), Y0=Y0.requires_grad_(True), G=G,
                 h=torch.tensor(case["h"], device=DEV, requires_grad=True))
    return s


def _options(case):
    return dict(all_seeds=case["all_seeds"], kernel=case["kernel"], metric=case["metric"])


def _rows(t, rows):
    """t with zero rows up to a fixed number."""
    return torch.nn.functional.pad(t, (0, 0, 0, rows - t.shape[0]))


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "step":
        return list(fms.mean_shift_step(s["X"], s["Y"], c["h"], with_wsum=True,
                                        workspace=s["ws"]))
    if kind == "coarse":
        return list(fms.mean_shift_step_coarse(s["X"], s["Y"], c["h"], with_wsum=True,
                                               workspace=s["ws"]))
    if kind == "cluster":
        r = fms.cluster(s["X"], c["h"], 1e-3 * c["h"], 300, rng_seed=s["rng_seed"],
                        workspace=s["ws"], out=s["out"], **s["opts"])
        return [s["out"][0], len(r.modes), r.labels, r.margins]
    if kind == "host":
        r = fms.cluster_host(s["X"], c["h"], 1e-3 * c["h"], 300, rng_seed=s["rng_seed"],
                             workspace=s["ws"], out=s["out"])
        return [s["out"][0], len(r.modes), r.labels]
    if kind == "batched":
        r = fms.cluster_batched(s["X"], c["h"], 1e-3 * c["h"], 300, offsets=s["offs"],
                                rng_seed=s["rng_seed"], workspace=s["ws"])
        return [_rows(torch.cat(r.modes), SET_MODES * c["B"]), r.n_modes, r.labels, r.margins]
    out = fms.unrolled_mean_shift(s["X"], s["Y0"], s["h"], T=c["T"], k=c["ckpt"])
    dX, dY0, dh = torch.autograd.grad(out, (s["X"], s["Y0"], s["h"]), s["G"])
    return [out.detach(), dX, dY0, dh]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _evals(case):
    """Seed-point evaluations of a pass: every seed against every point, for the updates that
    the workloads take to converge (about 8 a seed, 256 seeds)."""
    kind = case["kind"]
    if kind in ("step", "coarse"):
        return float(case["n"]) * case["m"]
    if kind == "cluster" and case["all_seeds"]:
        return 7.0 * case["n"] * case["n"]
    if kind in ("cluster", "host"):
        return 8.0 * min(256, case["n"]) * case["n"]
    if kind == "batched":
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"]) \
            if case["hi"] > case["lo"] else case["lo"]
        return 8.0 * 256 * case["B"] * mean
    return float(case["B"]) * case["n"] * case["m"] * case["T"]


def work(case):
    d = case["d"]
    # distance 3d, weight 1 (the exponential counted once), sums 1 + 2d
    per = 5 * d + 2
    kind = case["kind"]
    if kind in ("step", "coarse"):
        bytes_ = 4.0 * d * (case["n"] + 2 * case["m"]) + 4.0 * case["m"]
    elif kind == "cluster":
        bytes_ = case["n"] * (4.0 * d + 8.0)
    elif kind == "host":
        bytes_ = case["n"] * (4.0 * d + 4.0)
    elif kind == "batched":
        mean = _evals(case) / (8.0 * 256)
        bytes_ = mean * (4.0 * d + 8.0)
    else:
        # points and their gradient, seeds, result, upstream gradient, seed gradient
        bytes_ = 4.0 * d * case["B"] * (2 * case["n"] + 4 * case["m"])
        # the adjoint: inner product with the upstream gradient and its three sums
        per = (5 * d + 2) + (11 * d + 6)
    return {"bytes": bytes_, "flops": per * _evals(case)}


def tolerance(case):
    kind = case["kind"]
    if kind == "coarse":
        # weights rounded to BF16: the sums of weights are 1.8e-3 from the 64-bit ones
        return {"rel": 7e-3, "max": 5e-2}
    if kind == "unrolled":
        # dL/dh, one sum of terms of both signs, is up to 1.6e-4 off; the rest 1e-6
        return {"rel": 7e-4, "max": 2e-2}
    if kind == "step":
        return {"rel": 1e-5, "max": 1e-4}
    # modes, labels (whole numbers; a point between two modes may go either way), margins
    return {"rel": 1e-5, "max": 1e-4, "differ": 1e-4}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------

_PAIRS = 1 << 25   # seed-point pairs held at once


def _d2(Y, X):
    return ((Y * Y).sum(1)[:, None] + (X * X).sum(1)[None, :] - 2.0 * (Y @ X.T)).clamp_(min=0.0)


def _update64(X, Y, h, flat=False):
    """(mean, sum of weights) of each row of Y."""
    out, ws = torch.empty_like(Y), torch.empty(Y.shape[0], dtype=Y.dtype, device=Y.device)
    step = max(1, _PAIRS // X.shape[0])
    for a in range(0, Y.shape[0], step):
        D = _d2(Y[a:a + step], X)
        if flat:
            w = (D <= h * h).to(Y.dtype)
        else:
            w = torch.exp(D.mul_(-0.5 / (h * h)))
        ws[a:a + step] = w.sum(1)
        out[a:a + step] = (w @ X) / ws[a:a + step, None]
    return out, ws


def _travel64(X, Y, h, tol, max_iter, flat, sphere):
    """Every seed to convergence: (positions, update of convergence or -1)."""
    Y = Y.clone()
    conv = torch.full((Y.shape[0],), -1, dtype=torch.int64, device=Y.device)
    live = torch.arange(Y.shape[0], device=Y.device)
    for t in range(1, max_iter + 1):
        new, _ = _update64(X, Y[live], h, flat)
        if sphere:
            new = new / new.norm(dim=1, keepdim=True)
        done = (new - Y[live]).norm(dim=1) <= tol
        Y[live] = new
        conv[live[done]] = t
        live = live[~done]
        if live.numel() == 0:
            break
    return Y, conv


def _prune64(X, Y, h, flat):
    """Greedy suppression in order of density (ties: the earlier seed first)."""
    score = _update64(X, Y, h, flat)[1]
    order = torch.argsort(score, descending=True, stable=True)
    P = Y[order]
    alive = torch.ones(P.shape[0], dtype=torch.bool, device=P.device)
    acc = []
    while True:
        left = torch.nonzero(alive)
        if left.numel() == 0:
            break
        i = int(left[0])
        acc.append(i)
        alive &= (P - P[i]).norm(dim=1) >= h
        alive[i] = False
    idx = order[torch.tensor(acc, dtype=torch.long, device=P.device)]
    return idx, score[idx]


def _permutation(n, seed, start, stop):
    """Entries of the library's documented seed permutation (SplitMix64 keys, a balanced
    six-round Feistel network, cycle-walked into [0, n))."""
    m64 = (1 << 64) - 1

    def mix(z):
        z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m64
        z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m64
        return z ^ (z >> 31)

    hb = 1
    while 4 ** hb < n:
        hb += 1
    mask = (1 << hb) - 1
    keys = [mix((seed + (r + 1) * 0x9E3779B97F4A7C15) & m64) for r in range(6)]
    out = []
    for r in range(start, stop):
        x = r
        while True:
            left, right = x >> hb, x & mask
            for key in keys:
                left, right = right, left ^ (mix(key ^ right) & mask)
            x = (left << hb) | right
            if x < n:
                break
        out.append(x)
    return torch.tensor(out, dtype=torch.long, device=DEV)


def _cluster64(X, h, rng_seed, all_seeds=False, flat=False, sphere=False, want_margins=True):
    """Faster Mean-shift with the default options: modes in order and the margins."""
    X = X.double()
    if sphere:
        X = X / X.norm(dim=1, keepdim=True)
    n, tol, max_iter = X.shape[0], 1e-3 * h, 300
    gamma = 1.0 if all_seeds else float(np.float32(0.95))
    N = n if all_seeds else min(128, n)
    seeds = torch.arange(n, device=DEV) if all_seeds else _permutation(n, rng_seed, 0, N)
    pos, conv = _travel64(X, X[seeds], h, tol, max_iter, flat, sphere)
    while True:
        if all_seeds:
            kept = torch.arange(N, device=DEV)
        else:
            c = torch.where(conv < 0, max_iter + 1, conv)
            t_star = min(int(torch.sort(c).values[max(1, math.ceil(gamma * N)) - 1]), max_iter)
            kept = torch.nonzero(c <= t_star)[:, 0]
        acc, _ = _prune64(X, pos[kept], h, flat)
        M = acc.shape[0]
        if all_seeds or not (N < 8 * M and N < n):
            break
        N2 = min(2 * N, n)
        new = _permutation(n, rng_seed, N, N2)
        p2, c2 = _travel64(X, X[new], h, tol, max_iter, flat, sphere)
        pos, conv, N = torch.cat([pos, p2]), torch.cat([conv, c2]), N2
    fine, _ = _travel64(X, pos[kept[acc]], h, 1e-5 * h, 50, flat, sphere)
    acc, score = _prune64(X, fine, h, flat)
    modes = fine[acc]   # in order of density already
    if not want_margins:
        return modes, None
    margins = torch.empty(n, dtype=torch.float64, device=DEV)
    if M < 2 or modes.shape[0] < 2:
        return modes, margins.fill_(math.inf)
    step = max(1, _PAIRS // modes.shape[0])
    for a in range(0, n, step):
        two = _d2(X[a:a + step], modes).sqrt().topk(2, dim=1, largest=False).values
        margins[a:a + step] = two[:, 1] - two[:, 0]
    return modes, margins


def _unrolled64(X, Y0, G, h, T):
    """Positions after T updates, and the gradients, of one set."""
    Ys = [Y0]
    for _ in range(T):
        Ys.append(_update64(X, Ys[-1], h)[0])
    dX, g, dh = torch.zeros_like(X), G, torch.zeros((), dtype=X.dtype, device=X.device)
    h2 = h * h
    step = max(1, _PAIRS // X.shape[0])
    for t in range(T - 1, -1, -1):
        gn = torch.empty_like(g)
        for a in range(0, g.shape[0], step):
            y, mu, gg = Ys[t][a:a + step], Ys[t + 1][a:a + step], g[a:a + step]
            D = _d2(y, X)
            P = torch.exp(D * (-0.5 / h2))
            P /= P.sum(1, keepdim=True)
            PA = P * (gg @ X.T - (gg * mu).sum(1, keepdim=True))
            gn[a:a + step] = (PA @ X - PA.sum(1, keepdim=True) * mu) / h2
            dX += P.T @ gg - (PA.sum(0)[:, None] * X - PA.T @ y) / h2
            dh += (PA * D).sum() / (h2 * h)
        g = gn
    return Ys[-1], dX, g, dh


def exact(case, seed):
    if _evals(case) > 6e10:   # over about 20 seconds
        return None
    kind = case["kind"]
    data = _inputs(case, seed)
    rng_seed = int(seed) % 1000
    if kind in ("step", "coarse"):
        return list(_update64(data[0].double(), data[1].double(), case["h"]))
    if kind == "cluster":
        modes, margins = _cluster64(data, case["h"], rng_seed, case["all_seeds"],
                                    case["kernel"] == "flat", case["metric"] == "cosine")
        return [_rows(modes, MODES), None, None, margins]
    if kind == "host":
        modes = _cluster64(data, case["h"], rng_seed, want_margins=False)[0]
        return [_rows(modes, MODES), None, None]
    if kind == "batched":
        X, offs = data
        got = [_cluster64(X[int(a):int(b)], case["h"], rng_seed)
               for a, b in zip(offs[:-1], offs[1:])]
        return [_rows(torch.cat([m for m, _ in got]), SET_MODES * case["B"]), None, None,
                torch.cat([m for _, m in got])]
    X, Y0, G = (v.double() for v in data)
    got = [_unrolled64(X[b], Y0[b], G[b], case["h"], case["T"]) for b in range(case["B"])]
    return [torch.stack([r[0] for r in got]), torch.stack([r[1] for r in got]),
            torch.stack([r[2] for r in got]), sum(r[3] for r in got)]
