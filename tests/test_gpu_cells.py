"""Sorted cells and whole trajectories in one launch, at the sizes where their
rules begin: one update by groups (n m times the padded width >= 2.5e9), a block
per seed (d > 7; points sorted from n = 16,384 on) and every point a seed by groups
(d <= 7; sorted from n = 8,192 on), against the FP64 oracle.

Tolerances: one update as in test_gpu_step_parity (FP32 weights, sums of n terms);
clusterings by the cluster parity bar (modes within 1e-3 h, identical labels away
from ties)."""
import numpy as np
import pytest
import torch

import fms_inputs as fi
import oracle as orc
from fms_compare import compare_clustering

pytestmark = pytest.mark.gpu

fms = pytest.importorskip("paper_2112_13891_gb300")


def _blobs(seed, n, d, k, box, sigma):
    rng = np.random.default_rng(seed)
    c = rng.uniform(0, box, (k, d))
    return (c[rng.integers(0, k, n)] + sigma * rng.standard_normal((n, d))).astype(np.float32)


# just above the rule's line; a last sort block of one row; fewer seeds than points
@pytest.mark.parametrize("n,m,d,box,h", [(20_620, 20_623, 3, 200.0, 5.0), (14_580, 14_579, 6, 60.0, 4.0),
                                         (10_241, 10_400, 9, 50.0, 2.5), (51_201, 2_080, 16, 50.0, 2.5),
                                         (25_000, 25_003, 3, 200.0, 5.0), (17_680, 17_679, 6, 60.0, 4.0),
                                         (12_289, 12_800, 9, 50.0, 2.5), (76_801, 2_049, 16, 50.0, 2.5),
                                         (8_900, 8_891, 32, 12.0, 1.5),
                                         # 256, 257 chunks of the sort and many: a scan of its counters
                                         (262_144, 2_400, 3, 200.0, 5.0), (262_145, 2_049, 5, 60.0, 4.0),
                                         (1_500_000, 2_050, 9, 50.0, 2.5),
                                         (7_300, 7_291, 32, 12.0, 1.5)])
def test_step_by_groups(n, m, d, box, h):
    X = _blobs(n, n, d, 12, box, 1.0)
    rng = np.random.default_rng(1)
    Y = (X[rng.integers(0, n, m)] + 0.3 * rng.standard_normal((m, d))).astype(np.float32)
    # 5 h beyond the outermost point: W ~ 1e-5 of a point's, so the cutoff widens
    # (every weight still above 2^-126 = exp(-87.3): exp(-||y - x||^2 / 2h^2) at 5 h
    # is exp(-12.5))
    Y[7] = X[X[:, 0].argmax()]
    Y[7, 0] += 5.0 * h
    Y[m - 1] = X.max(axis=0) + 100.0 * h            # every weight zero
    out, W = fms.mean_shift_step(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), h,
                                 with_wsum=True)
    out, W = out.cpu().numpy().astype(np.float64), W.cpu().numpy().astype(np.float64)
    pick = np.unique(np.r_[0, 7, m - 2, rng.integers(0, m - 1, 200)])
    ref, refW = orc.step(X, Y[pick], h), orc.kde(X, Y[pick], h)
    assert np.abs(W[pick] / refW - 1).max() <= 1e-4
    assert np.abs(out[pick] - ref).max() <= 2e-4 * h + 2.0 ** -20 * np.abs(ref).max()
    assert W[m - 1] == 0.0 and np.isnan(out[m - 1]).all()   # 0 / 0, as without cells


@pytest.mark.parametrize("n", [7_300, 8_900])
def test_step_by_groups_keeps_nonfinite(n):
    m = n
    X = torch.randn((n, 32), device="cuda")
    X[5, 3] = float("inf")
    out = fms.mean_shift_step(X, torch.randn((m, 32), device="cuda"), 1.0)
    assert torch.isnan(out).any(dim=1).all()   # an infinite point reaches every seed


def _cluster(w, **kw):
    X = torch.from_numpy(w.X).cuda()
    res = fms.cluster(X, w.h, w.tol, w.max_iter, **kw)
    again = fms.cluster(X, w.h, w.tol, w.max_iter, **kw)
    assert torch.equal(res.modes, again.modes) and torch.equal(res.labels, again.labels)
    ref = orc.cluster(w.X, w.h, w.tol, w.max_iter, **kw)
    cmp = compare_clustering(res.modes.cpu().numpy(), res.labels.cpu().numpy(), ref, w.h)
    assert cmp["mode_ok"] and cmp["label_mismatch"] == 0, cmp
    return res, ref


@pytest.mark.parametrize("d,per,sigma,kw", [
    (8, 1366, 1.0, {}), (9, 1366, 1.0, {}), (16, 1366, 1.0, {}), (16, 1365, 1.0, {}),
    (33, 1400, 0.5, {}), (64, 1366, 0.4, {}), (16, 1400, 0.6, dict(kernel="flat")),
    (8, 2731, 1.0, {}), (9, 2730, 1.0, {}), (16, 2731, 1.0, {}), (33, 2740, 0.5, {}), (64, 2731, 0.4, {}),
    (16, 2750, 0.6, dict(kernel="flat"))])
def test_block_per_seed(d, per, sigma, kw):
    # 6 blobs: 16,386 points sorted, 16,380 not
    w = fi.separated_blobs(seed=d + per, k=6, d=d, per=per, sigma=sigma,
                           h=2.0 if not kw else 8.0)
    res, ref = _cluster(w, rng_seed=2, **kw)
    assert res.stats["n_seeds_final"] == ref.n_seeds and res.stats["t_star_last"] == ref.t_star[-1]


def test_block_per_seed_cosine():
    for per in (700, 1400):
        _cluster(fi.directional_blobs(seed=3, k=12, d=16, per=per, spread=0.05, h=0.15),
                 metric="cosine", rng_seed=1)


@pytest.mark.parametrize("d,n,kw", [(3, 4096, {}), (3, 4095, {}), (1, 4500, {}), (7, 4321, {}),
                                    (2, 63, {}), (3, 4100, dict(kernel="flat")),
                                    (3, 4100, dict(metric="cosine")), (3, 8192, {}), (3, 8191, {}),
                                    (1, 8500, {}), (7, 8321, {}), (3, 8200, dict(kernel="flat")),
                                    (3, 8300, dict(metric="cosine"))])
def test_every_point_a_seed(d, n, kw):
    if kw.get("metric") == "cosine":
        w = fi.directional_blobs(seed=5, k=5, d=d, per=n // 5, spread=0.05, h=0.15)
    else:
        k = 3 if d == 1 else 6
        w = fi.separated_blobs(seed=d + n, k=k, d=d, per=max(1, n // k), sigma=1.0,
                               h=2.0 if "kernel" not in kw else 6.0)
        w["X"] = np.concatenate([w.X, w.X[: n - len(w.X)] + 0.01]).astype(np.float32)
    _cluster(w, all_seeds=True, **kw)


# d > 7: sets below and above the mean size from which they are sorted (512), sets of
# one chunk, one row more and several chunks of the sort (1,024 rows), unconverged
# seeds kept (gamma = 1)
@pytest.mark.parametrize("d,per,kw", [(8, (100, 60, 128), {}), (16, (256, 205, 700), {}),
                                      (33, (256, 341, 200), {}), (9, (300, 120, 205), dict(gamma=1.0))])
def test_batched_queue(d, per, kw):
    h = 2.5
    sets = [fi.separated_blobs(seed=7 * d + i, k=4 + (i > 0), d=d, per=p, sigma=0.8, h=h)
            for i, p in enumerate(per)]
    X = [torch.from_numpy(w.X).cuda() for w in sets]
    res = fms.cluster_batched(X, h, 1e-3 * h, 300, rng_seed=3, max_modes=64, **kw)
    off = np.concatenate([[0], np.cumsum([w.X.shape[0] for w in sets])])
    for b, w in enumerate(sets):
        ref = orc.cluster(w.X, h, 1e-3 * h, 300, rng_seed=3, **kw)
        cmp = compare_clustering(res.modes[b].cpu().numpy(),
                                 res.labels[off[b]:off[b + 1]].cpu().numpy(), ref, h)
        assert cmp["mode_ok"] and cmp["label_mismatch"] == 0, (b, cmp)


# the tensor-core step from 6e8 pairs on: tiles of one cell, tile pairs out of reach
# skipped.  The bound is the BF16 one of test_gpu_coarse_step.
@pytest.mark.parametrize("n,m,d,box,h", [(24_577, 24_500, 9, 60.0, 2.5), (49_000, 12_300, 16, 50.0, 2.5),
                                         (600_001, 1_001, 3, 100.0, 3.0), (24_600, 24_601, 32, 3.0, 2.0)])
def test_coarse_step_by_cells(n, m, d, box, h):
    from test_gpu_coarse_step import _bound
    X = _blobs(n + d, n, d, 12, box, 1.0)
    rng = np.random.default_rng(2)
    Y = (X[rng.integers(0, n, m)] + 0.3 * rng.standard_normal((m, d))).astype(np.float32)
    Y[3] = X.max(axis=0) + 100.0 * h                # every weight zero
    out, W = fms.mean_shift_step_coarse(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), h,
                                        with_wsum=True)
    out, W = out.cpu().numpy().astype(np.float64), W.cpu().numpy().astype(np.float64)
    pick = np.unique(np.r_[0, m - 1, rng.integers(4, m, 24)])
    ref, refW = orc.step(X, Y[pick], h), orc.kde(X, Y[pick], h)
    bnd, eps = _bound(X, Y[pick], h, ref)
    assert np.all(np.abs(out[pick] - ref).max(axis=1) <= bnd)
    assert np.all(np.abs(W[pick] - refW) <= 1.5 * eps * refW)
    assert W[3] == 0.0 and np.isnan(out[3]).all()


def _greedy(X, score, r2):
    """Greedy radius suppression in order of (score descending, index ascending);
    exact for integer points."""
    alive = np.ones(len(X), bool)
    out = []
    for i in np.lexsort((np.arange(len(X)), -score)):
        if alive[i]:
            out.append(i)
            alive &= ~(((X - X[i]) ** 2).sum(axis=1) < r2)
    return X[out]


# Integer points far apart next to h stay where they are, with their multiplicity for a
# density, so the merge alone decides: every comparison of distances is between an
# integer and r^2 = 4.5.  Neighbours lie in chains, so that passing over a candidate is
# often wrong.  Sizes at the edges of the sort (256 counted, 512, 1,024, 2,048, 8,192
# slots) and of a batch; at d = 32 and 64 not all coordinates fit in shared memory.
# d <= 7: densities are exact, many of them tied (lowest index first).  Above, the
# densities are good to |s x|^2 2^-23 (s = 0.85 / h, 45 a coordinate, d = 64: 1 %), so no two
# points have multiplicities closer than 1 in 64 and their order is certain.
@pytest.mark.parametrize("refine", [False, True])
@pytest.mark.parametrize("n,d", [(31, 3), (33, 3), (256, 2), (257, 7), (1025, 5), (2049, 4),
                                 (8200, 3), (22, 9), (23, 16), (32, 16), (54, 32), (63, 32),
                                 (45, 64), (64, 64)])
def test_merge_of_points_that_stay(n, d, refine):
    rng = np.random.default_rng(n + d)
    k = max(n // (12 if d <= 7 else 4), 1)
    side = max(int(np.ceil(k ** (1.0 / d))), 1)
    centre = 3 * rng.integers(0, side + 1, (k, d))
    X = centre[rng.integers(0, k, n)]
    for _ in range(3):
        X[np.arange(n), rng.integers(0, d, n)] += rng.integers(-1, 2, n)
    X, times = np.unique(X, axis=0, return_counts=True)
    at = rng.permutation(len(X))
    X, times = X[at], times[at] if d <= 7 else 1 + np.arange(len(X))
    rows = np.repeat(X, times, axis=0).astype(np.float32)
    r = fms.cluster(torch.from_numpy(rows).cuda(), 0.05 if d <= 7 else 0.15, 1e-3, 20,
                    all_seeds=True, gamma=1.0, merge_radius=float(np.sqrt(4.5)),
                    skip_refine=not refine, precision="fp32")
    got = np.rint(r.modes.cpu().numpy()).astype(int)
    want = _greedy(X, times, 4.5)
    assert len(got) == len(want)
    assert {tuple(p) for p in got} == {tuple(p) for p in want}


def test_block_per_seed_long_sums():
    """A window that holds every point: the mode is their mean, and its error that of the
    sums of x - y.  Rounding the differences to FP32 leaves 2.6e-9 whatever n is (y's last
    bits, the same for all rows); sums of 128 terms at a time add 7e-10 at random, one
    chain of n / 32 terms (whose terms have one sign for long runs: the rows of a cell lie
    on one side) 4e-9 at n = 10^6."""
    n, d = 1_000_000, 64
    X = 0.3 * torch.randn((n, d), generator=torch.Generator(device="cuda").manual_seed(3),
                          device="cuda")
    r = fms.cluster(X, 8.0, 8e-3, 50, kernel="flat")
    assert len(r.modes) == 1
    err = r.modes[0].double() - X.double().mean(0)
    assert err.pow(2).mean().sqrt().item() <= 3.6e-9 and err.abs().max().item() <= 9e-9


@pytest.mark.parametrize("d,B", [(16, 0), (32, 0), (16, 3), (3, 3)])
def test_rounds_repeat_to_the_bit(d, B):
    """Several rounds of doubled seeds (70 clusters: 128 seeds become 1,024): the seeds that
    a round's stop leaves (half of them, at gamma = 0.5) are taken up again, and when a seed
    notices a stop depends on timing, which other work on the GPU varies here.  The modes
    (unrefined: positions of seeds), margins and labels must not."""
    sets = [fi.separated_blobs(seed=d + b, k=70, d=d, per=240 + 10 * b, sigma=0.9, h=2.0)
            for b in range(max(B, 1))]
    Xs = [torch.from_numpy(w.X).cuda() for w in sets]
    big = torch.randn((2048, 2048), device="cuda")
    side = torch.cuda.Stream()
    kw = dict(gamma=0.5, skip_refine=True, n_initial=48)
    first = None
    for i in range(24):
        if i % 3:
            with torch.cuda.stream(side):
                for _ in range(i):
                    big = (big @ big).clamp_(-1, 1)
        if B:
            r = fms.cluster_batched(Xs, 2.0, 2e-3, 300, rng_seed=1, max_modes=128, **kw)
            modes = torch.cat(r.modes)
            assert r.stats["rounds"] > 2
        else:
            r = fms.cluster(Xs[0], 2.0, 2e-3, 300, rng_seed=1, **kw)
            modes = r.modes
            assert r.stats["rounds"] > 2 and len(modes) == 70
        now = (modes, r.labels, r.margins)
        first = first or [t.clone() for t in now]
        assert all(torch.equal(a, b) for a, b in zip(first, now)), i


def test_evaluations_beyond_32_bits():
    """One seed over 18 million points that it all sees, 130 updates: 2.3e9 evaluations
    (a pass with too small a cutoff more)."""
    n, d, updates = 18_000_000, 9, 130
    X = torch.randn((n, d), generator=torch.Generator(device="cuda").manual_seed(1),
                    device="cuda")
    r = fms.cluster(X, 5.0, 1e-14, updates, n_initial=1, L=0.01, gamma=1.0, skip_refine=True)
    assert r.stats["iterations"] == updates
    assert n * updates <= r.stats["evals"] <= n * (updates + 2)


# The updates where cells would leave nothing out (one blob of half a bandwidth, blobs next
# to each other, centres of a sphere in reach of the coarse step's tiles) are made over
# every pair; both sides of the decision at the smallest sizes where it is made.
@pytest.mark.parametrize("n,m,d,k,box", [(25_000, 25_003, 3, 1, 0.0), (262_144, 2_400, 3, 6, 3.0),
                                         (17_680, 17_679, 7, 1, 0.0), (17_680, 17_700, 8, 3, 2.0),
                                         (76_801, 2_049, 16, 1, 0.0), (8_900, 8_891, 32, 4, 1.0),
                                         (25_000, 25_003, 3, 30, 100.0), (12_500, 12_600, 16, 90, 60.0)])
@pytest.mark.parametrize("coarse", [False, True])
def test_step_where_cells_may_leave_nothing_out(n, m, d, k, box, coarse):
    from test_gpu_coarse_step import _bound
    h = 1.0
    X = _blobs(n + k, n, d, k, box, 0.5)
    rng = np.random.default_rng(3)
    Y = (X[rng.integers(0, n, m)] + 0.1 * rng.standard_normal((m, d))).astype(np.float32)
    Y[5] = X.max(axis=0) + 100.0                    # every weight zero
    fn = fms.mean_shift_step_coarse if coarse else fms.mean_shift_step
    out, W = fn(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), h, with_wsum=True)
    out, W = out.cpu().numpy().astype(np.float64), W.cpu().numpy().astype(np.float64)
    pick = np.unique(np.r_[0, m - 1, rng.integers(6, m, 60)])
    ref, refW = orc.step(X, Y[pick], h), orc.kde(X, Y[pick], h)
    if coarse:
        bnd, eps = _bound(X, Y[pick], h, ref)
        assert np.all(np.abs(out[pick] - ref).max(axis=1) <= bnd)
        assert np.all(np.abs(W[pick] - refW) <= 1.5 * eps * refW)
    else:
        assert np.abs(W[pick] / refW - 1).max() <= 1e-4
        assert np.abs(out[pick] - ref).max() <= 2e-4 * h + 2.0 ** -20 * np.abs(ref).max()
    assert W[5] == 0.0 and np.isnan(out[5]).all()


# Clusters on the axes, 6.4 h apart: each reaches the others' rows, so nothing is sorted,
# and all rows in one launch (few pairs) or the steps (many) take the updates; a limit L that
# doubles the seeds across that line.  Every point a seed: all rows up to 10,240, then steps.
@pytest.mark.parametrize("d,n,k,kw", [
    (16, 20_000, 12, {}), (16, 20_000, 12, dict(n_initial=4096)), (48, 17_000, 14, dict(n_initial=512)),
    (32, 40_000, 16, {}), (9, 20_000, 7, dict(n_initial=2048)),
    (16, 20_000, 12, dict(L=128.0)), (40, 18_000, 9, dict(L=200.0)), (16, 17_000, 8, dict(gamma=1.0)),
    (16, 20_000, 12, dict(metric="cosine", L=64.0)), (16, 17_000, 5, dict(kernel="flat", n_initial=3000)),
    (7, 9_000, 6, dict(all_seeds=True)), (5, 12_000, 5, dict(all_seeds=True))])
def test_clusters_in_reach_of_each_other(d, n, k, kw):
    h = 1.0 if kw.get("metric") != "cosine" else 0.25
    if kw.get("kernel") == "flat":
        h = 3.0
    rng = np.random.default_rng(d + n)
    c = np.eye(d)[:k] * (4.5 if h >= 1.0 else 1.0)
    X = (c[rng.integers(0, k, n)] + (0.4 if h >= 1.0 else 0.03) * rng.standard_normal((n, d)))
    w = dict(X=X.astype(np.float32), h=h, tol=1e-3 * h, max_iter=300)
    res, ref = _cluster(type("W", (), w), rng_seed=2, **kw)
    assert len(ref.modes) == k
    if not kw.get("all_seeds"):
        assert res.stats["n_seeds_final"] == ref.n_seeds and res.stats["t_star_last"] == ref.t_star[-1]
