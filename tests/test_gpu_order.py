"""The order of modes of nearly the same density (and with it the label numbers).

Two blobs are exact copies of each other, a power of two apart (or, for directions,
with their coordinates in another order), but for one point that is moved by so little
that the two densities differ by 5e-9 to 5e-8 of themselves: far more than FP64 and the
refinement leave undecided (1e-10), less than FP32 weights tell apart (1e-7).  The
order must be the FP64 oracle's."""
import numpy as np
import pytest
import torch

import oracle as orc

pytestmark = pytest.mark.gpu

fms = pytest.importorskip("paper_2112_13891_gb300")


def _twins(seed, d, n, h, cosine=False):
    rng = np.random.default_rng(seed)
    q = 2.0 ** -10
    X = np.round(rng.standard_normal((n, d)) / q) * q
    if cosine:   # directions about the first axis, rolled about the last one
        X *= 2.0 ** -4
        X[:, 0] = 1.0
    unit = (lambda v: v / np.linalg.norm(v, axis=-1, keepdims=True)) if cosine else (lambda v: v)
    dens = lambda p, m: np.exp(-((unit(p) - m) ** 2).sum(-1) / (2 * h * h))
    m = unit(unit(X).mean(0))
    for _ in range(200):
        w = dens(X, m)
        m = unit((w[:, None] * unit(X)).sum(0) / w.sum())
    w = dens(X, m)
    for j in range(5, 22):   # the smallest move of a point that makes the gap
        Z = X.copy()
        Z[:, 1] += 2.0 ** -j * rng.choice([-1, 1], n)
        gap = np.abs(dens(Z, m) - w) / w.sum()
        pick = np.nonzero((gap > 1e-8) & (gap < 2e-8) & (Z.astype(np.float32) == Z).all(1))[0]
        if len(pick):
            break
    i = int(rng.choice(pick))
    twin = X.copy()
    twin[i] = Z[i]
    both = [X, twin]
    at = int(rng.integers(2))
    if cosine:
        both[at] = np.roll(both[at], d - 1, axis=1)
    else:
        both[at] = both[at] + np.where(np.arange(d) == d - 1, 64.0, 0.0)
    P = np.concatenate(both)[rng.permutation(2 * n)]
    assert (P.astype(np.float32) == P).all()
    return P.astype(np.float32)


def _check(modes, labels, X, ref, h):
    assert len(ref.scores) == 2
    gap = abs(ref.scores[0] - ref.scores[1]) / ref.scores[0]
    assert 5e-9 < gap < 5e-8, gap
    assert np.abs(modes - ref.modes).max() <= 1e-3 * h
    keep = ref.margins >= 1e-2 * h
    assert (labels[keep] == ref.labels[keep]).all()


@pytest.mark.parametrize("d,n", [(16, 300), (9, 100), (3, 300), (3, 1100), (40, 280)])
def test_batched(d, n):
    h = 2.5
    sets = [_twins(17 * i + d, d, n, h) for i in range(24)]
    r = fms.cluster_batched([torch.from_numpy(s).cuda() for s in sets], h, 1e-3 * h, 300,
                            rng_seed=5, max_modes=4)
    lab = r.labels.cpu().numpy()
    for i, s in enumerate(sets):
        ref = orc.cluster(s, h, 1e-3 * h, 300, rng_seed=5)
        _check(r.modes[i].cpu().numpy(), lab[2 * n * i:2 * n * (i + 1)], s, ref, h)


@pytest.mark.parametrize("d,n,kw", [
    (3, 2000, {}), (2, 400, {}), (7, 1000, {}), (3, 700, dict(all_seeds=True)),
    (3, 2500, dict(all_seeds=True)), (16, 500, {}), (16, 9000, {}), (48, 500, {}),
    (16, 400, dict(precision="tensor")), (9, 300, dict(all_seeds=True)),
    (16, 1000, dict(metric="cosine")), (3, 1000, dict(metric="cosine"))])
def test_single(d, n, kw):
    cosine = kw.get("metric") == "cosine"
    h = 0.25 if cosine else 2.5
    okw = {k: v for k, v in kw.items() if k != "precision"}
    for i in range(6):
        X = _twins(31 * i + d, d, n, h, cosine)
        ref = orc.cluster(X, h, 1e-3 * h, 300, rng_seed=i, **okw)
        Xt = torch.from_numpy(X).cuda()
        for _ in range(2):   # (the second call as a graph, where the form has one)
            r = fms.cluster(Xt, h, 1e-3 * h, 300, rng_seed=i, **kw)
        _check(r.modes.cpu().numpy(), r.labels.cpu().numpy(), X, ref, h)


def test_many_ties():
    """More modes than one block's ranks hold, most of them tied: one-point modes of a
    lattice (equal densities, in order of their coordinates) and blobs of a few points."""
    h = 0.05
    g = np.stack(np.meshgrid(np.arange(40), np.arange(40)), -1).reshape(-1, 2).astype(np.float32)
    twice = g[:: 7]
    X = np.concatenate([g, twice])
    X = X[np.random.default_rng(0).permutation(len(X))]
    r = fms.cluster(torch.from_numpy(X).cuda(), h, 1e-3 * h, 20, all_seeds=True)
    got = np.rint(r.modes.cpu().numpy()).astype(int)
    in_two = {tuple(p) for p in twice.astype(int)}
    want = sorted(in_two) + sorted({tuple(p) for p in g.astype(int)} - in_two)
    assert [tuple(p) for p in got] == want
