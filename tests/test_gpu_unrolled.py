"""GPU parity of the differentiable unrolled steps and their adjoint (A9).

Forward and adjoint are compared with the FP64 oracle (whose adjoint is
pinned by finite differences and autograd) on sets small enough for its dense
numpy code; FP32 budget: relative 2e-4 of each quantity's scale (weights carry
~1e-6 relative error, sums over <= 512 terms).  At the full configuration
(8 sets x 16,384 points, d = 16, T = 20, k = 5) the forward is checked on
sampled seeds (trajectories are independent of each other) and the backward
for finiteness and for the scaling identity
    h dL/dh = Y_T . G - X . dL/dX - Y0 . dL/dY0
(Y_T(cX, cY0, ch) = c Y_T(X, Y0, h), so differentiating L = G . Y_T along
(X, Y0, h) at c = 1 gives it).  A seed farther than 13 h from every point,
whose Gaussian weights all underflow in FP32, must come out as the oracle's
(which weighs relative to the nearest point), with finite gradients.
"""
import os
import subprocess
import sys
import threading

import numpy as np
import pytest
import torch

import fms_inputs as fi
import oracle as orc

pytestmark = pytest.mark.gpu

fms = pytest.importorskip("paper_2112_13891_gb300")
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _sets(seed, B, n, d, k=4):
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(B):
        c = rng.uniform(0, 12, (k, d))
        X = c[rng.integers(0, k, n)] + rng.standard_normal((n, d))
        out.append(X)
    return np.stack(out).astype(np.float32)


@pytest.mark.parametrize("d,n,T,k", [(2, 200, 3, 2), (4, 257, 4, 3), (16, 300, 5, 2), (7, 130, 2, 5),
                                     (1, 150, 3, 2), (32, 140, 3, 2)])
def test_forward_and_adjoint_match_oracle(d, n, T, k):
    B, h = 2, 2.0
    X = _sets(d * 100 + n, B, n, d)
    rng = np.random.default_rng(7)
    Y0 = (X + 0.3 * rng.standard_normal(X.shape)).astype(np.float32)
    G = rng.standard_normal(X.shape).astype(np.float32)
    Xt, Yt = torch.from_numpy(X).cuda(), torch.from_numpy(Y0).cuda()
    YT, ck = fms.unrolled_forward(Xt, Yt, h, T, k)
    dX, dY, dh = fms.unrolled_backward(Xt, ck, n, h, T, k, torch.from_numpy(G).cuda())
    torch.cuda.synchronize()
    for b in range(B):
        ref = orc.unrolled_forward(X[b], Y0[b], h, T)[-1]
        assert np.abs(YT[b].cpu().numpy() - ref).max() <= 2e-4 * (1 + np.abs(ref).max())
        rdX, rdY, rdh = orc.unrolled_backward(X[b], Y0[b], h, T, G[b])
        for got, want in ((dX[b], rdX), (dY[b], rdY)):
            got = got.cpu().numpy().astype(np.float64)
            assert np.abs(got - want).max() <= 2e-4 * (1 + np.abs(want).max()), np.abs(got - want).max()
        assert abs(dh[b].item() - rdh) <= 2e-4 * (1 + abs(rdh))


def test_autograd_function():
    B, n, d, h, T, k = 1, 150, 4, 1.5, 3, 2
    X = _sets(3, B, n, d)
    Xt = torch.from_numpy(X).cuda().requires_grad_(True)
    Yt = (torch.from_numpy(X).cuda() + 0.1).requires_grad_(True)
    ht = torch.tensor(h, device="cuda", requires_grad=True)
    out = fms.unrolled_mean_shift(Xt, Yt, ht, T, k)
    G = torch.randn_like(out)
    (out * G).sum().backward()
    rdX, rdY, rdh = orc.unrolled_backward(X[0], (X[0] + 0.1).astype(np.float32), h, T,
                                          G[0].cpu().numpy())
    assert np.abs(Xt.grad[0].cpu().numpy() - rdX).max() <= 2e-4 * (1 + np.abs(rdX).max())
    assert np.abs(Yt.grad[0].cpu().numpy() - rdY).max() <= 2e-4 * (1 + np.abs(rdY).max())
    assert abs(ht.grad.item() - rdh) <= 2e-4 * (1 + abs(rdh))


def test_full_configuration_sampled():
    w = fi.unrolled_16d()
    X = w.X                                        # [8, 16384, 16]
    B, n, d = X.shape
    h, T, k = w.h, w.T, w.k_ckpt
    Xt = torch.from_numpy(X).cuda()
    YT, ck = fms.unrolled_forward(Xt, Xt, h, T, k)
    G = torch.randn_like(YT)
    dX, dY, dh = fms.unrolled_backward(Xt, ck, n, h, T, k, G)
    torch.cuda.synchronize()
    rng = np.random.default_rng(0)
    for b in (0, B - 1):
        idx = rng.choice(n, 8, replace=False)
        ref = orc.unrolled_forward(X[b], X[b][idx], h, T)[-1]
        assert np.abs(YT[b].cpu().numpy()[idx] - ref).max() <= 1e-3 * (1 + np.abs(ref).max())
    assert torch.isfinite(dX).all() and torch.isfinite(dY).all() and torch.isfinite(dh).all()
    # scale invariance: Y_T(cX, cY0, ch) = c Y_T(X, Y0, h)  =>  h dL/dh = -(X.dX + Y0.dY) + Y_T.G
    lhs = h * dh.cpu().numpy()
    rhs = (-(Xt * dX).sum(dim=(1, 2)) - (Xt * dY).sum(dim=(1, 2)) + (YT * G).sum(dim=(1, 2)))
    rhs = rhs.double().cpu().numpy()
    scale = ((Xt * dX).abs().sum(dim=(1, 2)) + (YT * G).abs().sum(dim=(1, 2))).double().cpu().numpy()
    assert np.all(np.abs(lhs - rhs) <= 1e-3 * scale), (lhs, rhs)


def test_far_seed_matches_oracle():
    # seed 0 starts 20 h away from every point: exp(-D^2 / 2h^2) < 1e-86, so
    # every unshifted FP32 weight is 0; the library recomputes such seeds with
    # weights relative to the nearest point, as the oracle does
    B, n, d, h, T, k = 1, 180, 3, 1.0, 3, 2
    X = _sets(44, B, n, d)
    rng = np.random.default_rng(9)
    Y0 = (X + 0.2 * rng.standard_normal(X.shape)).astype(np.float32)
    far = X[0].max(axis=0) + 20.0 * h
    Y0[0, 0] = far.astype(np.float32)
    D = np.sqrt(((X[0].astype(np.float64) - Y0[0, 0]) ** 2).sum(-1))
    assert D.min() > 15.0 * h
    G = rng.standard_normal(Y0.shape).astype(np.float32)
    Xt, Yt = torch.from_numpy(X).cuda(), torch.from_numpy(Y0).cuda()
    YT, ck = fms.unrolled_forward(Xt, Yt, h, T, k)
    dX, dY, dh = fms.unrolled_backward(Xt, ck, n, h, T, k, torch.from_numpy(G).cuda())
    torch.cuda.synchronize()
    ref = orc.unrolled_forward(X[0], Y0[0], h, T)[-1]
    got = YT[0].cpu().numpy()
    assert np.all(np.isfinite(got))
    assert np.abs(got - ref).max() <= 2e-4 * (1 + np.abs(ref).max())
    rdX, rdY, rdh = orc.unrolled_backward(X[0], Y0[0], h, T, G[0])
    for g_, want in ((dX[0], rdX), (dY[0], rdY)):
        g_ = g_.cpu().numpy().astype(np.float64)
        assert np.all(np.isfinite(g_))
        assert np.abs(g_ - want).max() <= 2e-4 * (1 + np.abs(want).max())
    assert abs(dh[0].item() - rdh) <= 2e-4 * (1 + abs(rdh))


def test_fp64_kernels_match_oracle_tightly():
    # the FP64 entry points run the same kernels in double precision: forward
    # and adjoint agree with the FP64 oracle to ~1e-10 (rounding order only)
    B, n, d, h, T, k = 2, 120, 4, 1.5, 4, 3
    X = _sets(61, B, n, d).astype(np.float64)
    rng = np.random.default_rng(3)
    Y0 = X + 0.25 * rng.standard_normal(X.shape)
    G = rng.standard_normal(X.shape)
    Xt, Yt = torch.from_numpy(X).cuda(), torch.from_numpy(Y0).cuda()
    YT, ck = fms.unrolled_forward(Xt, Yt, h, T, k)
    assert YT.dtype == torch.float64
    dX, dY, dh = fms.unrolled_backward(Xt, ck, n, h, T, k, torch.from_numpy(G).cuda())
    torch.cuda.synchronize()
    for b in range(B):
        ref = orc.unrolled_forward(X[b], Y0[b], h, T)[-1]
        assert np.abs(YT[b].cpu().numpy() - ref).max() <= 1e-10 * (1 + np.abs(ref).max())
        rdX, rdY, rdh = orc.unrolled_backward(X[b], Y0[b], h, T, G[b])
        for got, want in ((dX[b], rdX), (dY[b], rdY)):
            got = got.cpu().numpy()
            assert np.abs(got - want).max() <= 1e-9 * (1 + np.abs(want).max())
        assert abs(dh[b].item() - rdh) <= 1e-9 * (1 + abs(rdh))


def test_gradcheck_fp64_on_gpu():
    # torch.autograd.gradcheck of the library's adjoint (FP64 kernels on the
    # GPU) against central finite differences of its own forward, n = 64, d = 4
    B, n, d, T, k = 1, 64, 4, 3, 2
    X = torch.from_numpy(_sets(62, B, n, d).astype(np.float64)).cuda().requires_grad_(True)
    g = torch.Generator(device="cuda").manual_seed(5)
    Y0 = (X.detach() + 0.2 * torch.randn(X.shape, generator=g, device="cuda",
                                          dtype=torch.float64)).requires_grad_(True)
    h = torch.tensor(1.7, dtype=torch.float64, device="cuda", requires_grad=True)
    fn = lambda X_, Y_, h_: fms.unrolled_mean_shift(X_, Y_, h_, T, k)
    assert torch.autograd.gradcheck(fn, (X, Y0, h), eps=1e-6, atol=1e-7, rtol=1e-5)


def _wide_sets(seed, B, n, d, k, box, sigma=1.0):
    rng = np.random.default_rng(seed)
    return np.stack([rng.uniform(0, box, (k, d))[rng.integers(0, k, n)]
                     + sigma * rng.standard_normal((n, d)) for _ in range(B)]).astype(np.float32)


# Sorted cells serve B n m >= 4,194,304: the sizes lie just above it, with a last
# sort block of one row (2049), fewer seeds than points, one large cluster (every
# cell seen), and clusters of very different sizes.
@pytest.mark.parametrize("B,n,m,d,k,box,T,kk", [
    (1, 2049, 2049, 3, 8, 100.0, 5, 2), (1, 4200, 1001, 16, 6, 50.0, 4, 3),
    (2, 1500, 1500, 2, 1, 5.0, 3, 9), (1, 2050, 2048, 32, 5, 40.0, 3, 1),
    (1, 2100, 2000, 7, 4, 30.0, 11, 10)])
def test_sorted_cells_match_oracle(B, n, m, d, k, box, T, kk):
    h = 2.0
    X = _wide_sets(d * 7 + n, B, n, d, k, box)
    rng = np.random.default_rng(5)
    Y0 = (X[:, :m] + 0.3 * rng.standard_normal((B, m, d))).astype(np.float32)
    if d == 3:
        Y0[0, 5] = X[0].max(axis=0) + 60.0       # every weight zero in FP32
        Y0[0, 6] = X[0].max(axis=0) + 5.0 * h    # W far below 1: the cutoff widens
    G = rng.standard_normal(Y0.shape).astype(np.float32)
    Xt, Yt = torch.from_numpy(X).cuda(), torch.from_numpy(Y0).cuda()
    YT, ck = fms.unrolled_forward(Xt, Yt, h, T, kk)
    dX, dY, dh = fms.unrolled_backward(Xt, ck, m, h, T, kk, torch.from_numpy(G).cuda())
    again = fms.unrolled_backward(Xt, ck, m, h, T, kk, torch.from_numpy(G).cuda())
    torch.cuda.synchronize()
    for one, two in zip((dX, dY, dh), again):
        assert torch.equal(one, two)
    for b in range(B):
        ref = orc.unrolled_forward(X[b], Y0[b], h, T)[-1]
        assert np.abs(YT[b].cpu().numpy() - ref).max() <= 2e-4 * (1 + np.abs(ref).max())
        rdX, rdY, rdh = orc.unrolled_backward(X[b], Y0[b], h, T, G[b])
        for got, want in ((dX[b], rdX), (dY[b], rdY)):
            got = got.cpu().numpy().astype(np.float64)
            assert np.abs(got - want).max() <= 2e-4 * (1 + np.abs(want).max())
        assert abs(dh[b].item() - rdh) <= 2e-4 * (1 + abs(rdh))


def test_sorted_cells_f64_match_oracle():
    B, n, d, h, T, k = 1, 2100, 3, 2.0, 3, 2
    X = _wide_sets(3, B, n, d, 6, 60.0).astype(np.float64)
    G = np.random.default_rng(1).standard_normal(X.shape)
    Xt = torch.from_numpy(X).cuda()
    YT, ck = fms.unrolled_forward(Xt, Xt, h, T, k)
    dX, dY, dh = fms.unrolled_backward(Xt, ck, n, h, T, k, torch.from_numpy(G).cuda())
    torch.cuda.synchronize()
    ref = orc.unrolled_forward(X[0], X[0], h, T)[-1]
    rdX, rdY, rdh = orc.unrolled_backward(X[0], X[0], h, T, G[0])
    assert np.abs(YT[0].cpu().numpy() - ref).max() <= 1e-9 * (1 + np.abs(ref).max())
    assert np.abs(dX[0].cpu().numpy() - rdX).max() <= 1e-9 * (1 + np.abs(rdX).max())
    assert np.abs(dY[0].cpu().numpy() - rdY).max() <= 1e-9 * (1 + np.abs(rdY).max())
    assert abs(dh[0].item() - rdh) <= 1e-9 * (1 + abs(rdh))


# Few unsorted points stay in shared memory beside the backward's static arrays, so the
# dynamic size alone passes 48 KB (the default limit, which counts both) a few points
# later than the sum does: with 16 warps a block at n = 2,067 .. 2,074 for d = 3, and
# elsewhere for the other widths.  A fresh process: a larger call raises the limit.
_SWEEP = """
import torch
import paper_2112_13891_gb300 as fms
g = torch.Generator(device="cuda").manual_seed(1)
for B, ns, m, d, dt in ((1, range(2060, 2081), 700, 3, torch.float32),
                        (1, range(2446, 2462), 3000, 3, torch.float32),
                        (4, range(740, 755), 100, 6, torch.float32),
                        (1, range(368, 380), 60, 12, torch.float32),
                        (1, range(800, 1300, 3), 64, 3, torch.float64)):
    for n in ns:
        X = torch.randn((B, n, d), generator=g, device="cuda", dtype=dt)
        Y = torch.randn((B, m, d), generator=g, device="cuda", dtype=dt)
        out, ck = fms.unrolled_forward(X, Y, 1.0, 2, 2)
        dX, dY, dh = fms.unrolled_backward(X, ck, m, 1.0, 2, 2, torch.ones_like(Y))
        assert torch.isfinite(dX).all() and torch.isfinite(dY).all(), (B, n, m, d)
print("done")
"""


def test_resident_points_of_every_size():
    r = subprocess.run([sys.executable, "-c", _SWEEP], capture_output=True, text=True, cwd=ROOT,
                       timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, r.stderr[-2000:]


def test_threads_with_different_sizes():
    """Calls of two host threads on their own streams, whose blocks take different amounts
    of shared memory, do not disturb each other."""
    def work(n, failed):
        try:
            with torch.cuda.stream(torch.cuda.Stream()):
                g = torch.Generator(device="cuda").manual_seed(n)
                X = torch.randn((1, n, 3), generator=g, device="cuda")
                Y = torch.randn((1, 700, 3), generator=g, device="cuda")
                first = None
                for _ in range(300):
                    out, ck = fms.unrolled_forward(X, Y, 1.0, 1, 1)
                    dX, dY, dh = fms.unrolled_backward(X, ck, 700, 1.0, 1, 1, torch.ones_like(Y))
                    first = first if first is not None else dX.clone()
                assert torch.equal(first, dX)
                torch.cuda.current_stream().synchronize()
        except Exception as e:   # (seen by the main thread)
            failed.append(repr(e))
    failed = []
    ts = [threading.Thread(target=work, args=(n, failed)) for n in (2900, 2200, 2500)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not failed, failed


# One blob, or blobs in reach of each other: every point counts for every seed, and the
# sorted form takes them all (the sizes as above; FP64 alike).
@pytest.mark.parametrize("B,n,m,d,k,box,T,kk,dt", [
    (1, 2049, 2049, 3, 1, 1.0, 5, 2, np.float32), (1, 4200, 1001, 16, 3, 2.0, 4, 3, np.float32),
    (5, 1000, 900, 2, 4, 4.0, 3, 9, np.float32), (1, 2050, 2048, 32, 1, 1.0, 3, 1, np.float32),
    (2, 1500, 1450, 7, 2, 2.0, 4, 3, np.float64)])
def test_sorted_cells_that_leave_nothing_out(B, n, m, d, k, box, T, kk, dt):
    h = 2.0
    X = _wide_sets(d * 7 + n, B, n, d, k, box).astype(dt)
    rng = np.random.default_rng(5)
    Y0 = (X[:, :m] + 0.3 * rng.standard_normal((B, m, d))).astype(dt)
    if d == 3:
        Y0[0, 5] = X[0].max(axis=0) + 60.0       # every weight zero in FP32
    G = rng.standard_normal(Y0.shape).astype(dt)
    YT, ck = fms.unrolled_forward(torch.from_numpy(X).cuda(), torch.from_numpy(Y0).cuda(), h, T, kk)
    dX, dY, dh = fms.unrolled_backward(torch.from_numpy(X).cuda(), ck, m, h, T, kk,
                                       torch.from_numpy(G).cuda())
    torch.cuda.synchronize()
    tol = 2e-4 if dt == np.float32 else 1e-9
    for b in range(B):
        ref = orc.unrolled_forward(X[b], Y0[b], h, T)[-1]
        assert np.abs(YT[b].cpu().numpy() - ref).max() <= tol * (1 + np.abs(ref).max())
        rdX, rdY, rdh = orc.unrolled_backward(X[b], Y0[b], h, T, G[b])
        for got, want in ((dX[b], rdX), (dY[b], rdY)):
            got = got.cpu().numpy().astype(np.float64)
            assert np.abs(got - want).max() <= tol * (1 + np.abs(want).max())
        assert abs(dh[b].item() - rdh) <= tol * (1 + abs(rdh))
