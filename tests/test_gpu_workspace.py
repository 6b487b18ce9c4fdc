"""A call writes nothing beyond the bytes that its size function asks for: every entry
point that takes a workspace, at sizes where the points are sorted into cells (chunks of
1,024 rows: a multiple and a remainder), with guard bytes behind it."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

fms = pytest.importorskip("paper_2112_13891_gb300")
GUARD = 1 << 16


def _blobs(seed, n, d, k=12, box=50.0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    c = box * torch.rand((k, d), generator=g, device="cuda")
    return c[torch.randint(k, (n,), generator=g, device="cuda")] + torch.randn(
        (n, d), generator=g, device="cuda")


class _Guarded(fms.Workspace):
    def __init__(self, nbytes):
        super().__init__(nbytes + GUARD)
        self.all = self.buf
        self.all.fill_(0xA5)
        self.buf = self.all[:nbytes]

    def check(self):
        torch.cuda.synchronize()
        assert (self.all[-GUARD:] == 0xA5).all()


@pytest.mark.parametrize("n", [16_384, 20_001, 262_144, 270_337])
@pytest.mark.parametrize("d,kw", [(16, {}), (9, dict(metric="cosine")), (3, {}),
                                  (3, dict(all_seeds=True))])
def test_cluster(n, d, kw):
    X = _blobs(n + d, n, d)
    ws = _Guarded(fms.workspace_size(n, d, **kw))
    for _ in range(2):   # (the second call as a graph)
        fms.cluster(X, 2.5, 2.5e-3, 300, workspace=ws, **kw)
    ws.check()


@pytest.mark.parametrize("n,m", [(262_144, 2_400), (65_536, 20_480), (50_000, 20_001)])
@pytest.mark.parametrize("d", [3, 9, 32])
def test_steps(n, m, d):
    X = _blobs(n + d, n, d)
    Y = X[:m] + 0.1
    want = fms.mean_shift_step(X[:, :], Y, 2.5)
    for fn, size in ((fms.mean_shift_step, fms._lib.fms_step_workspace_size),
                     (fms.mean_shift_step_coarse, fms._lib.fms_coarse_step_workspace_size)):
        ws = _Guarded(int(size(n, d, m)))
        out = fn(X, Y, 2.5, workspace=ws)
        ws.check()
        assert (out - want).abs().max() < 0.1


@pytest.mark.parametrize("d", [3, 16])
def test_batched(d):
    X = _blobs(d, 61_440, d)
    offs = np.array([0, 2048, 4096, 40_000, 61_440], dtype=np.int64)
    o = fms.make_options()
    ws = _Guarded(int(fms._lib.fms_batched_workspace_size(offs.ctypes.data, 4, d,
                                                          fms.ctypes.byref(o))))
    for _ in range(2):
        fms.cluster_batched(X, 2.5, 2.5e-3, 300, offsets=offs, workspace=ws, max_modes=64)
    ws.check()
