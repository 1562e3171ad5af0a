"""What some inputs may cost beside others of the same sizes: paths that still give the right bits, but by the long way round.
Times are medians of several runs on one device, and the limits lie well between what the paths take and what the way round
takes (both beside each limit)."""
import numpy as np
import pytest
import torch

from oracle import guard_oracle as go
from parity_util import assert_bit_equal, to_np

pytestmark = pytest.mark.gpu


def _window_us(X, W):
    """Time of the window kernel alone, first and later evaluations of windows that share no step."""
    from paper_2605_17879_b200 import guard
    T, R, M = X.shape
    g = guard.Guard(R, M, W, W // 2, dir=[1] * M, capacity=T, min_signals=1)
    g.set_sliding(False)
    out = g.alloc_outputs()
    us = []
    for i in range(14):
        if i == 4:
            g.profile_enable(2)
        g.ingest(X[i * W % T:i * W % T + W])
        torch.cuda.synchronize()
        g.score(out)
        torch.cuda.synchronize()
        if i >= 4:
            us.append(g.profile_read()[0] * 1000.0)
    assert g.sync_status() == 0
    g.close()
    return float(np.median(us))


@pytest.mark.parametrize("W", [64, 1000])
def test_windows_of_large_constants(W):
    """A series that stays at two million is as good as one that stays at 1.5 (1.02; 1.6 where its range misses it)."""
    R, M = (8192, 8) if W == 64 else (1024, 8)
    small = torch.full((2 * W, R, M), 1.5, device="cuda")
    large = small + 2.0e6 + torch.arange(R, device="cuda").view(1, R, 1)
    assert _window_us(large, W) < 1.3 * _window_us(small, W)


def _floats_apart(R, M, T, scale, seed):
    """Values that scatter over some twenty neighbouring floats."""
    z = torch.randn(T, R, M, generator=torch.Generator().manual_seed(seed))
    step = float(np.spacing(np.float32(abs(scale))))
    return torch.full((T, R, M), scale, dtype=torch.float32) + (step * torch.round(5.0 * z)).float()


@pytest.mark.parametrize("W,R", [(1000, 1024), (1500, 512)])
def test_windows_of_few_steps_between_floats(W, R):
    """... about two million cost hardly more than a scatter of 3 % about one (1.4; 9 to 14 where every range misses)."""
    near = _floats_apart(R, 8, 2 * W, 2.0e6, W).cuda()
    wide = (1.0 + 0.03 * torch.randn(2 * W, R, 8, generator=torch.Generator().manual_seed(W))).cuda()
    assert _window_us(near, W) < 3.0 * _window_us(wide, W)


@pytest.mark.parametrize("W,scale", [(60, 2.0e6), (200, 2.0e6), (1000, -7.0e-12), (1500, 3.0e30), (300, 3.4e38), (300, 1.0e-38)])
def test_medians_of_few_steps_between_floats(W, scale):
    from paper_2605_17879_b200 import guard
    R, M, B = 40, 4, W // 2
    X = _floats_apart(R, M, 4 * W, scale, W)
    dirs = [1, 1, -1, 1]
    g = guard.Guard(R, M, W, W // 2, dir=dirs, capacity=W + B, min_signals=1)
    g.set_sliding(False)
    o = go.Oracle(R, M, W, W // 2, 0, dir=dirs, min_signals=1)
    Xd, Xh = X.cuda(), X.numpy()
    for t in range(0, 4 * W, B):
        g.ingest(Xd[t:t + B])
        o.ingest(Xh[t:t + B])
        assert_bit_equal(to_np(g.score()["wmed"]), o.score()["wmed"], "t=%d" % t)
    assert g.sync_status() == 0
    g.close()


def _step_us(X, W):
    """Time of a step with its evaluation, windows sliding on from a full one."""
    from paper_2605_17879_b200 import guard
    T, R, M = X.shape
    g = guard.Guard(R, M, W, W // 2, dir=[1] * M, capacity=W + 16, min_signals=1)
    out = g.alloc_outputs()
    g.ingest(X[:W])
    g.score(out)
    us, per = [], (T - W) // 6
    for i in range(6):
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for t in range(W + i * per, W + (i + 1) * per):
            g.ingest(X[t:t + 1])
            g.score(out)
        b.record()
        torch.cuda.synchronize()
        us.append(a.elapsed_time(b) * 1000.0 / per)
    assert g.sync_status() == 0
    g.close()
    return float(np.median(us))


@pytest.mark.parametrize("R,M,W,constant", [(256, 8, 100, 8), (512, 8, 200, 8), (2048, 8, 200, 2)])
def test_steps_of_constant_series(R, M, W, constant):
    """Series that keep no list are rebuilt in every evaluation: by the whole chip (1.2, 1.6 and 1.6 times a step of continuous
    values), not by the few CTAs that a small fleet has at 128 series each (5.9, 8.6 and 2.7)."""
    X = (1.0 + 0.03 * torch.randn(W + 120, R, M, generator=torch.Generator().manual_seed(R))).cuda()
    C = X.clone()
    C[:, :, M - constant:] = C[:1, :, M - constant:]
    assert _step_us(C, W) < 2.2 * _step_us(X, W)


def _sweep_us(G, N, M):
    from paper_2605_17879_b200 import guard
    S = (1.0 + 0.01 * torch.randn(3, G, N, M, generator=torch.Generator().manual_seed(G + N + M))).cuda()
    ws = torch.empty(int(guard.lib().guard_sweep_workspace_bytes(G, N, M)), dtype=torch.uint8, device="cuda")
    out = guard.sweep_qualify(S[0], G, 1, dir=[1] * M, workspace=ws)
    us = []
    for _ in range(6):
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for i in range(30):
            guard.sweep_qualify(S[i % 3], G, 1, dir=[1] * M, workspace=ws, out=out)
        b.record()
        torch.cuda.synchronize()
        us.append(a.elapsed_time(b) * 1000.0 / 30)
    assert int(out["status"].cpu()[0]) == 0
    return float(np.median(us))


@pytest.mark.parametrize("G,N", [(4096, 33), (16384, 64)])
def test_sweeps_of_fewer_metrics(G, N):
    """Fewer metrics are fewer values: one takes 0.8 and 0.95 of the time of four (2.2 and 2.9 where all lanes of a warp share the
    scan of its bins), two 0.9 and 1.35 (1.6 and 1.95)."""
    four = _sweep_us(G, N, 4)
    assert _sweep_us(G, N, 1) < 1.4 * four
    assert _sweep_us(G, N, 2) < (1.25 if G == 4096 else 1.6) * four
