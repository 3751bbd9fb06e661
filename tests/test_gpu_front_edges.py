"""The front-end kernels at odd sizes, unaligned pointers and the ends of their ranges."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import speckle_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    return torch


def _plan(W, H, F):
    from paper_1701_00581_gb300 import Channel, Plan
    return Plan(Channel(W=W, H=H, N=64, R=4, max_frames=F))


def _unaligned(torch, a, shift):
    """The array on the GPU, `shift` elements past an aligned address."""
    t = torch.from_numpy(a)
    buf = torch.empty(a.size + shift, dtype=t.dtype, device="cuda:0")
    v = buf[shift:].view(a.shape)
    v.copy_(t.to("cuda:0"))
    return v


@pytest.mark.parametrize("W,H,F", [(64, 64, 1), (65, 67, 5), (130, 66, 9), (1, 3, 2), (256, 128, 300)])
@pytest.mark.parametrize("u16", [True, False])
@pytest.mark.parametrize("shift", [0, 1, 2])
def test_calibrate_and_shift(torch, W, H, F, u16, shift):
    """The same bits as the formula in FP32 (one subtraction, one division), and copies of samples."""
    rng = np.random.default_rng(W * 1000 + H + F)
    raw = rng.integers(0, 4096, (F, H, W)).astype(np.uint16 if u16 else np.float32)
    dark = (90 + 20 * rng.random((H, W))).astype(np.float32)
    gain = np.where(rng.random((H, W)) < 0.05, 0, 0.5 + rng.random((H, W))).astype(np.float32)
    sh = rng.integers(-40, 41, (F, 2)).astype(np.int32)
    plan = _plan(W, H, F)
    d_raw = _unaligned(torch, raw, shift)
    out = _unaligned(torch, np.zeros((F, H, W), np.float32), shift)
    plan.stage_calibrate(d_raw, F, torch.from_numpy(dark).cuda(), torch.from_numpy(gain).cuda(), out)
    want = np.where(gain > 0, (raw.astype(np.float32) - dark) / np.where(gain > 0, gain, 1), 0).astype(np.float32)
    assert np.array_equal(out.cpu().numpy(), want)
    moved = _unaligned(torch, np.zeros((F, H, W), np.float32), shift)
    plan.stage_shift(d_raw, F, torch.from_numpy(sh).cuda(), moved)
    assert np.array_equal(moved.cpu().numpy(), O.apply_shifts(raw, sh).astype(np.float32))


# windows below, at and past the chunk (32) and the staged tile (256 columns, 16 rows a share), every number of
# shift groups, one shift alone
@pytest.mark.parametrize("G,S", [(1, 0), (5, 3), (32, 5), (33, 6), (100, 11), (128, 12), (257, 18), (300, 31)])
@pytest.mark.parametrize("u16", [True, False])
def test_tracking(torch, G, S, u16):
    """The surface against FP64: each 32-sample chunk rounds at most 32 times, so every value is within
    33 * 2^-24 of the sum of its products' magnitudes (the reference window's rounding to FP32 adds as much again);
    the shift is the first maximum of the surface the call returned."""
    rng = np.random.default_rng(G * 100 + S)
    F, W, H = 3, G + 2 * S + 7, G + 2 * S + 4
    frames = rng.integers(0, 4096, (F, H, W)).astype(np.uint16 if u16 else np.float32)
    plan = _plan(W, H, F)
    rw = torch.empty((G, G), dtype=torch.float32, device="cuda:0")
    cc = torch.empty((F, 2 * S + 1, 2 * S + 1), dtype=torch.float64, device="cuda:0")
    sh = torch.empty((F, 2), dtype=torch.int32, device="cuda:0")
    plan.stage_track(torch.from_numpy(frames).cuda(), F, 1, G, S, rw, cc, sh)
    got, a = cc.cpu().numpy(), frames.astype(np.float64)
    x0, y0 = (W - G) // 2, (H - G) // 2
    r = a[1, y0:y0 + G, x0:x0 + G]
    r = r - r.mean()
    for f in range(F):
        for j in range(2 * S + 1):
            for i in range(2 * S + 1):
                t = a[f, y0 + j - S:y0 + j - S + G, x0 + i - S:x0 + i - S + G]
                assert abs(got[f, j, i] - (t * r).sum()) <= 67 * 2.0 ** -24 * (np.abs(t) * (np.abs(r) + 4096)).sum()
        k = int(np.argmax(got[f]))
        assert sh[f].tolist() == [k % (2 * S + 1) - S, k // (2 * S + 1) - S]


def test_tracking_of_special_values(torch):
    """An infinite sample makes every sum that holds it infinite and the first +inf wins; NaN is never picked,
    unless it comes first."""
    G, S, W, H = 40, 4, 64, 64
    rng = np.random.default_rng(7)
    frames = rng.random((4, H, W)).astype(np.float32)
    x0 = y0 = 12
    frames[0, y0 + 5, x0 + 5] += 2.0                      # every shift moves it within the window of the frames below
    frames[1, y0 - S + 44, x0 - S + 44] = np.inf          # in the window of a few shifts
    frames[2, y0 - S + 44, x0 - S + 44] = np.nan
    frames[3, y0 - S, x0 - S] = np.nan                    # in the window of the first shift alone
    rw = torch.empty((G, G), dtype=torch.float32, device="cuda:0")
    n = 2 * S + 1
    cc = torch.empty((4, n, n), dtype=torch.float64, device="cuda:0")
    sh = torch.empty((4, 2), dtype=torch.int32, device="cuda:0")
    _plan(W, H, 4).stage_track(torch.from_numpy(frames).cuda(), 4, 0, G, S, rw, cc, sh)
    got = cc.cpu().numpy()
    assert np.isfinite(got[0]).all()
    r = rw.cpu().numpy().astype(np.float64)
    for f in (1, 2, 3):
        a = frames[f].astype(np.float64)
        for j in range(n):
            for i in range(n):
                t = a[y0 + j - S:y0 + j - S + G, x0 + i - S:x0 + i - S + G]
                want = (t * r).sum()
                assert np.isnan(got[f, j, i]) == np.isnan(want) and np.isposinf(got[f, j, i]) == np.isposinf(want)
                assert np.isneginf(got[f, j, i]) == np.isneginf(want)
        best = 0
        for k in range(1, n * n):
            if got[f].flat[k] > got[f].flat[best]:
                best = k
        assert sh[f].tolist() == [best % n - S, best // n - S]
