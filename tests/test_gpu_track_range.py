"""Tracking sums past the range of a float."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# two row shares and one; a thread's 32-sample chunks stay below 2^128 (32 x 4096^2 x 2^98 = 2^127) while its 150 and
# 380 chunks of the reference frame at zero shift (about 32 x 1180^2 each) do not
@pytest.mark.parametrize("G,S", [(257, 18), (300, 31)])
def test_sum_past_float_range(G, S):
    """Counts times 2^49, a scale that rounds nothing: the FP64 surface within 67 * 2^-24 of the sum of the products'
    magnitudes (33 for a chunk's roundings, as much for the reference window's rounding, one to spare)."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    from paper_1701_00581_gb300 import Channel, Plan
    rng = np.random.default_rng(G)
    F, W, H, n = 2, G + 2 * S, G + 2 * S + 1, 2 * S + 1
    a = rng.integers(0, 4096, (F, H, W)).astype(np.float64)
    plan = Plan(Channel(W=W, H=H, N=64, R=4, max_frames=F))
    rw = torch.empty((G, G), dtype=torch.float32, device="cuda:0")
    cc = torch.empty((F, n, n), dtype=torch.float64, device="cuda:0")
    sh = torch.empty((F, 2), dtype=torch.int32, device="cuda:0")
    plan.stage_track(torch.from_numpy((a * 2.0 ** 49).astype(np.float32)).cuda(), F, 1, G, S, rw, cc, sh)
    got = cc.cpu().numpy() * 2.0 ** -98
    x0, y0 = (W - G) // 2, (H - G) // 2
    r = a[1, y0:y0 + G, x0:x0 + G]
    r = r - r.mean()
    assert (r * r).sum() / (8 * 2) * 2.0 ** 98 > np.finfo(np.float32).max        # a CTA's share, halved between two threads
    for f in range(F):
        for j in range(n):
            for i in range(n):
                t = a[f, y0 + j - S:y0 + j - S + G, x0 + i - S:x0 + i - S + G]
                assert abs(got[f, j, i] - (t * r).sum()) <= 67 * 2.0 ** -24 * (np.abs(t) * (np.abs(r) + 4096)).sum()
    assert sh[1].tolist() == [0, 0]


def test_time_of_a_burst_that_overflows():
    """Frames whose every sum overflows, and frames of NaNs, take the FP64 sums in every thread: the first from memory,
    two loads for six products, the second no further than a chunk.  Both take less than twelve times the time of a
    finite burst, which has two staged 16-byte loads for 48 products (one shift a thread at a time took fifty)."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    from paper_1701_00581_gb300 import Channel, Plan
    F, side, G, S = 100, 512, 256, 16
    plan = Plan(Channel(W=side, H=side, N=64, R=4, max_frames=F))
    rw = torch.empty((G, G), dtype=torch.float32, device="cuda:0")
    cc = torch.empty((F, 2 * S + 1, 2 * S + 1), dtype=torch.float64, device="cuda:0")
    sh = torch.empty((F, 2), dtype=torch.int32, device="cuda:0")
    steps = torch.arange(side, device="cuda:0").remainder(2).float()          # columns of 0 and 1: chunks of 16 r
    ms = {}
    for name, scale in (("finite", 1.0), ("overflow", 2.5e18), ("nan", float("nan"))):
        frames = (scale * steps).expand(F, side, side).contiguous()
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        t = []
        for _ in range(4):
            a.record()
            plan.stage_track(frames, F, 0, G, S, rw, cc, sh)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        ms[name] = min(t[1:])
        assert bool(torch.isnan(cc).all()) if name == "nan" else bool(torch.isfinite(cc).all())
    print(ms)
    assert max(ms["overflow"], ms["nan"]) < 12 * ms["finite"], ms
