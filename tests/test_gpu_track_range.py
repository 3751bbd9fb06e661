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
