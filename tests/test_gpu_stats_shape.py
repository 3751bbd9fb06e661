"""The statistics stage's launch follows the subfield's size."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu


def test_many_small_subfields():
    """225 half boxes of 380 pairs are two CTAs' work each, one wave in all: ten frames of them take less than twice one
    subfield's time, which is the launch's own (the best of five groups of 40)."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    from paper_1701_00581_gb300 import Channel, Plan
    ms = []
    for side in (1, 8):
        plan = Plan(Channel(W=64 * side, H=64 * side, N=64, R=8, max_frames=10))
        n = plan.info["n_sub"]
        ws, lay = plan.workspace(10, n)
        ws.zero_()
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        t = []
        for _ in range(6):
            torch.cuda.synchronize()
            a.record()
            for _ in range(40):
                plan.stage_stats(10, n, ws, lay)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        ms.append(min(t[1:]))
    assert n == 225 and ms[1] < 2 * ms[0], ms
