"""The bispectrum's fixed costs: what a launch takes beside the products of its frames."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu


def _ms(F, stage="bispectrum", reps=40, graph=False, **kw):
    """Time of `reps` launches, the best of five groups; with `graph` replayed from a CUDA graph, without the host."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    from paper_1701_00581_gb300 import Channel, Plan
    plan = Plan(Channel(max_frames=F, **kw))
    n = plan.info["n_sub"]
    ws, lay = plan.workspace(F, n)
    ws.zero_()
    s = torch.cuda.Stream()
    one = getattr(plan, "stage_" + stage)

    def run():
        for _ in range(reps):
            one(F, n, ws, lay, s)
    with torch.cuda.stream(s):
        run()
        torch.cuda.synchronize()
        if graph:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                run()
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        t = []
        for _ in range(6):
            torch.cuda.synchronize()
            a.record(s)
            g.replay() if graph else run()
            b.record(s)
            b.synchronize()
            t.append(a.elapsed_time(b))
    return min(t[1:])


def test_one_frame_is_a_few_latencies():
    """One frame of one 64^2 subfield is a chain of memory latencies, as the statistics of one frame are: less than
    twice their time (2.3 times with a latency more for every pair stored in both orders)."""
    kw = dict(W=64, H=64, N=64, R=8, graph=True)
    assert _ms(1, **kw) < 2.0 * _ms(1, "stats", **kw)


def test_bfloat16_costs_what_half_does():
    """The two storage types differ in their conversion alone, a shift against an instruction."""
    from paper_1701_00581_gb300 import SM_ACC_KAHAN, SM_BF16, SM_FP16
    kw = dict(W=512, H=512, N=256, R=24, acc_mode=SM_ACC_KAHAN, reps=2)
    assert _ms(30, spectra_prec=SM_BF16, **kw) < 1.02 * _ms(30, spectra_prec=SM_FP16, **kw)


@pytest.mark.parametrize("prec", [0, 1])
def test_last_stage_holds_its_frames_alone(prec):
    """Nine frames take as many stages as twelve (FP16: seven as nine), three; what the last one lacks is neither
    staged nor multiplied, so they take 9/12 (7/9) of the products' time."""
    kw = dict(W=512, H=512, N=128, R=16, spectra_prec=prec)
    few, all_ = (7, 9) if prec else (9, 12)
    assert _ms(few, **kw) < 0.93 * _ms(all_, **kw)


def test_compensated_sums_skip_an_empty_pass():
    """R = 1: every offset lies in a block's first four columns, so the compensated sums stream the frames once, as
    the plain ones do (twice: about twice the time)."""
    from paper_1701_00581_gb300 import SM_ACC_KAHAN
    kw = dict(W=512, H=512, N=128, R=1)
    assert _ms(100, acc_mode=SM_ACC_KAHAN, **kw) < 1.6 * _ms(100, **kw)
