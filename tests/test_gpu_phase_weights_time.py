"""The recursion's SNR weighting beside the unit weighting."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_snr_weights(prec):
    """A term's SNR weight is two products of three loaded powers where the unit weight is a root; both divide.  So it
    takes at most 1.3 times the unit weight's time (2.1, 1.4 and 1.6 times with a division for every index and its
    loads one after another).  225 subfields of 128^2, the best of three."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    from paper_1701_00581_gb300 import SM_W_SNR, SM_W_UNIT, Channel, Plan
    F, side = 2, 1024
    g = torch.Generator(device="cuda:0").manual_seed(3)
    frames = torch.randint(900, 3000, (F, side, side), generator=g, dtype=torch.int16, device="cuda:0").view(torch.uint16)
    ms = {}
    for weight in (SM_W_UNIT, SM_W_SNR):
        plan = Plan(Channel(W=side, H=side, N=128, R=16, max_frames=F, phase_prec=prec, phase_weight=weight))
        n = plan.info["n_sub"]
        ws, lay = plan.workspace(F, n)
        plan.stage_spectra(frames, F, 0, n, ws, lay)
        plan.stage_stats(F, n, ws, lay)
        plan.stage_bispectrum(F, n, ws, lay)
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        t = []
        for _ in range(4):
            a.record()
            plan.stage_phase(n, ws, lay)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        ms[weight] = min(t[1:])
    assert n == 225 and ms[SM_W_SNR] < 1.3 * ms[SM_W_UNIT], ms
