"""A cube without a usable annulus: the largest candidate, and no candidate is evaluated for it."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import speckle_oracle as O
from tests import _cases as CS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [64, 128])
def test_no_usable_annulus(N):
    """64 exactly (an ordinary curve: the FP64 fit of the same statistics, which evaluates the same costs to 1e-15), and
    in less time than the fit of the ordinary curve takes (the best of five groups of 40)."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    from paper_1701_00581_gb300 import Channel, Plan
    F = 20
    plan = Plan(Channel(W=N, H=N, N=N, R=4, max_frames=F))
    ws, lay = plan.workspace(F, 1)
    v = plan.views(ws, lay, F, 1)
    K = plan.info["K"]
    ky, kx = np.mgrid[0:K + 1, -K:K + 1]
    rho = np.minimum(np.hypot(kx, ky) / (CS.FC * N), 0.999999)
    v["P"].fill_(1.0)
    v["noise"].fill_(0.0)
    ms = {}
    for name, ratio in (("curve", O.ratio_model(rho, 9.0)), ("none", 0.0 * rho)):
        v["M"].zero_()
        M = np.sqrt((ratio * (F - 1) + 1) / F).astype(np.complex64)
        v["M"][:, :, :2 * K + 1] = torch.from_numpy(M).cuda()
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        plan.stage_seeing(F, 0, 1, ws, lay)
        t = []
        for _ in range(5):
            torch.cuda.synchronize()
            a.record()
            for _ in range(40):
                plan.stage_seeing(F, 0, 1, ws, lay)
            b.record()
            b.synchronize()
            t.append(a.elapsed_time(b))
        ms[name] = min(t)
        Pf, Mf, c = np.ones((N, N)), np.zeros((N, N), dtype=np.complex128), N // 2
        Mf[c:c + K + 1, c - K:c + K + 1] = M
        want = O.fit_d_over_r0(*O.spectral_ratio(Pf, Mf, 0.0, F, N, CS.FC), N, CS.FC)
        got = float(v["seeing"][0])
        assert got == want == 64.0 if name == "none" else abs(got - want) <= 1e-9 * want
    assert ms["none"] < ms["curve"], ms
