"""The modulus at powers and transfer functions near the ends of a float's range."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import speckle_oracle as O
from tests import _cases as CS

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lo,hi", [(-45, -27), (-31, -29), (25, 38.5)])
@pytest.mark.parametrize("big_stf", [False, True])
def test_modulus_range(lo, hi, big_stf):
    """A against the FP64 formula rounded to FP32: one unit in the last place at most, for a halfway case of the 46-bit
    path; rounded as the formula otherwise, so all but a few in a thousand are equal.  An infinite power over an
    infinite transfer function is NaN, over a finite one infinite."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    from paper_1701_00581_gb300 import Channel, Plan
    N, nsub = 128, 3
    plan = Plan(Channel(W=512, H=512, N=N, R=4, max_frames=2))
    ws, lay = plan.workspace(2, nsub)
    v = plan.views(ws, lay, 2, nsub)
    K, c = plan.info["K"], N // 2
    rng = np.random.default_rng([lo + 100, int(big_stf)])
    P = (10.0 ** rng.uniform(lo, hi, tuple(v["P"].shape))).astype(np.float32)
    noise = (10.0 ** rng.uniform(lo, hi - 1, nsub)).astype(np.float32)
    stf = 10.0 ** (rng.uniform(60, 80, (N, N)) if big_stf else rng.uniform(-6, 0, (N, N)))
    P[:, 4, K + 3] = P[:, 5, K + 3] = np.inf
    stf[c + 4, c + 3] = np.inf
    stf[c + 6, c + 3] = np.nan
    v["P"].copy_(torch.from_numpy(P))
    v["noise"].copy_(torch.from_numpy(noise))
    plan.stage_amplitude(nsub, torch.from_numpy(stf).cuda(), ws, lay)
    got = v["A"].cpu().numpy()[:, :, :2 * K + 1]
    t0 = O.otf_t0(N, CS.FC)[c:c + K + 1, c - K:c + K + 1]
    s = np.fmax(stf[c:c + K + 1, c - K:c + K + 1], 1e-4)
    with np.errstate(invalid="ignore"):
        want = np.sqrt(np.fmax(P[:, :, :2 * K + 1].astype(np.float64) - noise[:, None, None], 0) / s) * t0
    want[:, t0 <= 0] = 0
    want[:, 0, K] = 1
    want = want.astype(np.float32)
    assert np.array_equal(np.isinf(got), np.isinf(want)) and np.array_equal(np.isnan(got), np.isnan(want))
    m = np.isfinite(want)
    assert (np.abs(got[m] - want[m]) <= np.spacing(want[m])).all()
    assert np.mean(got[m] == want[m]) > 0.995
