"""The seeing fit and the modulus at the ends of their ranges, on statistics written by the test."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import speckle_oracle as O
from tests import _cases as CS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    return torch


# D/r0 inside the candidates' range, at both ends and past them; exact model curves and perturbed ones (the fit then
# has several candidates in question); curves that stop at the first annulus
@pytest.mark.parametrize("N", [64, 256])
@pytest.mark.parametrize("x", [0.5, 1.0, 1.7, 5.0, 9.31, 30.0, 64.0, 200.0])
@pytest.mark.parametrize("spread", [0.0, 0.02, 0.3])
def test_seeing_fit(torch, N, x, spread):
    """Spectral ratios of a known D/r0 against the FP64 fit of the same P and M: both evaluate the same 256
    candidates in FP64 to rounding (1e-15 of J), and take the first minimum and the same parabola."""
    from paper_1701_00581_gb300 import Channel, Plan
    F = 20
    plan = Plan(Channel(W=N, H=N, N=N, R=4, max_frames=F))
    ws, lay = plan.workspace(F, 1)
    v = plan.views(ws, lay, F, 1)
    K, pitch, r, c = plan.info["K"], plan.info["box_pitch"], CS.FC * N, N // 2
    rng = np.random.default_rng([N, int(100 * x), int(100 * spread)])
    ky, kx = np.mgrid[0:K + 1, -K:K + 1]
    rho = np.minimum(np.hypot(kx, ky) / r, 0.999999)
    ratio = np.clip(O.ratio_model(rho, x) * (1 + spread * rng.standard_normal(rho.shape)), 0, None)
    P = (1.0 + rng.random(rho.shape)).astype(np.float32)
    M = np.sqrt((ratio * (F - 1) + 1) * P / F).astype(np.complex64)
    v["P"].zero_()
    v["M"].zero_()
    v["P"][0, :, :2 * K + 1] = torch.from_numpy(P).cuda()
    v["M"][0, :, :2 * K + 1] = torch.from_numpy(M).cuda()
    v["noise"].fill_(0.125)
    plan.stage_seeing(F, 0, 1, ws, lay)
    Pf, Mf = np.zeros((N, N)), np.zeros((N, N), dtype=np.complex128)
    Pf[c:c + K + 1, c - K:c + K + 1] = P
    Mf[c:c + K + 1, c - K:c + K + 1] = M
    num, den = O.spectral_ratio(Pf, Mf, 0.125, F, N, CS.FC)
    want = O.fit_d_over_r0(num, den, N, CS.FC)
    got = float(v["seeing"][0])
    assert abs(got - want) <= 1e-9 * want


@pytest.mark.parametrize("nsub", [1, 3, 49])
def test_modulus(torch, nsub):
    """A against the FP64 formula rounded to FP32: computed to about 46 bits before its one rounding, so at most one
    unit in the last place away (a halfway case); special values as the FP64 formula has them."""
    from paper_1701_00581_gb300 import Channel, Plan
    N = 128
    plan = Plan(Channel(W=512, H=512, N=N, R=4, max_frames=2))
    ws, lay = plan.workspace(2, nsub)
    v = plan.views(ws, lay, 2, nsub)
    K, c = plan.info["K"], N // 2
    rng = np.random.default_rng(nsub)
    P = (10.0 ** rng.uniform(-12, 0, tuple(v["P"].shape))).astype(np.float32)
    noise = (10.0 ** rng.uniform(-12, -3, nsub)).astype(np.float32)
    P[:, 3, K + 3] = np.nan
    P[:, 4, K + 3] = np.inf
    P[:, 5, K + 3] = noise
    P[:, 6, K + 3] = np.nextafter(noise, np.float32(1))
    stf = 10.0 ** rng.uniform(-6, 0, (N, N))
    v["P"].copy_(torch.from_numpy(P))
    v["noise"].copy_(torch.from_numpy(noise))
    plan.stage_amplitude(nsub, torch.from_numpy(stf).cuda(), ws, lay)
    got = v["A"].cpu().numpy()[:, :, :2 * K + 1]
    t0 = O.otf_t0(N, CS.FC)[c:c + K + 1, c - K:c + K + 1]
    s = np.maximum(stf[c:c + K + 1, c - K:c + K + 1], 1e-4)
    with np.errstate(invalid="ignore"):
        want = np.sqrt(np.fmax(P[:, :, :2 * K + 1].astype(np.float64) - noise[:, None, None], 0) / s) * t0
    want[:, t0 <= 0] = 0
    want[:, 0, K] = 1
    want = want.astype(np.float32)
    assert np.array_equal(np.isinf(got), np.isinf(want)) and not np.isnan(got).any()
    m = np.isfinite(want)
    assert (np.abs(got[m] - want[m]) <= np.spacing(want[m])).all()
    assert np.mean(got[m] == want[m]) > 0.999
