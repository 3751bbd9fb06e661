"""The seeing fit with Korff constants so small that the model falls from 1 to 0 where an FP32 exponential is denormal."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import speckle_oracle as O
from tests import _cases as CS

pytestmark = pytest.mark.gpu


def _second_best(x, ck, N):
    """The lowest cost of another candidate for the model's own curve at x."""
    r = CS.FC * N
    rho = np.arange(1, int(np.ceil(r))) / r
    m = O.ratio_model(rho, x, ck)
    stop = int(np.argmax(~(m >= 0.05))) if not (m >= 0.05).all() else len(m)
    J = [np.sum((m[:stop] - O.ratio_model(rho[:stop], np.exp(np.log(64.0) * i / 255), ck)) ** 2) for i in range(256)]
    return np.partition(J, 1)[1]


@pytest.mark.parametrize("ck", [1e-29, 1e-36, 1e-40, 1e-42, 1e-44])
def test_fit(ck):
    """The model's own curve at every second candidate: the FP64 fit of the same P and M, where no other candidate
    costs less than 1e-3 (at small D/r0 the model is 1 at every annulus, whatever the candidate).  A cost is the same
    to 1e-12 in both evaluations, so the refined minima agree to 1e-9."""
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    from paper_1701_00581_gb300 import Channel, Plan
    N, F = 256, 20
    x = np.exp(np.log(64.0) * np.arange(1, 256, 2) / 255)
    n = len(x)
    plan = Plan(Channel(W=N * n, H=N, N=N, R=4, stride=N, max_frames=F, ck=ck))
    assert plan.info["n_sub"] == plan.info["n_cubes"] == n
    ws, lay = plan.workspace(F, n)
    v = plan.views(ws, lay, F, n)
    K, r, c = plan.info["K"], CS.FC * N, N // 2
    ky, kx = np.mgrid[0:K + 1, -K:K + 1]
    rho = np.minimum(O.annulus_index(kx, ky) / r, 0.999999)
    v["P"].fill_(1.0)
    v["M"].zero_()
    v["noise"].fill_(0.0)
    M = np.zeros((n, K + 1, 2 * K + 1), np.complex64)
    for i in range(n):
        M[i] = np.sqrt((O.ratio_model(rho, x[i], ck) * (F - 1) + 1) / F)
    v["M"][:, :, :2 * K + 1] = torch.from_numpy(M).cuda()
    plan.stage_seeing(F, 0, n, ws, lay)
    got = v["seeing"].cpu().numpy()[:n]
    Pf, Mf = np.ones((N, N)), np.zeros((N, N), dtype=np.complex128)
    fitted = 0
    for i in range(n):
        if _second_best(x[i], ck, N) < 1e-3:
            continue
        fitted += 1
        Mf[c:c + K + 1, c - K:c + K + 1] = M[i]
        num, den = O.spectral_ratio(Pf, Mf, 0.0, F, N, CS.FC)
        want = O.fit_d_over_r0(num, den, N, CS.FC, ck)
        assert abs(got[i] - want) <= 1e-9 * want, (i, x[i], got[i], want)
    assert fitted >= 40
