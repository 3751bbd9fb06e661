"""The phase recursion's batches, units and clusters at the edges of their ranges."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import speckle_oracle as O
from synth import burst as S
from tests import _cases as CS
from tests.test_gpu_precision import _oracle_B_from_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    return torch


def _stages(torch, plan, F, seed):
    """Spectra, statistics and bispectrum of every subfield of one blob burst; the workspace and its views."""
    n = plan.info["n_sub"]
    spec = S.BurstSpec(W=plan.ch.W, H=plan.ch.H, F=F, N=plan.ch.N, dr0=(4.0, 6.0), counts=False)
    frames = torch.from_numpy(S.make_burst(spec, channel=60, burst=seed)["frames"]).to("cuda:0")
    ws, lay = plan.workspace(F, n)
    ws.zero_()
    plan.stage_spectra(frames, F, 0, n, ws, lay)
    plan.stage_stats(F, n, ws, lay)
    plan.stage_bispectrum(F, n, ws, lay)
    return ws, lay, plan.views(ws, lay, F, n)


# one offset ring, few late terms; offsets up to the cutoff, where v itself can be a late phasor; a radius whose
# rows do not fill their units; subfields where a batch has few points
@pytest.mark.parametrize("N,R", [(64, 1), (64, 3), (64, 18), (128, 5), (128, 20)])
@pytest.mark.parametrize("weight", ["bispec", "unit", "snr"])
def test_recursion_matches_the_oracle(torch, N, R, weight):
    """FP64 recursion on the GPU's own B, M and P against the oracle's: both sum the same terms in FP64 in another
    order, so they differ by rounding (1e-16 a term, at most a few thousand terms and rings) below 1e-9."""
    from paper_1701_00581_gb300 import (SM_PHASE_FP64, SM_W_BISPEC, SM_W_SNR, SM_W_UNIT, Channel, Plan)
    w = {"bispec": SM_W_BISPEC, "unit": SM_W_UNIT, "snr": SM_W_SNR}[weight]
    plan = Plan(Channel(W=N, H=N, N=N, R=R, max_frames=4, phase_prec=SM_PHASE_FP64, phase_weight=w))
    ws, lay, v = _stages(torch, plan, 4, 1)
    plan.stage_phase(1, ws, lay)
    torch.cuda.synchronize()
    K, c = plan.info["K"], N // 2
    B, pairs = _oracle_B_from_gpu(plan, v["B"][0].cpu().numpy(), N, R)
    full = {}
    for name in ("M", "P"):
        a = np.zeros((N, N), dtype=np.complex128)
        a[c:c + K + 1, c - K:c + K + 1] = v[name][0].cpu().numpy()[:, :2 * K + 1]
        a[1:, 1:] = np.where(a[1:, 1:] != 0, a[1:, 1:], np.conj(a[1:, 1:][::-1, ::-1]))      # the lower half plane
        full[name] = a
    zo = O.phase_recursion(B, pairs, full["M"], N, CS.FC, R, weight={"bispec": O.W_BISPEC, "unit": O.W_UNIT,
                                                                    "snr": O.W_SNR}[weight], P=full["P"].real)
    zo = zo[c:c + K + 1, c - K:c + K + 1]
    zg = v["z"][0].cpu().numpy()[:, :2 * K + 1]
    m = np.abs(zo) > 0
    assert np.abs(zg[m] - zo[m]).max() < 1e-9


@pytest.mark.parametrize("phase", ["fp32", "ff"])
def test_phasors_do_not_depend_on_the_cluster(torch, phase):
    """1, 2, 4 or 8 CTAs per subfield (the number follows from how many subfields the call has): the same bits."""
    from paper_1701_00581_gb300 import SM_PHASE_FF, SM_PHASE_FP32, Channel, Plan
    prec = {"fp32": SM_PHASE_FP32, "ff": SM_PHASE_FF}[phase]
    plan = Plan(Channel(W=897, H=897, N=128, R=16, max_frames=2, phase_prec=prec))
    n = plan.info["n_sub"]
    assert n > 152
    ws, lay, v = _stages(torch, plan, 2, 2)
    got = {}
    for k in (n, 100, 40, 20, 1):
        v["z"].zero_()
        plan.stage_phase(k, ws, lay)
        torch.cuda.synchronize()
        got[k] = v["z"].cpu().numpy().copy()
    for k, z in got.items():
        assert np.array_equal(z[:k], got[n][:k]), k
        assert not z[k:].any(), k


@pytest.mark.parametrize("N,R,prec", [(64, 8, 0), (128, 5, 1), (256, 3, 2)])
def test_phasors_are_written_whole(torch, N, R, prec):
    """Every value of z is written, zero outside the cutoff, whatever the workspace held."""
    from paper_1701_00581_gb300 import Channel, Plan
    plan = Plan(Channel(W=N, H=N, N=N, R=R, phase_prec=prec, max_frames=2))
    ws, lay = plan.workspace(2, 1)
    ws.view(torch.uint8).fill_(0xff)
    frames = torch.from_numpy(np.random.default_rng(N).random((2, N, N), dtype=np.float32) + 1).cuda()
    plan.stage_spectra(frames, 2, 0, 1, ws, lay)
    plan.stage_stats(2, 1, ws, lay)
    plan.stage_bispectrum(2, 1, ws, lay)
    plan.stage_phase(1, ws, lay)
    z = plan.views(ws, lay, 2, 1)["z"][0].cpu().numpy()
    K = plan.info["K"]
    ky, kx = np.mgrid[0:z.shape[0], -K:z.shape[1] - K]
    inside = kx ** 2 + ky ** 2 <= (0.2885 * N) ** 2
    assert np.isfinite(z.view(np.float64)).all()
    assert (z[~inside] == 0).all() and (np.abs(np.abs(z[inside]) - 1) <= 1e-6).all()
