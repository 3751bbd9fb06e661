"""The bispectrum's packed tasks: every used pair is computed and stored, once or in both orders, at odd radii,
even and odd cutoffs, radii up to the cutoff and frame counts off the stages of four."""
from __future__ import annotations

import numpy as np
import pytest

from oracle import speckle_oracle as O
from synth import burst as S
from tests import _cases as CS

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("no CUDA device")
    return torch


@pytest.mark.parametrize("N,R,fc,F", [(64, 1, 0.2885, 1), (64, 8, 0.2885, 5), (64, 7, 0.25, 4), (64, 18, 0.2885, 3),
                                      (64, 3, 0.05, 2), (128, 9, 0.27, 7), (128, 36, 0.2885, 2), (256, 24, 0.2885, 3),
                                      (256, 5, 0.2, 6)])
@pytest.mark.parametrize("mode", ["fp32", "kahan", "fp16", "bf16"])
def test_every_pair(torch, N, R, fc, F, mode):
    """Against the FP64 sum over the GPU's own spectra.  Per component a frame's triple product rounds at most 5
    times and its sum twice a frame: an error below (2 F + 10) 2^-24 of the mean product magnitude, for the complex
    value twice that.  The workspace starts as NaN, so an unwritten pair shows; both orders of a pair hold the same
    bits."""
    from paper_1701_00581_gb300 import (SM_ACC_KAHAN, SM_ACC_PLAIN, SM_BF16, SM_FP16, SM_FP32, Channel, Plan)
    plan = Plan(Channel(W=N, H=N, N=N, R=R, fc=fc, max_frames=F,
                        spectra_prec={"fp16": SM_FP16, "bf16": SM_BF16}.get(mode, SM_FP32),
                        acc_mode=SM_ACC_KAHAN if mode == "kahan" else SM_ACC_PLAIN))
    spec = S.BurstSpec(W=N, H=N, F=F, N=N, dr0=(4.0, 8.0), counts=True, fc=max(fc, 0.1))
    frames = torch.from_numpy(S.make_burst(spec, channel=70, burst=R)["frames"]).to("cuda:0")
    ws, lay = plan.workspace(F, 1)
    ws.fill_(0xff)
    plan.stage_spectra(frames, F, 0, 1, ws, lay)
    plan.stage_bispectrum(F, 1, ws, lay)
    torch.cuda.synchronize()
    v = plan.views(ws, lay, F, 1)
    K, c = plan.info["K"], N // 2
    sp = v["spec"][0]
    if mode in ("fp16", "bf16"):
        sp = torch.view_as_complex(sp.float().contiguous()) * (1.0 / 16384.0 if mode == "fp16" else 1.0)
    sp = sp.cpu().numpy().astype(np.complex128)[:, :, :2 * K + 1]
    wv = CS.used_pairs(N, R, fc).astype(np.int64)
    wx, wy, vx, vy = wv.T
    ux, uy = wx - vx, wy - vy

    def at(x, y):
        return (y + R) * (2 * K + 1) + x + K
    flat = sp.reshape(F, -1)
    want, size = np.zeros(len(wv), np.complex128), np.zeros(len(wv))
    for f in range(F):
        t = flat[f][at(ux, uy)] * flat[f][at(vx, vy)] * np.conj(flat[f][at(wx, wy)])
        want += t / F
        size += np.abs(t) / F
    idx = plan.pair_index(wv)
    B = v["B"][0].cpu().numpy()
    got = B[idx]
    assert np.isfinite(got.view(np.float32)).all()
    assert (np.abs(got - want) <= 2 * (2 * F + 10) * 2.0 ** -24 * size + 1e-37).all()
    both = ux * ux + uy * uy <= R * R
    if both.any():
        other = plan.pair_index(np.stack([wx, wy, ux, uy], 1)[both])
        assert np.array_equal(B[idx[both]], B[other])
