"""Subfield spectra at the edges of the transform kernels: both thread layouts of 64 x 64 tiles, cutoffs from two
columns to the last one that a size admits, ragged and narrow tiles, both sample types."""
from __future__ import annotations

import math

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


@pytest.mark.parametrize("u16", [False, True])
@pytest.mark.parametrize("side", ["few", "many"])
@pytest.mark.parametrize("N,fc", [(64, 0.04), (64, 0.2885), (64, 0.499), (128, 0.02), (128, 0.2885), (128, 0.499),
                                  (256, 0.01), (256, 0.1), (256, 0.2945)])
def test_spectra_edges(torch, N, fc, side, u16):
    """Against the FP64 transform.  In units of the windowed flux the samples' magnitudes add up to 1, so each of the
    2 log2(N) butterfly levels adds at most 6 roundings of 2^-24 (root, product and sum of both components) and the
    window, the unpacking of the row pairs, the mean's removal and the normalisation 16 more."""
    from paper_1701_00581_gb300 import Channel, Plan
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    W, H = N + N // 2 + 1, N - 3
    n = len(O.subfield_grid(W, H, N, N // 2))
    F = 3 if side == "few" else 3 * sms // n + 1       # the layouts of N = 64 meet at three tiles per multiprocessor
    if side == "many" and N > 64:
        F = 2 * sms // n + 1                           # more than one wave of the larger sizes
    plan = Plan(Channel(W=W, H=H, N=N, R=2, fc=fc, max_frames=F))
    rng = np.random.default_rng([N, int(1000 * fc), F])
    fr = rng.integers(0, 4096, (F, H, W)).astype(np.uint16 if u16 else np.float32)
    ws, lay = plan.workspace(F, n)
    t = torch.from_numpy(fr.view(np.int16) if u16 else fr).cuda()
    plan.stage_spectra(t.view(torch.uint16) if u16 else t, F, 0, n, ws, lay)
    v = plan.views(ws, lay, F, n)
    K = plan.info["K"]
    iy, ix = CS.box_to_grid_index(N, K, 2)
    pick = sorted({0, 1, F - 1})
    tol = (12 * math.log2(N) + 16) * 2.0 ** -24
    for s, sub in enumerate(plan.subfields()):
        In, flux, mu = O.frame_spectra(fr[pick], tuple(int(e) for e in sub), N, N // 8)
        got = v["spec"][s].cpu().numpy()[pick][:, :, :2 * K + 1]
        assert np.abs(got - In[:, iy][:, :, ix]).max() <= tol
        assert np.abs(v["flux"][s].cpu().numpy()[pick] / flux - 1).max() <= 1e-6
        assert np.abs(v["mu"][s].cpu().numpy()[pick] / mu - 1).max() <= 1e-6
