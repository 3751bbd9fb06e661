"""What a user of the reconstruction library has it do, as measurable cases.

Every case goes from inputs a program holds (frames of a burst, a model STF,
a plan and its workspace, a batch or an engine) through one of the public
entry points to the arrays the program takes away.  Kinds:

* ``call``     one burst through ``Plan.reconstruct`` (device frames, caller's workspace);
* ``noalloc``  one burst through ``Plan.reconstruct_noalloc`` (fixed scratch);
* ``batch``    several bursts through ``Batch.reconstruct``;
* ``engine``   several bursts from pinned host memory through ``Engine.submit`` / ``poll``;
* ``front``    raw frames through calibration, correlation tracking and shifting.

Frames are synthetic: Gaussian blobs on a unit background, convolved with the
PSFs of Kolmogorov phase screens, with noise, as 12-bit counts or float32.
``exact`` restates the whole method in 64-bit torch.
"""
import functools
import math

import numpy as np
import torch

from paper_1701_00581_gb300 import Batch, Channel, Engine, Plan

FC = 0.2885           # optics cutoff of the TiO and H-alpha channels, cycles per pixel
CK = 0.435            # Korff constant of the model STF
BLOBS = (0.8, 1.4, 2.4, 4.0)   # widths of the scene's structures, px: down to the diffraction limit
NOISE = 0.005         # additive noise, fraction of the mean
PREC = {"fp32": 0, "fp16": 1, "bf16": 2}
ACC = {"plain": 0, "kahan": 1}
PHASE = {"fp32": 0, "fp64": 1, "ff": 2}
WEIGHT = {"bispec": 0, "unit": 1, "snr": 2}


def _case(name, kind, W, H, N, R, F, **kw):
    """A case with every option at its default unless given."""
    c = {"name": name, "kind": kind, "W": W, "H": H, "N": N, "R": R, "F": F, "stride": N // 2, "fc": FC,
         "u16": True, "stf": False, "prec": "fp32", "acc": "plain", "phase": "fp32", "weight": "bispec",
         "iters": 0, "central": False, "photon_gain": 0.0, "bursts": 1, "dr0_lo": 5.0, "dr0_hi": 12.0,
         "extra_N": 0}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one 64 x 64 subfield at known seeing; launches and latency count
        _case("subfield64", "call", 64, 64, 64, 8, 100, u16=False, stf=True, dr0_lo=6.0, dr0_hi=6.0),
        # many small bursts at once: eight single-subfield bursts in one batched launch
        _case("subfield64_batch8", "batch", 64, 64, 64, 8, 100, u16=False, bursts=8, dr0_lo=6.0, dr0_hi=6.0),
        # a control loop that may not allocate: short burst, odd ragged frame, fixed scratch
        _case("ragged_noalloc", "noalloc", 301, 227, 64, 8, 61, stf=True),
        # an ordinary H-alpha burst, seeing estimated from the burst
        _case("halpha1024", "call", 1024, 1024, 128, 16, 100),
        # serving: three H-alpha bursts from pinned host memory through the engine, two in flight
        _case("halpha_served", "engine", 1024, 1024, 128, 16, 100, bursts=3),
        # a full TiO (or G-band) burst: the largest ordinary call
        _case("tio2560", "call", 2560, 2160, 256, 24, 100),
        # a region of interest of a calibrated TiO burst: float32 frames, ragged edges, odd radius, short burst
        _case("tio_roi_ragged", "call", 901, 683, 256, 21, 63, u16=False),
        # the reduced-storage mode: half-precision spectra, compensated sums, float-float recursion
        _case("tio_fp16_kahan_ff", "call", 768, 512, 256, 24, 100, prec="fp16", acc="kahan", phase="ff"),
        # a batch of bursts of two channels (two of each) in one launch
        _case("mixed_batch", "batch", 768, 512, 256, 24, 100, bursts=4, extra_N=128),
        # the paper's layout: subfields every N / 4, central-block mosaic
        _case("paper_layout", "call", 1024, 768, 256, 24, 100, stride=64, central=True),
        # photon-bias removal, unit weights and least-squares sweeps after the recursion
        _case("refined", "call", 640, 479, 128, 16, 80, u16=False, weight="unit", iters=5, photon_gain=8000.0),
        # the front end of a raw TiO burst: flat/dark, correlation tracking, shifting
        _case("front_tio", "front", 2560, 2160, 256, 24, 100),
    ]


def draw(rng):
    """One more case of the same ranges: kinds, subfield sizes, frame sizes, radii, burst lengths, options."""
    kind = rng.choice(["call", "call", "call", "noalloc", "batch", "engine", "front"])

    def span(lo, hi):                                  # log-uniform, odd sizes among them
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "front":
        return _drawn("front", span(600, 2560), span(600, 2160), 256, 24, span(10, 100), rng.random() < 0.5)
    N = rng.choice([64, 128, 256])
    R = rng.randint(*{64: (4, 8), 128: (8, 16), 256: (14, 24)}[N])
    F = span(30, 100)
    stride = rng.choice([N // 2, N // 2, N // 2, N // 4])
    if kind == "noalloc":
        N, R, stride = 64, rng.randint(4, 8), 32
        W, H = span(64, 640), span(64, 640)
    elif kind == "call":
        W, H = span(N, min(2560, 12 * N)), span(N, min(2160, 10 * N))
    else:
        W, H = span(N, 5 * N), span(N, 5 * N)
    c = _drawn(kind, W, H, N, R, F, rng.random() < 0.7)
    c["stride"] = stride
    c["fc"] = rng.choice([FC, FC, round(rng.uniform(0.25, FC), 4)])
    c["stf"] = bool(rng.random() < 0.4)
    c["central"] = stride == N // 4 and rng.random() < 0.7
    if kind == "batch":
        c["bursts"] = rng.randint(2, 6)
        c["extra_N"] = rng.choice([0, 0, 64, 128])
    elif kind == "engine":
        c["bursts"] = rng.randint(1, 4)
    if kind in ("call", "batch", "engine"):
        c["prec"] = rng.choice(["fp32", "fp32", "fp32", "fp16", "bf16"])
    if kind == "call":
        c["acc"] = rng.choice(["plain", "plain", "plain", "kahan"])
        c["phase"] = rng.choice(["fp32", "fp32", "fp32", "ff"])
        c["weight"] = rng.choice(["bispec", "bispec", "unit"])
        c["iters"] = rng.choice([0, 0, 0, 3])
        c["photon_gain"] = rng.choice([0.0, 0.0, 4.0 if c["u16"] else 8000.0])   # about 8000 photons a pixel
    # no more subfields, and no more work, than a full TiO burst
    while len(_tiles(c["W"], c["H"], N, stride, c["central"])) * c["bursts"] * (N / 256.0) ** 2 > 304:
        c["W"], c["H"] = max(N, c["W"] * 3 // 4), max(N, c["H"] * 3 // 4)
    while work(c)["flops"] * (1.0 + 0.3 * c["iters"]) > 2.0e12:
        c["F"] = c["F"] * 3 // 4
    return c


def _drawn(kind, W, H, N, R, F, u16):
    c = _case("", kind, W, H, N, R, F, u16=u16)
    del c["name"]
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gauss(n, sigma, dev):
    x = torch.arange(n, device=dev, dtype=torch.float64)
    x = torch.minimum(x, n - x)
    return torch.exp(-0.5 * (x / sigma) ** 2)


def _scene(W, H, g, dev):
    """Unit background plus periodic Gaussian blobs, float64 [H, W]."""
    out = torch.ones((H, W), dtype=torch.float64, device=dev)
    for sigma in BLOBS:                                # ten blobs per 64 x 64 px of each width
        amp = 0.05 + 0.25 * torch.rand((H, W), generator=g, device=dev, dtype=torch.float64)
        pts = torch.where(torch.rand((H, W), generator=g, device=dev) < 10 / 64.0 ** 2, amp, torch.zeros_like(amp))
        k = torch.fft.rfft2(_gauss(H, sigma, dev)[:, None] * _gauss(W, sigma, dev)[None, :])
        out += torch.fft.irfft2(torch.fft.rfft2(pts) * k, s=(H, W))
    return out


def _psfs(N, fc, dr0, g, dev):
    """Short-exposure PSFs through Kolmogorov screens, one per D/r0: [F, N, N], origin at [0, 0]."""
    G, dp = 2 * N, fc * N
    f = torch.fft.fftfreq(G, d=1.0 / dp, device=dev, dtype=torch.float64)
    kap = torch.hypot(f[:, None], f[None, :])
    kap[0, 0] = math.inf
    c = (N - 1) / 2.0
    y = torch.arange(N, device=dev, dtype=torch.float64) - c
    pupil = ((y[:, None] ** 2 + y[None, :] ** 2) <= (dp / 2.0) ** 2).double()
    out = torch.empty((len(dr0), N, N), dtype=torch.float64, device=dev)
    for i, x in enumerate(dr0):
        amp = math.sqrt(0.023) * float(x) ** (5.0 / 6.0) * kap ** (-11.0 / 6.0) * (dp / G)
        z = torch.complex(torch.randn((G, G), generator=g, device=dev, dtype=torch.float64),
                          torch.randn((G, G), generator=g, device=dev, dtype=torch.float64))
        screen = (torch.fft.ifft2(z * amp) * (G * G)).real[:N, :N]
        p = torch.fft.fft2(pupil * torch.exp(1j * screen)).abs() ** 2
        out[i] = p / p.sum()
    return out


def _frames(case, seed, k=0, W=None, H=None, N=None):
    """Burst k of a case: (frames on the GPU [F, H, W] uint16 or float32, D/r0 per frame)."""
    W, H, N = W or case["W"], H or case["H"], N or case["N"]
    dev = "cuda"
    g = torch.Generator(device=dev).manual_seed(1000003 * int(seed) + 101 * k + 7)
    rng = np.random.default_rng([int(seed), k, 17])
    F = case["F"]
    dr0 = rng.uniform(case["dr0_lo"], case["dr0_hi"], F)
    scene = _scene(W, H, g, dev)
    scene *= (2000.0 if case["u16"] else 1.0) / scene.mean()
    sc = torch.fft.rfft2(scene)
    psf = _psfs(N, case["fc"], dr0, g, dev)
    off = torch.arange(N, device=dev)
    off = torch.where(off < N // 2, off, off - N)
    iy, ix = off.remainder(H), off.remainder(W)
    frames = torch.empty((F, H, W), dtype=torch.int16 if case["u16"] else torch.float32, device=dev)
    for f in range(F):
        big = torch.zeros((H, W), dtype=torch.float64, device=dev)
        big[iy[:, None], ix[None, :]] = psf[f]
        img = torch.fft.irfft2(sc * torch.fft.rfft2(big), s=(H, W))
        img += torch.randn((H, W), generator=g, device=dev) * (img.mean() * NOISE)
        frames[f] = img.round().clamp(0, 4095) if case["u16"] else img
    return (frames.view(torch.uint16) if case["u16"] else frames), dr0


def _t0(k2, r):
    rho = torch.sqrt(k2) / r
    p = rho.clamp(max=1.0)
    return torch.where(rho <= 1.0, (2 / math.pi) * (torch.acos(p) - p * torch.sqrt(1 - p * p)), torch.zeros_like(p))


def _model_stf(N, fc, dr0, dev="cuda"):
    """Model speckle transfer function [N, N], centred, averaged over the frames' D/r0."""
    k = torch.arange(-(N // 2), N - N // 2, device=dev, dtype=torch.float64)
    k2 = k[:, None] ** 2 + k[None, :] ** 2
    t0 = _t0(k2, fc * N)
    rho = torch.sqrt(k2) / (fc * N)
    acc = torch.zeros_like(t0)
    for d in dr0:
        acc += t0 * t0 * torch.exp(-6.88 * (rho * float(d)) ** (5.0 / 3.0)) + CK * t0 / float(d) ** 2
    acc /= len(dr0)
    return acc / acc[N // 2, N // 2]


def _channel(case, W=None, H=None, N=None, R=None):
    N = N or case["N"]
    return Channel(W=W or case["W"], H=H or case["H"], N=N, R=R or case["R"],
                   stride=case["stride"] * N // case["N"], fc=case["fc"],
                   spectra_prec=PREC[case["prec"]], phase_weight=WEIGHT[case["weight"]], ck=CK,
                   max_frames=case["F"], acc_mode=ACC[case["acc"]], phase_prec=PHASE[case["phase"]],
                   phase_iters=case["iters"], edge_mode=1 if case["central"] else 0,
                   mosaic_mode=1 if case["central"] else 0, photon_gain=case["photon_gain"])


def _estimable(W, H, N, stride):
    """Whether the seeing can be estimated: a full-size subfield on the N grid exists."""
    return N % stride == 0 and W >= N and H >= N


def _shapes(case):
    """(W, H, N, R) of each burst of a batch: the case's own and, every second one, the smaller channel's."""
    one = (case["W"], case["H"], case["N"], case["R"])
    n2 = case["extra_N"]
    if not n2 or n2 >= case["N"]:
        return [one] * case["bursts"]
    q = case["N"] // n2
    two = (max(n2, case["W"] // q + 1), max(n2, case["H"] // q + 1), n2, max(4, case["R"] * n2 // case["N"] + 2))
    return [one if i % 2 == 0 else two for i in range(case["bursts"])]


def _job(case, seed, k, shape, plan):
    """Buffers of one burst: frames, STF (or None), workspace, outputs."""
    W, H, N, _ = shape
    frames, dr0 = _frames(case, seed, k, W, H, N)
    stf = _model_stf(N, case["fc"], dr0) if case["stf"] or not _estimable(W, H, N, plan.ch.stride) or case["F"] < 2 \
        else None
    ws, lay = plan.workspace(case["F"], plan.info["n_sub"])
    return {"frames": frames, "stf": stf, "ws": ws, "lay": lay,
            "out": torch.empty((H, W), dtype=torch.float32, device="cuda"),
            "valid": torch.empty((H, W), dtype=torch.uint8, device="cuda")}


def prepare(case, seed):
    kind, F = case["kind"], case["F"]
    if kind == "call":
        plan = Plan(_channel(case))
        return {"kind": kind, "plan": plan, "F": F,
                "job": _job(case, seed, 0, (case["W"], case["H"], case["N"], case["R"]), plan)}
    if kind == "noalloc":
        plan = Plan(_channel(case))
        frames, dr0 = _frames(case, seed)
        return {"kind": kind, "plan": plan, "F": F, "frames": frames, "stf": _model_stf(case["N"], case["fc"], dr0),
                "out": torch.empty((case["H"], case["W"]), dtype=torch.float32, device="cuda"),
                "valid": torch.empty((case["H"], case["W"]), dtype=torch.uint8, device="cuda")}
    if kind == "batch":
        shapes, plans = _shapes(case), {}
        for s in shapes:
            if s not in plans:
                plans[s] = Plan(_channel(case, *s))
        jobs = [_job(case, seed, k, s, plans[s]) for k, s in enumerate(shapes)]
        batch = Batch([plans[s] for s in shapes], [F] * len(shapes), [0 if case["u16"] else 1] * len(shapes))
        return {"kind": kind, "plans": plans, "batch": batch, "jobs": jobs}
    if kind == "engine":
        ch = _channel(case)
        plan = Plan(ch)
        lay = plan.layout(F, plan.info["n_sub"])
        burst = F * case["W"] * case["H"] * (2 if case["u16"] else 4) + 32 * case["W"] * case["H"] + (8 << 20)
        eng = Engine([ch], hbm_budget_bytes=int(lay.bytes) + 2 * burst + (64 << 20), max_inflight=2)
        jobs = []
        for k in range(case["bursts"]):
            frames, dr0 = _frames(case, seed, k)
            host = torch.empty(frames.shape, dtype=frames.dtype, pin_memory=True)
            host.copy_(frames)
            given = case["stf"] or not _estimable(case["W"], case["H"], case["N"], case["stride"]) or F < 2
            jobs.append({"frames": host.numpy(), "dr0": dr0 if given else None, "pin": host,
                         "out": torch.empty((case["H"], case["W"]), dtype=torch.float32, pin_memory=True).numpy(),
                         "valid": torch.empty((case["H"], case["W"]), dtype=torch.uint8, pin_memory=True).numpy()})
        return {"kind": kind, "engine": eng, "jobs": jobs}
    # front: raw counts = gain * drifting frames + dark
    plan = Plan(_channel(case))
    W, H = case["W"], case["H"]
    frames, _ = _frames(dict(case, u16=True), seed)
    g = torch.Generator(device="cuda").manual_seed(77 + int(seed))
    rng = np.random.default_rng([int(seed), 5])
    dark = 90.0 + 20.0 * torch.rand((H, W), generator=g, device="cuda")
    flat = dark + 1500.0 * (0.9 + 0.2 * torch.rand((H, W), generator=g, device="cuda"))
    flat[torch.rand((H, W), generator=g, device="cuda") < 1e-4] = 0.0          # dead pixels
    resp = (flat - dark).clamp(min=0.0) / 1500.0
    raw = torch.empty_like(frames)
    src, dst = frames.view(torch.int16), raw.view(torch.int16)
    for f in range(F):
        sx, sy = (int(v) for v in rng.integers(-12, 13, 2))
        dst[f] = (torch.roll(src[f], (sy, sx), (0, 1)).float() * resp + dark).round().clamp(0, 4095)
    if not case["u16"]:
        raw = raw.view(torch.int16).float()
    gain = torch.empty((H, W), dtype=torch.float32, device="cuda")
    plan.stage_gain(flat, dark, gain)
    G, S = 256, 16
    return {"kind": "front", "plan": plan, "F": F, "raw": raw, "dark": dark, "flat": flat, "gain": gain, "G": G, "S": S,
            "frames": torch.empty((F, H, W), dtype=torch.float32, device="cuda"),
            "aligned": torch.empty((F, H, W), dtype=torch.float32, device="cuda"),
            "window": torch.empty((G, G), dtype=torch.float32, device="cuda"),
            "cc": torch.empty((F, 2 * S + 1, 2 * S + 1), dtype=torch.float64, device="cuda"),
            "shifts": torch.empty((F, 2), dtype=torch.int32, device="cuda")}


def run(s):
    kind = s["kind"]
    if kind == "call":
        j, plan = s["job"], s["plan"]
        plan.reconstruct(j["frames"], s["F"], j["stf"], plan.info["n_sub"], j["ws"], j["lay"], j["out"], j["valid"])
        return {"out": j["out"], "valid": j["valid"]}
    if kind == "noalloc":
        s["plan"].reconstruct_noalloc(s["frames"], s["F"], s["stf"], s["out"], s["valid"])
        return {"out": s["out"], "valid": s["valid"]}
    if kind == "batch":
        s["batch"].reconstruct(s["jobs"])
        return [{"out": j["out"], "valid": j["valid"]} for j in s["jobs"]]
    if kind == "engine":
        eng, flying = s["engine"], []
        for j in s["jobs"]:
            if len(flying) == 2:
                eng.poll(flying.pop(0))
            flying.append(eng.submit(0, j["frames"], j["out"], j["valid"], d_over_r0=j["dr0"]))
        for t in flying:
            eng.poll(t)
        return [{"out": j["out"], "valid": j["valid"]} for j in s["jobs"]]
    p, F = s["plan"], s["F"]
    p.stage_calibrate(s["raw"], F, s["dark"], s["gain"], s["frames"])
    p.stage_track(s["frames"], F, 0, s["G"], s["S"], s["window"], s["cc"], s["shifts"])
    p.stage_shift(s["frames"], F, s["shifts"], s["aligned"])
    return {"frames": s["frames"], "aligned": s["aligned"], "shifts": s["shifts"]}


# ---------------------------------------------------------------------------
# the work a pass cannot do without
# ---------------------------------------------------------------------------
@functools.lru_cache(maxsize=64)
def _pairs(N, fc, R):
    """Every (wx, wy, vx, vy) the recursion reads, w in rings of equal |w|^2, int16 [n, 4]."""
    r2 = math.floor((fc * N) ** 2)
    K = math.floor(fc * N)
    ky, kx = np.mgrid[0:K + 1, -K:K + 1]
    q = kx * kx + ky * ky
    m = ((ky > 0) | (kx > 0)) & (q >= 2) & (q <= r2)
    w = np.stack([kx[m], ky[m]], 1)
    w = w[np.argsort((w ** 2).sum(1), kind="stable")]
    vy, vx = np.mgrid[-R:R + 1, -R:R + 1]
    v2 = vx * vx + vy * vy
    m = (v2 > 0) & (v2 <= R * R)
    v = np.stack([vx[m], vy[m]], 1)
    out = []
    for a in range(0, len(w), 512):
        b = w[a:a + 512]
        w2 = (b ** 2).sum(1)[:, None]
        ok = ((v ** 2).sum(1)[None] < w2) & (((b[:, None] - v[None]) ** 2).sum(2) < w2)
        i, j = np.nonzero(ok)
        out.append(np.concatenate([b[i], v[j]], 1).astype(np.int16))
    return np.concatenate(out)


def _tiles(W, H, N, stride, drop):
    def starts(L):
        if drop:
            return [k * stride for k in range((L - N) // stride + 1)] if L >= N else []
        return [k * stride for k in range(1 if L <= N else math.ceil((L - N) / stride) + 1)]
    return [(x, y, min(N, W - x), min(N, H - y)) for y in starts(H) for x in starts(W)]


def work(case):
    """Frames in, mosaic (or aligned frames) out; the FLOPs of the transforms and of the used triple products."""
    F = case["F"]
    size = 2 if case["u16"] else 4
    px = case["W"] * case["H"]
    if case["kind"] == "front":
        side = 33
        return {"bytes": F * px * (size + 8) + 8 * px, "flops": 2.0 * F * (side * 256) ** 2 + 3.0 * F * px}
    total = {"bytes": 0.0, "flops": 0.0}
    for W, H, N, R in (_shapes(case) if case["kind"] == "batch" else
                       [(case["W"], case["H"], case["N"], case["R"])] * case["bursts"]):
        n = len(_tiles(W, H, N, case["stride"] * N // case["N"], case["central"]))
        K = math.floor(case["fc"] * N)
        fft = 5.0 * N * math.log2(N) * (N // 2 + K + 1)
        total["bytes"] += F * W * H * size + 5 * W * H
        total["flops"] += n * (F * (fft + 14.0 * len(_pairs(N, case["fc"], R))) + fft +
                               8.0 * (1 + 3 * case["iters"]) * len(_pairs(N, case["fc"], R)))
    return total


# ---------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------
def _tukey(L, taper, dev):
    x = torch.arange(L, device=dev, dtype=torch.float64)
    p = torch.minimum(x, L - 1 - x)
    return torch.where(p < taper, 0.5 * (1 - torch.cos(math.pi * (p + 0.5) / taper)), torch.ones_like(p))


def _fit_seeing(P, M, noise, F, N, fc):
    """D/r0 of one cube from the spectral ratio of its centred power P and mean spectrum M (numpy)."""
    r = fc * N
    c = N // 2
    k = np.arange(-c, N - c)
    kx, ky = np.meshgrid(k, k)
    q = kx * kx + ky * ky
    dom = ((ky > 0) | ((ky == 0) & (kx > 0))) & (q <= math.floor(r * r))
    b = np.rint(np.sqrt(q[dom])).astype(int)
    num = np.bincount(b, ((F * np.abs(M[dom]) ** 2 - P[dom]) / (F - 1)), minlength=2)
    den = np.bincount(b, P[dom] - noise, minlength=2)
    bins = []
    for i in range(1, len(num)):
        if not i < r or not den[i] > 0 or num[i] / den[i] < 0.05:
            break
        bins.append(i)
    if not bins:
        return 64.0
    bins = np.array(bins)
    rho = bins / r
    t0 = (2 / np.pi) * (np.arccos(rho) - rho * np.sqrt(1 - rho * rho))
    lx = math.log(64.0) * (np.arange(256) / 255)
    x = np.exp(lx)[:, None]
    e = np.exp(-6.88 * (rho * x) ** (5 / 3))
    model = t0 * t0 * e * (1 + CK / x ** 2) / (t0 * t0 * e + CK * t0 / x ** 2)
    J = ((num[bins] / den[bins] - model) ** 2).sum(1)
    i = int(np.argmin(J))
    t = lx[i]
    if 0 < i < 255:
        curv = J[i - 1] - 2 * J[i] + J[i + 1]
        if curv > 0:
            t += 0.5 * (lx[1] - lx[0]) * (J[i - 1] - J[i + 1]) / curv
    return math.exp(t)


def _exact_burst(case, frames, stf, W, H, N, R):
    """The mosaic of one burst in 64 bits, and None for the mask."""
    dev, F, fc = "cuda", case["F"], case["fc"]
    stride = case["stride"] * N // case["N"]
    r, c, taper = fc * N, N // 2, N // 8
    K = math.floor(r)
    tiles = _tiles(W, H, N, stride, case["central"])
    pairs = torch.from_numpy(_pairs(N, fc, R).astype(np.int64)).to(dev)
    wx, wy, vx, vy = pairs.T

    def at(x, y):
        return (y + c) * N + x + c
    iw, iv, iu = at(wx, wy), at(vx, vy), at(wx - vx, wy - vy)
    iwn, ivn, iun = at(-wx, -wy), at(-vx, -vy), at(vx - wx, vy - wy)
    first = torch.ones(len(iw), dtype=torch.bool, device=dev)
    first[1:] = iw[1:] != iw[:-1]
    point = torch.cumsum(first, 0) - 1                                   # pair -> point, points in ring order
    pw, pwn = iw[first], iwn[first]
    q = (wx * wx + wy * wy)[first].cpu().numpy()
    ring_p = [0] + (np.nonzero(np.diff(q))[0] + 1).tolist() + [len(q)]
    ends = torch.nonzero(first).flatten().cpu().numpy().tolist() + [len(iw)]
    k = torch.arange(-c, N - c, device=dev)
    k2 = (k[:, None] ** 2 + k[None, :] ** 2)
    t0 = _t0(k2.double(), r)
    corner = (k2 > r * r) & (k[:, None] >= 1) & (k[:, None] <= K) & (k[None, :].abs() <= K)
    wins = {}

    def window(w, h):
        if (w, h) not in wins:
            wins[w, h] = _tukey(h, taper, dev)[:, None] * _tukey(w, taper, dev)[None, :]
        return wins[w, h]

    def spectra(t):
        x, y, w, h = t
        win = window(w, h)
        raw = frames[:, y:y + h, x:x + w].double() if not case["u16"] else \
            frames[:, y:y + h, x:x + w].contiguous().view(torch.int16).double()
        mu = (raw * win).sum((1, 2)) / win.sum()
        flux = mu * win.sum()
        I = torch.fft.fftshift(torch.fft.fft2(win * (raw - mu[:, None, None]), s=(N, N)), dim=(1, 2))
        I /= flux[:, None, None]
        I[:, c, c] = 1.0
        return I, flux, mu

    if stf is None:
        xs = []
        for t in tiles:
            if t[0] % N == 0 and t[1] % N == 0 and t[2] == N and t[3] == N:
                I, _, _ = spectra(t)
                P, M = (I.abs() ** 2).mean(0), I.mean(0)
                xs.append(_fit_seeing(P.cpu().numpy(), M.cpu().numpy(), float(P[corner].mean()), F, N, fc))
        stf = _model_stf(N, fc, [1.0 / np.mean(1.0 / np.array(xs))])
    num = torch.zeros((H, W), dtype=torch.float64, device=dev)
    den = torch.zeros((H, W), dtype=torch.float64, device=dev)
    step = max(1, int(4e8 // len(iw)))
    for s0 in range(0, len(tiles), step):
        part = tiles[s0:s0 + step]
        n = len(part)
        B = torch.zeros((len(iw), n), dtype=torch.complex128, device=dev)
        z = torch.zeros((N * N, n), dtype=torch.complex128, device=dev)
        A, Ps, flux, mu = [], [], [], []
        for i, t in enumerate(part):
            I, fl, m = spectra(t)
            P, M = (I.abs() ** 2).mean(0), I.mean(0).flatten()
            noise = P[corner].mean() if bool(corner.any()) else 0.0
            a = torch.sqrt((P - noise).clamp(min=0) / stf.clamp(min=1e-4)) * t0
            a[c, c] = 0.0
            A.append(a)
            flux.append(fl.mean())
            mu.append(m.mean())
            I = I.reshape(F, -1)
            acc = torch.zeros(len(iw), dtype=torch.complex128, device=dev)
            for f in range(F):
                acc += I[f][iu] * I[f][iv] * I[f][iw].conj()
            acc /= F
            P = P.flatten()
            if case["photon_gain"] > 0:
                ph = case["photon_gain"] * fl
                acc += -(P[iu] + P[iv] + P[iw]) * (1 / ph).mean() + 2 * (1 / ph ** 2).mean()
            if case["weight"] == "unit":
                ab = acc.abs()
                acc = torch.where(ab > 0, acc / ab, acc)
            elif case["weight"] == "snr":
                d = P[iu] * P[iv] * P[iw]
                acc = torch.where(d > 0, acc / d, torch.zeros_like(acc))
            B[:, i] = acc
            z[at(0, 0), i] = 1.0
            for x, y in ((1, 0), (0, 1)):
                e = M[at(x, y)] / M[at(x, y)].abs()
                z[at(x, y), i], z[at(-x, -y), i] = e, e.conj()

        def unit_of(S, old):
            ab = S.abs()
            return torch.where(ab > 0, S / ab, old)

        for a, b in zip(ring_p[:-1], ring_p[1:]):
            sl = slice(ends[a], ends[b])
            t = z[iu[sl]] * z[iv[sl]] * B[sl].conj()
            S = torch.zeros((b - a, n, 2), dtype=torch.float64, device=dev)
            S.index_add_(0, point[sl] - a, torch.view_as_real(t))
            e = unit_of(torch.view_as_complex(S), torch.ones((b - a, n), dtype=torch.complex128, device=dev))
            z[pw[a:b]], z[pwn[a:b]] = e, e.conj()
        for _ in range(case["iters"]):
            S = torch.zeros((N * N, n, 2), dtype=torch.float64, device=dev)
            for idx, neg, kx, ky, t in ((iw, iwn, wx, wy, lambda: z[iu] * z[iv] * B.conj()),
                                        (iu, iun, wx - vx, wy - vy, lambda: z[iw] * z[iv].conj() * B),
                                        (iv, ivn, vx, vy, lambda: z[iw] * z[iu].conj() * B)):
                up = ((ky > 0) | ((ky == 0) & (kx > 0)))
                v = t()
                v = torch.where(up[:, None], v, v.conj())
                S.index_add_(0, torch.where(up, idx, neg), torch.view_as_real(v.resolve_conj()))
            e = unit_of(torch.view_as_complex(S)[pw], z[pw])
            z = z.clone()
            z[pw], z[pwn] = e, e.conj()
        for i, (x, y, w, h) in enumerate(part):
            X = torch.fft.ifftshift(A[i] * z[:, i].view(N, N))
            rec = torch.fft.ifft2(X).real * flux[i]
            rec[:h, :w] += mu[i] * window(w, h)
            if case["central"]:
                o = (N - stride) // 2
                blk = (slice(o, o + stride), slice(o, o + stride))
                num[y + o:y + o + stride, x + o:x + o + stride] = rec[blk] / window(N, N)[blk]
                den[y + o:y + o + stride, x + o:x + o + stride] = 1.0
            else:
                num[y:y + h, x:x + w] += rec[:h, :w]
                den[y:y + h, x:x + w] += window(w, h)
    ok = den >= 0.25
    return {"out": torch.where(ok, num / torch.where(ok, den, torch.ones_like(den)), torch.zeros_like(num)),
            "valid": None}


def exact(case, seed):
    """run()'s outputs in 64 bits; None where that takes too long (full TiO bursts)."""
    kind, F = case["kind"], case["F"]
    if kind == "front":
        s = prepare(case, seed)
        W, H, G, S = case["W"], case["H"], s["G"], s["S"]
        d = s["flat"].double() - s["dark"].double()
        gain = torch.where(d > 0, d / d[d > 0].mean(), torch.zeros_like(d))
        raw = s["raw"].view(torch.int16) if case["u16"] else s["raw"]
        x0, y0 = (W - G) // 2, (H - G) // 2
        cal = torch.empty((F, H, W), dtype=torch.float64, device="cuda")
        al, sh = torch.empty_like(cal), []
        ref = None
        for f in range(F):
            cal[f] = torch.where(gain > 0, (raw[f].double() - s["dark"].double()) / gain, torch.zeros_like(gain))
            if f == 0:
                ref = cal[0, y0:y0 + G, x0:x0 + G]
                ref = ref - ref.mean()
            area = cal[f, y0 - S:y0 + G + S, x0 - S:x0 + G + S]
            n = G + 2 * S
            cc = torch.fft.ifft2(torch.fft.fft2(area) * torch.fft.fft2(ref, s=(n, n)).conj()).real
            best = int(torch.argmax(cc[:2 * S + 1, :2 * S + 1]))
            sy, sx = best // (2 * S + 1) - S, best % (2 * S + 1) - S
            sh.append((sx, sy))
            yy = (torch.arange(H, device="cuda") + sy).clamp(0, H - 1)
            xx = (torch.arange(W, device="cuda") + sx).clamp(0, W - 1)
            al[f] = cal[f][yy][:, xx]
        return {"frames": cal, "aligned": al, "shifts": torch.tensor(sh, dtype=torch.int32)}
    shapes = _shapes(case) if kind == "batch" else [(case["W"], case["H"], case["N"], case["R"])] * case["bursts"]
    cost = sum(len(_tiles(W, H, N, case["stride"] * N // case["N"], case["central"])) * F * len(_pairs(N, case["fc"], R))
               for W, H, N, R in shapes)
    if cost > 1e11:
        return None
    got = []
    for k, (W, H, N, R) in enumerate(shapes):
        frames, dr0 = _frames(case, seed, k, W, H, N)
        given = case["stf"] or kind == "noalloc" or F < 2 or \
            not _estimable(W, H, N, case["stride"] * N // case["N"])
        got.append(_exact_burst(case, frames, _model_stf(N, case["fc"], dr0) if given else None, W, H, N, R))
    return got[0] if kind in ("call", "noalloc") else got
