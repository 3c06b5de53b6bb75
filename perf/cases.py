"""What the performance of this framework is measured on: calls that a user's
program makes, through the public entry points, with inputs of the kind that
they meet (stabilised frames of a camera whose fingerprint is tested).

A case is a dict with a "kind" (which entry points), a frame size and options:

  pce         one aligned pair scored against a kept fingerprint
  search      the grid search over (scale, rotation) of stored residuals
  correction  the iterative coarse-to-fine correction
  literal     the search that warps the frame and extracts its residual per node
  residual    the 3x3 Wiener residual of a batch of frames
  wavelet     the wavelet-denoiser residual of a batch of frames
  enrol       a camera's fingerprint from still images, brought to a video's
              geometry, its spectrum cached and one frame scored against it

One library context serves all states, as in a program that tests many videos.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as tf

import paper_2207_14507_gb300 as prnu

DEV = "cuda:0"
TORCH_DTYPE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
PRNU_DTYPE = {"f32": prnu.PRNU_F32, "f16": prnu.PRNU_F16, "bf16": prnu.PRNU_BF16}
WEIGHT = prnu.PRNU_WEIGHT_BY_INTENSITY
NORMALISE = prnu.PRNU_NORMALISE


# ---------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest call: an unstabilised frame against one kept fingerprint
        dict(name="pce_720p", kind="pce", H=720, W=1280, fp="f32"),
        # a quick look at a few small frames: launches and latency count
        dict(name="search_256", kind="search", H=256, W=256, F=4, P=1, nlam=11, nth=11, dlam=0.008, dth=0.2,
             k=0, dtype="f32", fp="f32"),
        # the headline: full-HD frames over the full grid
        dict(name="search_1080p", kind="search", H=1080, W=1920, F=2, P=1, nlam=41, nth=41, dlam=0.005, dth=0.25,
             k=0, dtype="f32", fp="f32"),
        # a video's successive frames, each in a window around the last one's node; half storage
        dict(name="search_1080p_windows", kind="search", H=1080, W=1920, F=16, P=1, nlam=41, nth=41, dlam=0.005,
             dth=0.25, k=10, dtype="f16", fp="f16"),
        # 4K video, half storage
        dict(name="search_4k", kind="search", H=2160, W=3840, F=2, P=1, nlam=13, nth=13, dlam=0.01, dth=0.5,
             k=0, dtype="f16", fp="f16"),
        # a video against the cameras of a case (8 fingerprints per frame)
        dict(name="search_720p_8cameras", kind="search", H=720, W=1280, F=4, P=8, nlam=7, nth=7, dlam=0.01, dth=0.5,
             k=0, dtype="f16", fp="f16"),
        # a size of no compiled plan, bfloat16 storage
        dict(name="search_vga", kind="search", H=480, W=640, F=4, P=1, nlam=21, nth=21, dlam=0.01, dth=0.5,
             k=0, dtype="bf16", fp="f32"),
        # the search as the paper states it
        dict(name="literal_1080p", kind="literal", H=1080, W=1920, F=1, P=1, nlam=21, nth=21, dlam=0.01, dth=0.5),
        # the iterative correction with its dense first angle grid
        dict(name="correction_1080p", kind="correction", H=1080, W=1920, F=2, half=50, dtype="f32", fp="f32"),
        # ingest of a second of video into half storage
        dict(name="residual_1080p", kind="residual", H=1080, W=1920, F=30, pad=0, dtype="f16", weight=True,
             norm=True),
        # ingest with the paper's own denoiser
        dict(name="wavelet_1080p", kind="wavelet", H=1080, W=1920, F=8, pad=0, dtype="f32", weight=True, norm=False),
        # a camera enrolled from twelve-megapixel stills for full-HD video
        dict(name="enrol_12mp", kind="enrol", L=16, Hin=3000, Win=4000, scale=0.48, y0=180, x0=0, H=1080, W=1920),
    ]


def _smooth(lo, hi):
    """The even 5-smooth numbers in [lo, hi]."""
    out = []
    for n in range(lo + lo % 2, hi + 1, 2):
        m = n
        for p in (2, 3, 5):
            while m % p == 0:
                m //= p
        if m == 1:
            out.append(n)
    return out


def _log_pick(rng, values):
    """One of the sorted values, spread over their logarithm."""
    x = math.exp(rng.uniform(math.log(values[0]), math.log(values[-1])))
    return min(values, key=lambda v: abs(math.log(v / x)))


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _video_size(rng):
    if rng.random() < 0.5:
        return rng.choice([(256, 256), (720, 1280), (1080, 1920), (2160, 3840)])
    H = _log_pick(rng, _smooth(64, 2160))
    return H, _log_pick(rng, _smooth(max(64, H // 2), min(4096, 3 * H)))


def draw(rng):
    kind = rng.choice(["search"] * 6 + ["pce", "correction", "literal", "residual", "wavelet", "enrol"])
    if kind in ("residual", "wavelet"):
        H = _log_int(rng, 32, 2300)
        W = _log_int(rng, max(32, H // 2), min(4000, 3 * H))
        F = max(1, min(_log_int(rng, 1, 32), int((5e7 if kind == "residual" else 1.5e7) / (H * W))))
        return dict(kind=kind, H=H, W=W, F=F, pad=rng.choice([0, 0, 3, 16, 64]), dtype=rng.choice(["f32", "f16", "bf16"]),
                    weight=rng.random() < 0.8, norm=rng.random() < 0.5)
    if kind == "enrol":
        H, W = rng.choice([(720, 1280), (1080, 1920), (_log_pick(rng, _smooth(240, 1080)), _log_pick(rng, _smooth(320, 1920)))])
        s = rng.choice([0.48, 0.5, 0.64, 0.75, 1.0])
        Hin = int(math.ceil(H / s)) + rng.randint(1, 200)
        Win = int(math.ceil(W / s)) + rng.randint(1, 200)
        Hs, Ws = int(Hin * s), int(Win * s)
        return dict(kind=kind, L=max(1, min(_log_int(rng, 2, 40), int(1.5e8 / (Hin * Win)))), Hin=Hin, Win=Win, scale=s,
                    y0=rng.randint(0, Hs - H), x0=rng.randint(0, Ws - W), H=H, W=W)
    H, W = _video_size(rng)
    if kind == "pce":
        return dict(kind=kind, H=H, W=W, fp=rng.choice(["f32", "f16"]))
    if kind == "correction":
        half = rng.choice([10, 25, 50])
        return dict(kind=kind, H=H, W=W, F=max(1, min(rng.randint(1, 4), int(6e8 / (H * W * 22 * half)))), half=half,
                    dtype=rng.choice(["f32", "f16"]), fp=rng.choice(["f32", "f16"]))
    # total pixels of all candidates, at most a quarter of the largest listed case
    total = math.exp(rng.uniform(math.log(3e7), math.log(1.6e9 if kind == "search" else 3e8)))
    P = rng.choice([1, 1, 1, 2, 3, 5, 8, 16]) if kind == "search" else 1
    F = rng.randint(1, 6)
    nodes = max(9.0, total / (H * W * F * P))
    nlam = max(3, min(41, int(math.sqrt(nodes))))
    nth = max(3, min(81, int(nodes / nlam)))
    while F > 1 and H * W * F * P * nlam * nth > 2.5 * total:
        F -= 1
    grid = dict(nlam=nlam, nth=nth, dlam=round(rng.uniform(0.002, 0.2 / nlam), 5), dth=round(rng.uniform(0.02, 10.0 / nth), 4))
    if kind == "literal":
        return dict(kind=kind, H=H, W=W, F=F, P=1, **grid)
    k = rng.randint(1, 5) if min(nlam, nth) >= 5 and rng.random() < 0.4 else 0
    return dict(kind=kind, H=H, W=W, F=F, P=P, **grid, k=k, dtype=rng.choice(["f32", "f16", "bf16"]),
                fp=rng.choice(["f32", "f16"]))


# ---------------------------------------------------------------- inputs

_CTX = None


def _context():
    global _CTX
    if _CTX is None:
        _CTX = prnu.Context(0)
    return _CTX


class _Grid:
    def __init__(self, c):
        self.nlam, self.nth = c["nlam"], c["nth"]
        self.lam0 = 1.0 - c["dlam"] * (c["nlam"] - 1) / 2
        self.th0_deg = -c["dth"] * (c["nth"] - 1) / 2
        self.dlam, self.dth_deg = c["dlam"], c["dth"]

    def nodes(self):
        """The float32 node values the library searches, as doubles."""
        f = np.float32
        lam = f(np.float64(f(self.lam0)) + np.arange(self.nlam) * np.float64(f(self.dlam)))
        th = f(np.float64(f(self.th0_deg)) + np.arange(self.nth) * np.float64(f(self.dth_deg)))
        return lam.astype(np.float64), th.astype(np.float64)


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _content(H, W, g):
    """Smooth scene luminance in [16, 240]."""
    low = torch.randn((1, 1, H // 16 + 4, W // 16 + 4), generator=g, device=DEV)
    c = tf.interpolate(low, size=(H, W), mode="bicubic", align_corners=True)[0, 0]
    return 16 + 224 * (c - c.min()) / (c.max() - c.min())


def _warp(img, lam, th_deg, shift=(0.0, 0.0), inverse=True, border="zeros"):
    """img sampled at c + A (p - c) + shift: A = Rot(-th)/lam (the search's
    inverse warp), or lam Rot(th) with inverse False."""
    H, W = img.shape
    t = math.radians(th_deg)
    ct, st = math.cos(t), math.sin(t)
    a = (ct / lam, st / lam, -st / lam, ct / lam) if inverse else (lam * ct, -lam * st, lam * st, lam * ct)
    x = torch.arange(W, device=DEV, dtype=img.dtype) - (W - 1) / 2
    y = torch.arange(H, device=DEV, dtype=img.dtype)[:, None] - (H - 1) / 2
    qx = a[0] * x + a[1] * y + shift[1]
    qy = a[2] * x + a[3] * y + shift[0]
    grid = torch.stack((qx * (2 / (W - 1)), qy * (2 / (H - 1))), -1)
    return tf.grid_sample(img[None, None], grid[None], mode="bilinear", padding_mode=border, align_corners=True)[0, 0]


def _frames(case, seed, F, H, W, lam_span, th_span, fps=1):
    """fps fingerprints and F stabilised uint8 frames of the first one's camera, with their planted nodes."""
    g = _generator(seed)
    r = np.random.default_rng(seed)
    Ks = [0.02 * torch.randn((H, W), generator=g, device=DEV) for _ in range(fps)]
    out = torch.empty((F, H, W), dtype=torch.uint8, device=DEV)
    planted = []
    smax = min(H, W) // 16
    for f in range(F):
        lam, th = 1 + r.uniform(-1, 1) * lam_span, r.uniform(-1, 1) * th_span
        shift = (int(r.integers(-smax, smax + 1)), int(r.integers(-smax, smax + 1)))
        s = _content(H, W, g) * (1 + Ks[0]) + 2 * torch.randn((H, W), generator=g, device=DEV)
        out[f] = _warp(s, lam, th, shift, inverse=False, border="border").round_().clamp_(0, 255).to(torch.uint8)
        planted.append((lam, th))
    return Ks, out, planted


def _moments(x):
    """Sums of x and x^2 over the 3x3 neighbourhood, borders replicated."""
    p = tf.pad(x[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
    H, W = x.shape
    s1, s2 = torch.zeros_like(x), torch.zeros_like(x)
    for dy in range(3):
        for dx in range(3):
            v = p[dy:dy + H, dx:dx + W]
            s1 += v
            s2 += v * v
    return s1, s2


def _wiener(x, weight):
    """The 3x3 Wiener residual of one frame (double in, double out)."""
    s1, s2 = _moments(x)
    mu = s1 / 9
    var = (s2 / 9 - mu * mu).clamp_(min=0)
    nu2 = var.mean()
    den = torch.maximum(var, nu2)
    gain = torch.where(den > 0, (var - nu2).clamp(min=0) / torch.where(den > 0, den, 1.0), 1.0)
    w = (x - mu) * (1 - gain)
    return x * w if weight else w


def _stored_residuals(frames, dtype):
    """Stored residuals of the frames and their scales (half storage: unit RMS), made without the library."""
    F, H, W = frames.shape
    out = torch.empty((F, H, W), dtype=TORCH_DTYPE[dtype], device=DEV)
    scale = torch.ones(F, device=DEV)
    for f in range(F):
        R = _wiener(frames[f].double(), True)
        if dtype != "f32":
            scale[f] = (1 / R.square().mean().sqrt()).float()
            R = R * scale[f].double()
        out[f] = R.to(out.dtype)
    return out, scale


def _search_inputs(case, seed):
    span = 0.45 * case["dlam"] * (case["nlam"] - 1), 0.45 * case["dth"] * (case["nth"] - 1)
    Ks, frames, planted = _frames(case, seed, case["F"], case["H"], case["W"], *span, fps=case["P"])
    windows = None
    if case.get("k"):
        g, r = _Grid(case), np.random.default_rng(seed + 1)
        windows = np.empty((case["F"], 4), np.int32)
        for f, (lam, th) in enumerate(planted):
            k = int(r.integers(1 + (case["k"] > 2), case["k"] + 1))
            for o, v0, dv, n, v in ((0, g.lam0, g.dlam, g.nlam, lam), (2, g.th0_deg, g.dth_deg, g.nth, th)):
                c = int(round((v - v0) / dv))
                lo = min(max(c - k, 0), max(0, n - 1 - 2 * k))
                windows[f, o:o + 2] = lo, min(n - 1, lo + 2 * k)
    return Ks, frames, windows


def _correction_inputs(case, seed):
    Ks, frames, planted = _frames(case, seed, case["F"], case["H"], case["W"], 0.05, 0.1 * case["half"] * 0.8)
    r = np.random.default_rng(seed + 1)
    init_lam = np.array([p[0] + r.uniform(-0.03, 0.03) for p in planted], np.float32)
    init_th = np.array([p[1] + r.uniform(-0.06, 0.06) * case["half"] for p in planted], np.float32)
    return Ks[0], frames, init_lam, init_th


def _padded_frames(case, seed):
    """uint8 frames [F, H, W] with `pad` unused bytes after each row."""
    g = _generator(seed)
    buf = torch.zeros((case["F"], case["H"], case["W"] + case["pad"]), dtype=torch.uint8, device=DEV)
    frames = buf[:, :, :case["W"]]
    for f in range(case["F"]):
        s = _content(case["H"], case["W"], g) + 2 * torch.randn((case["H"], case["W"]), generator=g, device=DEV)
        frames[f] = s.round_().clamp_(0, 255).to(torch.uint8)
    return frames


def _enrol_inputs(case, seed):
    g = _generator(seed)
    Hin, Win = case["Hin"], case["Win"]
    K = 0.02 * torch.randn((Hin, Win), generator=g, device=DEV)
    frames = torch.empty((case["L"], Hin, Win), dtype=torch.uint8, device=DEV)
    for l in range(case["L"]):
        s = _content(Hin, Win, g) * (1 + K) + 2 * torch.randn((Hin, Win), generator=g, device=DEV)
        frames[l] = s.round_().clamp_(0, 255).to(torch.uint8)
    # the frame scored afterwards: a residual that holds the resized fingerprint
    small = tf.interpolate(K[None, None], size=(int(Hin * case["scale"]), int(Win * case["scale"])), mode="bilinear",
                           antialias=True)[0, 0][case["y0"]:case["y0"] + case["H"], case["x0"]:case["x0"] + case["W"]]
    X = 100 * small + 2 * torch.randn(small.shape, generator=g, device=DEV)
    return frames, X.contiguous()


# ---------------------------------------------------------------- prepare and run

class _State:
    """Inputs, and the fingerprint handles that the program keeps for them."""

    def __init__(self, case):
        self.case, self.ctx, self.handles = case, _context(), []

    def __del__(self):
        try:
            for h in self.handles:
                self.ctx.prnu_fingerprint_release(h)
        except Exception:   # the interpreter is going down
            pass


def prepare(case, seed):
    s = _State(case)
    kind, H, W = case["kind"], case["H"], case["W"]
    term = lambda K: s.handles.append(s.ctx.prnu_fingerprint_term(K, PRNU_DTYPE[case["fp"]]))  # noqa: E731
    if kind == "pce":
        g = _generator(seed)
        K = 0.02 * torch.randn((H, W), generator=g, device=DEV)
        s.X = 100 * K.roll((5, -9), (0, 1)) + 4 * torch.randn((H, W), generator=g, device=DEV)
        term(K)
    elif kind == "search":
        Ks, frames, s.windows = _search_inputs(case, seed)
        s.resid, s.scale = _stored_residuals(frames, case["dtype"])
        for K in Ks:
            term(K)
        s.grid = _Grid(case)
        s.all_pce = torch.empty((case["F"], case["P"], s.grid.nlam * s.grid.nth), dtype=torch.float64, device=DEV)
    elif kind == "correction":
        K, frames, s.init_lam, s.init_th = _correction_inputs(case, seed)
        s.resid, s.scale = _stored_residuals(frames, case["dtype"])
        term(K)
    elif kind == "literal":
        Ks, s.frames, _ = _search_inputs(case, seed)
        s.handles.append(s.ctx.prnu_fingerprint_term(Ks[0]))
        s.grid = _Grid(case)
    elif kind in ("residual", "wavelet"):
        s.frames = _padded_frames(case, seed)
        s.out = torch.empty((case["F"], H, W), dtype=TORCH_DTYPE[case["dtype"]], device=DEV)
        s.scale = torch.empty(case["F"], device=DEV)
        s.flags = (WEIGHT if case["weight"] else 0) | (NORMALISE if case["norm"] else 0)
    else:
        s.frames, s.X = _enrol_inputs(case, seed)
        s.K = torch.empty((case["Hin"], case["Win"]), device=DEV)
        s.Kv = torch.empty((H, W), device=DEV)
    return s


def _fields(res):
    return {k: np.ascontiguousarray(res[k]) for k in ("lam", "th_deg", "dy", "dx", "pce", "peak", "cand_idx")}


def run(s):
    c, ctx, kind = s.case, s.ctx, s.case["kind"]
    if kind == "pce":
        return ctx.pce_score(s.X, s.handles[0])
    if kind == "search":
        res = ctx.eis_grid_search(s.resid, s.handles, s.grid, windows=s.windows, scale=s.scale, all_pce=s.all_pce)
        return dict(_fields(res), all_pce=s.all_pce)
    if kind == "correction":
        res, its = ctx.eis_correction(s.resid, s.handles, s.init_lam, s.init_th, 3, c["half"], scale=s.scale)
        return dict(_fields(res), iters=its)
    if kind == "literal":
        return _fields(ctx.eis_grid_search_frames(s.frames, s.handles, s.grid))
    if kind == "residual":
        ctx.prnu_residual(s.frames, s.out, scale=s.scale, flags=s.flags, pitch=c["W"] + c["pad"])
        return dict(out=s.out, scale=s.scale)
    if kind == "wavelet":
        ctx.prnu_residual_wavelet(s.frames, s.out, flags=s.flags, scale=s.scale, pitch=c["W"] + c["pad"])
        return dict(out=s.out, scale=s.scale)
    ctx.prnu_fingerprint_estimate(s.frames, out=s.K)
    ctx.prnu_fingerprint_resize(s.K, c["scale"], c["y0"], c["x0"], c["H"], c["W"], out=s.Kv)
    h = ctx.prnu_fingerprint_term(s.Kv)
    score = ctx.pce_score(s.X, h)
    ctx.prnu_fingerprint_release(h)
    return dict(score, K=s.K, Kv=s.Kv)


# ---------------------------------------------------------------- work and tolerance

def _candidates(case):
    if case["kind"] == "correction":
        return case["F"] * (11 * (2 * case["half"] + 1) + 2 * 121)
    if case["kind"] == "pce":
        return 1
    n = case["nlam"] * case["nth"]
    if case.get("k"):
        k = (1 + (case["k"] > 2) + case["k"]) / 2
        n = min(n, (2 * k + 1) ** 2)
    return n * case["F"] * case["P"]


def work(case):
    kind, N = case["kind"], case["H"] * case["W"]
    size = {"f32": 4, "f16": 2, "bf16": 2}
    if kind in ("residual", "wavelet"):
        # 3x3 moments and the filter: about 40 operations a pixel; four levels of two 8-tap filters each way and
        # four window sums: about 250
        return {"bytes": case["F"] * N * (1 + size[case["dtype"]]), "flops": case["F"] * N * (40 if kind == "residual" else 250)}
    fft = 2.5 * N * math.log2(N)   # one real 2-D transform
    if kind == "enrol":
        Nin = case["Hin"] * case["Win"]
        taps = (2 / case["scale"] + 1) ** 2
        return {"bytes": case["L"] * Nin + 8 * Nin + 16 * N, "flops": case["L"] * Nin * 43 + N * 2 * taps + 3 * fft}
    n = _candidates(case)
    forward = n / case.get("P", 1)   # the warp and the forward transform do not depend on the fingerprint
    flops = forward * (fft + (0 if kind == "pce" else 14 * N)) + n * (fft + 3 * N + 3 * N)
    if kind == "literal":
        flops += forward * 40 * N
    stored = 1 if kind == "literal" else 4 if kind == "pce" else size[case["dtype"]]
    P, F = case.get("P", 1), case.get("F", 1)
    return {"bytes": N * (F * stored + P * size[case.get("fp", "f32")]), "flops": flops}


def tolerance(case):
    # about four times the error against exact(), where 16-bit storage does not round both alike
    kind, dtype = case["kind"], case.get("dtype")
    if kind in ("residual", "wavelet"):
        if dtype == "f32":   # 32-bit sums of a pixel's neighbourhood (8e-6 with the wavelet's eight passes)
            return {"rel": 2e-6 if kind == "residual" else 3e-5, "max": 1e-3}
        # a value on the edge of two 16-bit numbers may round either way
        return {"rel": 5e-4, "max": 2e-3} if dtype == "f16" else {"rel": 4e-3, "max": 1.6e-2}
    if kind in ("pce", "enrol"):   # 32-bit transforms: 2e-7
        return {"rel": 1e-6, "max": 4e-5}
    # sample points in 32 bits: to 1e-4 pixels, 1e-5 to 9e-5 of a PCE; the node and the shift are the same
    return {"rel": 2e-4, "max": 1e-3}


# ---------------------------------------------------------------- the same in 64 bits

def _score(X, Kf):
    """PCE, signed shift and peak of X (double [H, W]) against the spectrum of K - mean K."""
    H, W = X.shape
    C = torch.fft.irfft2(torch.fft.rfft2(X).conj() * Kf, s=(H, W))
    i = int(C.argmax())
    py, px = i // W, i % W
    peak = float(C[py, px])
    C2 = C.square_()
    ys = (torch.arange(py - 5, py + 6, device=DEV) % H)[:, None]
    xs = torch.arange(px - 5, px + 6, device=DEV) % W
    C2[ys, xs] = 0
    E = float(C2.sum()) / (H * W - 121)
    return math.copysign(peak * peak / E, peak), (py + H // 2) % H - H // 2, (px + W // 2) % W - W // 2, peak


def _spectrum(K):
    K = K.double()
    return torch.fft.rfft2(K - K.mean())


def _best(rows):
    """Rows (pce, dy, dx, peak, lam, th, index) -> the first of largest PCE."""
    return max(rows, key=lambda r: (r[0], -r[6]))


def _as_fields(best, shape, scale):
    a = np.array(best, np.float64)
    return dict(lam=a[:, 4].reshape(shape), th_deg=a[:, 5].reshape(shape), dy=None, dx=None,
                pce=a[:, 0].reshape(shape), peak=(a[:, 3] / scale).reshape(shape), cand_idx=None)


def _exact_search(case, seed):
    literal = case["kind"] == "literal"
    Ks, frames, windows = _search_inputs(case, seed)
    Kf = [_spectrum(K) for K in Ks]
    lams, ths = _Grid(case).nodes()
    F, P, n = case["F"], case["P"], len(lams) * len(ths)
    if not literal:
        resid, scale = _stored_residuals(frames, case["dtype"])
    every = np.full((F, P, n), np.nan)
    best = []
    for f in range(F):
        img = frames[f].double() if literal else resid[f].double()
        w = (0, len(lams) - 1, 0, len(ths) - 1) if windows is None else windows[f]
        rows = [[] for _ in range(P)]
        for i in range(w[0], w[1] + 1):
            for j in range(w[2], w[3] + 1):
                X = _warp(img, lams[i], ths[j])
                if literal:
                    X = _wiener(X, True)
                for p in range(P):
                    r = _score(X, Kf[p])
                    every[f, p, i * len(ths) + j] = r[0]
                    rows[p].append(r + (lams[i], ths[j], i * len(ths) + j))
        best += [_best(x) for x in rows]
    s = 1.0 if literal else np.repeat(scale.double().cpu().numpy(), P)
    out = _as_fields(best, (F, P), s)
    return out if literal else dict(out, all_pce=every)


def _exact_correction(case, seed):
    K, frames, init_lam, init_th = _correction_inputs(case, seed)
    resid, scale = _stored_residuals(frames, case["dtype"])
    Kf = _spectrum(K)
    best = []
    for f in range(case["F"]):
        cl, ct, found = init_lam[f], init_th[f], None
        for it in range(3):
            sl, st = np.float32(0.01 * 10.0 ** -it), np.float32(0.1 * 10.0 ** -it)
            hb = case["half"] if it == 0 else 5
            rows = []
            for a in range(-5, 6):
                for b in range(-hb, hb + 1):
                    lam = float(np.float32(float(cl) + a * float(sl)))
                    th = float(np.float32(float(ct) + b * float(st)))
                    rows.append(_score(_warp(resid[f].double(), lam, th), Kf) + (lam, th, len(rows)))
            top = _best(rows)
            if found is None or top[0] > found[0]:
                found = top
            if top[6] == 5 * (2 * hb + 1) + hb:
                break
            cl, ct = np.float32(top[4]), np.float32(top[5])
        best.append(found)
    return dict(_as_fields(best, (case["F"], 1), scale.double().cpu().numpy()), iters=None)


# Daubechies' 8-tap scaling filter (4 vanishing moments)
_DB8 = [0.2303778133088964, 0.7148465705529154, 0.6308807679298587, -0.0279837694168599, -0.1870348117190931,
        0.0308413818355607, 0.0328830116668852, -0.0105974017850690]


def _analyse(x, dim):
    """Low and high half of x along dim, periodic."""
    lo = hi = 0
    for k in range(8):
        v = x.roll(-k, dim)
        v = v[::2] if dim == 0 else v[:, ::2]
        lo = lo + _DB8[k] * v
        hi = hi + (-1) ** k * _DB8[7 - k] * v
    return lo, hi


def _synthesise(lo, hi, dim):
    shape = list(lo.shape)
    shape[dim] *= 2
    out = torch.zeros(shape, dtype=lo.dtype, device=lo.device)
    for k in range(8):
        up = torch.zeros_like(out)
        v = _DB8[k] * lo + (-1) ** k * _DB8[7 - k] * hi
        if dim == 0:
            up[::2] = v
        else:
            up[:, ::2] = v
        out += up.roll(k, dim)
    return out


def _noise_part(c, s0):
    e = tf.pad((c * c)[None, None], (4, 4, 4, 4))
    s2 = None
    for r in (1, 2, 3, 4):
        m = tf.avg_pool2d(e[:, :, 4 - r:e.shape[2] - 4 + r, 4 - r:e.shape[3] - 4 + r], 2 * r + 1, stride=1)[0, 0]
        v = (m - s0).clamp_(min=0)
        s2 = v if s2 is None else torch.minimum(s2, v)
    return c * s0 / (s2 + s0)


def _wavelet(x, weight, sigma0=3.0):
    H, W = x.shape
    Hp, Wp = -(-H // 16) * 16, -(-W // 16) * 16
    a = torch.cat((x, x[H - (Hp - H):].flip(0)), 0) if Hp > H else x
    a = torch.cat((a, a[:, W - (Wp - W):].flip(1)), 1) if Wp > W else a
    bands = []
    for _ in range(4):
        lo, hi = _analyse(a, 1)
        (a, lh), (hl, hh) = _analyse(lo, 0), _analyse(hi, 0)
        bands.append((lh, hl, hh))
    a = torch.zeros_like(a)
    for lh, hl, hh in reversed(bands):
        lh, hl, hh = (_noise_part(c, sigma0 * sigma0) for c in (lh, hl, hh))
        a = _synthesise(_synthesise(a, lh, 0), _synthesise(hl, hh, 0), 1)
    w = a[:H, :W]
    return x * w if weight else w


def _exact_residual(case, seed):
    frames = _padded_frames(case, seed)
    out = torch.empty(frames.shape, dtype=torch.float64, device=DEV)
    scale = torch.ones(case["F"], dtype=torch.float64, device=DEV)
    for f in range(case["F"]):
        out[f] = (_wiener if case["kind"] == "residual" else _wavelet)(frames[f].double(), case["weight"])
        if case["norm"]:
            scale[f] = 1 / out[f].square().mean().sqrt()
            out[f] *= scale[f]
    return dict(out=out, scale=scale)


def _resize_weights(n_in, scale, first, n):
    a = min(scale, 1.0)
    u = (torch.arange(n, dtype=torch.float64) + first + 0.5) / scale - 0.5
    m = torch.zeros((n, n_in), dtype=torch.float64)
    lo = torch.floor(u - 1 / a).long()
    for k in range(int(2 / a) + 3):
        j = lo + k
        t = (1 - (j - u).abs() * a).clamp(min=0)
        m.scatter_add_(1, j.clamp(0, n_in - 1)[:, None], t[:, None])
    return (m / m.sum(1, keepdim=True)).to(DEV)


def _exact_enrol(case, seed):
    frames, X = _enrol_inputs(case, seed)
    num = torch.zeros(frames.shape[1:], dtype=torch.float64, device=DEV)
    den = torch.zeros_like(num)
    for l in range(case["L"]):
        I = frames[l].double()
        num += _wiener(I, True)
        den += I * I
    K = torch.where(den > 0, num / torch.where(den > 0, den, 1.0), 0.0)
    Wy = _resize_weights(case["Hin"], case["scale"], case["y0"], case["H"])
    Wx = _resize_weights(case["Win"], case["scale"], case["x0"], case["W"])
    Kv = Wy @ K @ Wx.T
    pce, _, _, peak = _score(X.double(), _spectrum(Kv))
    return dict(pce=pce, dy=None, dx=None, peak=peak, K=K, Kv=Kv)


def exact(case, seed):
    kind = case["kind"]
    if kind == "pce":
        g = _generator(seed)
        K = 0.02 * torch.randn((case["H"], case["W"]), generator=g, device=DEV)
        X = 100 * K.roll((5, -9), (0, 1)) + 4 * torch.randn((case["H"], case["W"]), generator=g, device=DEV)
        pce, _, _, peak = _score(X.double(), _spectrum(K))
        return dict(pce=pce, dy=None, dx=None, peak=peak)
    if kind in ("search", "literal"):
        return _exact_search(case, seed)
    if kind == "correction":
        return _exact_correction(case, seed)
    if kind in ("residual", "wavelet"):
        return _exact_residual(case, seed)
    return _exact_enrol(case, seed)
