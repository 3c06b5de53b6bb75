"""The Wiener residual and the Eq. 2 estimate at the edges of their tiles.

A thread takes 4 adjacent pixels of 2 or 8 rows (8 once the batch fills the
GPU), loads words where rows are 4-byte aligned and bytes elsewhere, and stores
vectors where rows allow it; the estimate sums its integer denominator in FP32
over 256 frames at a time.  Bounds: V and D are exact, W is a handful of FP32
roundings (2e-6 of the largest value, as for the whole residual); the estimate
adds a compensated sum and a corrected quotient (1e-6)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module")
def ctx():
    import paper_2207_14507_gb300 as p
    p.build()
    c = p.Context(0)
    yield c
    c.close()


def _frames(F, H, W, pitch, offset, seed):
    """uint8 frames [F, H, W] at a byte offset and row pitch on the device, and on the host."""
    rng = np.random.default_rng(seed)
    host = rng.integers(0, 256, size=(F, H, W)).astype(np.uint8)
    host[:, : H // 2, : W // 2] = 77                      # local variance 0
    buf = torch.zeros(offset + F * H * pitch, dtype=torch.uint8, device=DEV)
    dev = buf[offset:].view(F, H, pitch)[:, :, :W]
    dev.copy_(torch.from_numpy(host))
    return host, dev


@pytest.mark.parametrize("F,H,W,pad,offset", [(1, 1, 1, 0, 0), (2, 9, 1, 2, 1), (2, 1, 7, 0, 3), (3, 17, 130, 2, 0),
                                              (2, 66, 129, 3, 4), (40, 130, 257, 3, 0), (40, 130, 260, 0, 2),
                                              (152, 64, 256, 0, 0), (80, 65, 131, 0, 1)])
def test_residual_tile_edges(ctx, F, H, W, pad, offset):
    import paper_2207_14507_gb300 as prnu
    host, dev = _frames(F, H, W, W + pad, offset, F * H + W)
    for dtype in (torch.float32, torch.float16):
        out = torch.full((F, H, W), float("nan"), dtype=dtype, device=DEV)
        scale = torch.empty(F, device=DEV)
        norm = dtype != torch.float32
        ctx.prnu_residual(dev, out, scale=scale, pitch=W + pad,
                          flags=prnu.PRNU_WEIGHT_BY_INTENSITY | (prnu.PRNU_NORMALISE if norm else 0))
        got, s = out.double().cpu().numpy(), scale.double().cpu().numpy()
        for f in (0, F // 2, F - 1):
            ref, _ = oracle.prnu_residual(host[f])
            rms = np.sqrt(np.mean(ref * ref))
            want = 1 / rms if norm and rms > 0 else 1.0
            assert abs(s[f] / want - 1) <= 1e-6
            top = np.abs(ref * want).max() + 1e-30
            assert np.max(np.abs(got[f] - ref * want)) <= (2.0 ** -11 * 1.01 if norm else 2e-6) * top


def _ieee_residual(x, weight):
    """The residual in IEEE single precision, from the exact integer moments."""
    H, W = x.shape
    p = np.pad(x.astype(np.int64), 1, mode="edge")
    win = [p[dy:dy + H, dx:dx + W] for dy in range(3) for dx in range(3)]
    s1, s2 = sum(win), sum(w * w for w in win)
    V, D = 9 * s2 - s1 * s1, 9 * p[1:-1, 1:-1] - s1
    nu2 = float(V.sum()) / (81.0 * float(H) * float(W))
    f = np.float32
    wiener = (V > 0) & (V.astype(f) >= f(81.0 * nu2))
    num = np.where(wiener, f(9) * D.astype(f) * f(nu2), D.astype(f))
    w = num / np.where(wiener, V, 9).astype(f)
    return x.astype(f) * w if weight else w


@pytest.mark.parametrize("sigma", [0.4, 1.5, 6.0, 25.0, 100.0])
def test_residual_has_the_bits_of_ieee_division(ctx, sigma):
    """W = 9 D nu2 / V or D / 9 by a reciprocal and one correction: the rounded
    quotient itself, as V is an integer below 1.31e6 (the argument stands at
    residual_w)."""
    rng = np.random.default_rng(int(10 * sigma))
    base = rng.uniform(20, 235, size=(8, 1, 1)) + 40 * np.sin(np.arange(600) / 50)
    host = np.clip(np.rint(base + sigma * rng.standard_normal((8, 500, 600))), 0, 255).astype(np.uint8)
    host[0] = rng.choice([0, 255], size=host[0].shape)    # the largest V
    for weight in (0, 1):
        out = torch.empty(host.shape, dtype=torch.float32, device=DEV)
        ctx.prnu_residual(torch.from_numpy(host).to(DEV), out, flags=weight)
        got = out.cpu().numpy()
        for f in range(len(host)):
            np.testing.assert_array_equal(got[f], _ieee_residual(host[f], weight))


@pytest.mark.parametrize("L,H,W,pad,offset", [(1, 5, 3, 0, 1), (3, 16, 128, 0, 0), (20, 33, 130, 2, 0), (300, 18, 37, 0, 0)])
def test_estimate_tile_edges(ctx, L, H, W, pad, offset):
    host, dev = _frames(L, H, W, W + pad, offset, 7 * L + W)
    host[:, 0, 0] = 0
    dev.copy_(torch.from_numpy(host))                     # a pixel dark in every frame
    got = ctx.prnu_fingerprint_estimate(dev, pitch=W + pad).double().cpu().numpy()
    ref = oracle.fingerprint_estimate(host)
    assert got[0, 0] == 0
    assert np.max(np.abs(got - ref)) <= 1e-6 * np.abs(ref).max() + 1e-30


@pytest.mark.parametrize("L,H,W", [(1025, 70, 130), (65537, 3, 5), (70000, 2, 4)])
def test_estimate_of_many_frames(ctx, L, H, W):
    """More frames than one launch's grid holds, and than one run of noise powers."""
    host, dev = _frames(L, H, W, W, 0, L)
    got = ctx.prnu_fingerprint_estimate(dev).double().cpu().numpy()
    ref = oracle.fingerprint_estimate(host)
    assert np.max(np.abs(got - ref)) <= 1e-6 * np.abs(ref).max()
