"""The wavelet residual at the edges of its tiles (64 x 64 pixels a block, 56 x 32
coefficients of the shrinkage): sizes of one block and less, of a few, with tiles
that hold no edge, ragged, with an even or odd row pitch; one chunk of frames
and several, normalised or not.  Bound: FP32 sums of eight filter passes, 1e-3 of
the largest value as for the whole denoiser, 2e-5 of the residual's norm (the
measured 7e-6 times three)."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.mark.parametrize("norm", [False, True])
@pytest.mark.parametrize("F,H,W,pad,sigma0", [(1, 16, 16, 0, 3.0), (2, 17, 31, 1, 3.0), (3, 64, 65, 0, 3.0),
                                              (2, 63, 129, 2, 0.5), (18, 40, 97, 3, 3.0), (2, 144, 80, 0, 1e10),
                                              (1, 130, 200, 0, 0.0), (1, 226, 334, 0, 3.0), (2, 240, 250, 1, 3.0), (1, 225, 259, 1, 3.0)])
def test_wavelet_tile_edges(F, H, W, pad, sigma0, norm):
    import paper_2207_14507_gb300 as prnu
    prnu.build()
    rng = np.random.default_rng(H * W + F)
    host = np.clip(128 + 40 * rng.standard_normal((F, H, W)), 0, 255).astype(np.uint8)
    buf = torch.zeros((F, H, W + pad), dtype=torch.uint8, device=DEV)
    buf[:, :, :W].copy_(torch.from_numpy(host))
    out = torch.full((F, H, W), float("nan"), device=DEV)
    scale = torch.empty(F, device=DEV)
    with prnu.Context(0) as ctx:
        ctx.prnu_residual_wavelet(buf[:, :, :W], out, sigma0=sigma0, pitch=W + pad, scale=scale,
                                  flags=prnu.PRNU_WEIGHT_BY_INTENSITY | (prnu.PRNU_NORMALISE if norm else 0))
        for dtype in (torch.float16, torch.bfloat16):   # the same values, rounded
            half = torch.empty((F, H, W), dtype=dtype, device=DEV)
            ctx.prnu_residual_wavelet(buf[:, :, :W], half, sigma0=sigma0, pitch=W + pad, scale=scale,
                                      flags=prnu.PRNU_WEIGHT_BY_INTENSITY | (prnu.PRNU_NORMALISE if norm else 0))
            assert torch.equal(half, out.to(dtype))
        got, s = out.double().cpu().numpy(), scale.double().cpu().numpy()
    for f in (0, F - 1):
        W0 = oracle.wavelet_residual(host[f].astype(np.float64), sigma0)
        ref = host[f] * (W0[0] if isinstance(W0, tuple) else W0)
        rms = np.sqrt(np.mean(ref * ref))
        want = 1 / rms if norm and rms > 0 else 1.0
        assert abs(s[f] / want - 1) <= 2e-5
        diff = got[f] - ref * want
        assert np.max(np.abs(diff)) <= 1e-3 * np.abs(ref * want).max() + 1e-30
        assert np.linalg.norm(diff) <= 2e-5 * np.linalg.norm(ref * want) + 1e-30
