"""Residuals and fingerprints that hold a NaN or an infinity: the correlation
has no ordered value, so the score is -inf at shift (0, 0), at the sizes with
and without planned kernels, in few and in many candidates, and the frames
beside it keep their bits."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
SIZES = [(256, 256), (720, 1280), (1080, 1920), (2160, 3840), (480, 640), (16, 16), (18, 1000)]


@pytest.fixture(scope="module")
def prnu():
    import paper_2207_14507_gb300 as p
    p.build()
    return p


@pytest.fixture(scope="module")
def ctx(prnu):
    with prnu.Context(0) as c:
        yield c


def _images(H, W, n, seed=5):
    g = torch.Generator(device=DEV).manual_seed(seed)
    return torch.randn((n, H, W), generator=g, device=DEV)


def _no_peak(r):
    return r["pce"] == -np.inf and r["peak"] == -np.inf and (r["dy"], r["dx"]) == (0, 0)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
@pytest.mark.parametrize("H,W", SIZES)
def test_pair_without_a_maximum(prnu, ctx, H, W, bad):
    X, K = _images(H, W, 2)
    want = ctx.pce_score(X, ctx.prnu_fingerprint_term(K))
    Xb, Kb = X.clone(), K.clone()
    Xb[H // 2, W // 3] = bad
    Kb[3, 5] = bad
    h, hb = ctx.prnu_fingerprint_term(K), ctx.prnu_fingerprint_term(Kb)
    assert _no_peak(ctx.pce_score(Xb, h)) and _no_peak(ctx.pce_score(X, hb))
    if H * W <= 1 << 20:
        assert _no_peak(prnu.pce_score_noalloc(Xb, K))
    assert ctx.pce_score(X, h) == want
    for v in (h, hb):
        ctx.prnu_fingerprint_release(v)


@pytest.mark.parametrize("dtype", ["float32", "float16"])
@pytest.mark.parametrize("persistent", [0, 1, 2])
@pytest.mark.parametrize("H,W,n", [(256, 256, 15), (720, 1280, 5), (1080, 1920, 3), (480, 640, 3), (480, 640, 13)])
def test_search_frames_beside_it_keep_their_bits(ctx, H, W, n, persistent, dtype):
    """A frame with a NaN between two good ones: n x n candidates each."""
    R = _images(H, W, 3).to(getattr(torch, dtype))
    hs = [ctx.prnu_fingerprint_term(K) for K in _images(H, W, 2, 6)]
    g = synth.Grid(0.99, 0.02 / n, n, -0.5, 1.0 / n, n)
    t = ctx.prnu_get_tuning(H, W)
    try:
        ctx.prnu_set_tuning(H, W, t["col_width"], t["pairs_per_block"], t["wave"], t["variant"], persistent)
        for P in (1, 2):
            want = ctx.eis_grid_search(R, hs[:P], g)
            bad = R.clone()
            bad[1, H // 2, 7] = np.nan
            got = ctx.eis_grid_search(bad, hs[:P], g)
            for f in (0, 2):
                assert got[f].tobytes() == want[f].tobytes()
            for r in got[1]:
                assert _no_peak(r) and r["cand_idx"] == 0
    finally:
        ctx.prnu_set_tuning(H, W, t["col_width"], t["pairs_per_block"], t["wave"], t["variant"], t["persistent"])
        for h in hs:
            ctx.prnu_fingerprint_release(h)


@pytest.mark.parametrize("loop", ["PRNU_LOOP_HOST", "PRNU_LOOP_DEVICE"])
@pytest.mark.parametrize("H,W", [(720, 1280), (480, 640)])
def test_served_beside_a_fingerprint_with_a_nan(prnu, H, W, loop):
    """Queries of a good and of a NaN fingerprint in shared waves."""
    g = synth.Grid(0.99, 0.005, 5, -0.5, 0.25, 5)
    frames = (128 + 20 * _images(H, W, 2)).clamp_(0, 255).to(torch.uint8)
    K = _images(H, W, 1, 6)[0]
    bad = K.clone()
    bad[1, 1] = np.nan
    with prnu.Context(0) as c:
        c.prnu_server_set_loop(getattr(prnu, loop))
        hs = [c.prnu_fingerprint_term(k) for k in (K, bad)]
        alone = c.query_poll(c.query_submit(frames, hs[:1], g), 2, 1, 60_000_000)
        ids = [(c.query_submit(frames, f, g), f) for f in (hs[1:], hs[:1], hs[::-1], hs[1:], hs[:1])]
        out = [c.query_poll(i, 2, len(f), 60_000_000) for i, f in ids]
    for res, (_, f) in zip(out, ids):
        for p, h in enumerate(f):
            for frame in range(2):
                r = res[frame, p]
                assert _no_peak(r) if h == hs[1] else r.tobytes() == alone[frame, 0].tobytes()


def test_correction_beside_a_frame_with_a_nan(ctx):
    R = _images(256, 256, 3)
    h = ctx.prnu_fingerprint_term(_images(256, 256, 1, 6)[0])
    want, n = ctx.eis_correction(R, [h], max_iter=2, th_half1=5)
    R[1, 100, 100] = np.inf
    got, m = ctx.eis_correction(R, [h], max_iter=2, th_half1=5)
    for f in (0, 2):
        assert got[f].tobytes() == want[f].tobytes() and m[f] == n[f]
    assert _no_peak(got[1, 0])
    ctx.prnu_fingerprint_release(h)
