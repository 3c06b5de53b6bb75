"""Every column-pass variant of a planned frame size gives the same bits.

The variants differ in the columns per block, the resident blocks and how the
strips move; the transform (two stages of 16 to 48 points, one column per
thread) is the same, so each candidate's PCE must agree bit for bit, with FP32
and FP16 fingerprints, one of them and two that each run their own forward
pass through the variant.  Two that share a forward pass take the split
kernels whatever the variant, once.  With FP32 fingerprints a variant that
holds FP16 bins only is replaced and is skipped.  The first variant is held to
the oracle at the planted node and its neighbours."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"


# column variants of a size, and those for FP16 fingerprints only
VARIANTS = {(256, 256): (3, ()), (720, 1280): (6, (0,)), (1080, 1920): (6, (0,)), (2160, 3840): (4, (1,))}


@pytest.mark.parametrize("half", [False, True], ids=["f32", "f16"])
@pytest.mark.parametrize("H,W", sorted(VARIANTS))
def test_every_column_variant_gives_the_same_bits(H, W, half):
    import paper_2207_14507_gb300 as prnu
    prnu.build()
    wl = synth.make_workload(2, H=H, W=W, F=1, on_grid=True, s_max=8)
    win = synth.snap_windows(wl.grid, wl.planted[:, :2], np.array([1]))
    fps = [wl.fingerprints[0], synth.fingerprint_field(H, W, np.random.default_rng(5))]
    store = prnu.PRNU_F16 if half else prnu.PRNU_F32
    with prnu.Context(0) as ctx:
        R = torch.empty(wl.frames.shape, dtype=torch.float32, device=DEV)
        ctx.prnu_residual(torch.from_numpy(wl.frames).to(DEV), R)
        hs = [ctx.prnu_fingerprint_term(torch.from_numpy(K).to(DEV), store) for K in fps]
        t = ctx.prnu_get_tuning(H, W)
        n, half_only = VARIANTS[(H, W)]
        runs = [(v, P, 0) for v in range(n) if half or v not in half_only for P in (1, 2)] + [(0, 2, 1)]
        seen = {}
        for v, P, share in runs:
            ctx.prnu_set_tuning(H, W, t["col_width"], t["pairs_per_block"], t["wave"], v, 0, 1, share)
            ap = torch.empty((1, P, wl.grid.size), dtype=torch.float64, device=DEV)
            ctx.eis_grid_search(R, hs[:P], wl.grid, windows=win, all_pce=ap)
            seen[(v, P, share)] = ap.cpu().numpy()
        with pytest.raises(prnu.PrnuError):
            ctx.prnu_set_tuning(H, W, t["col_width"], t["pairs_per_block"], t["wave"], n)
    first = next(v for v, _, _ in runs)   # both fingerprints through its own kernel
    for key, pce in seen.items():
        np.testing.assert_array_equal(pce[0], seen[(first, 2, 0)][0, :key[1]], err_msg=str(key))
    _, ref = oracle.grid_search([oracle.prnu_residual(wl.frames[0])[0]], [oracle.fingerprint_term(fps[0])], wl.grid,
                                windows=win)
    got, mask = seen[(first, 1, 0)][0, 0], ~np.isnan(ref[0, 0])
    # FP32: sample points to 1e-4 px; FP16 spectra: one rounding of 2^-11 per bin
    assert np.max(np.abs(got[mask] / ref[0, 0][mask] - 1)) <= (1e-2 if half else 1e-3)
