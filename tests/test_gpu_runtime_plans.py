"""Frame sizes without compile-time plans: two-stage passes with runtime radices
(3 to 32, and 25 to 54 for heights), three stages for the wider rows, and the
ping-pong stages that take the other heights.

Each length stands for other radices as a height and as a width; the candidates
of a small grid (sample points on and outside the frame) are held to the FP64
oracle.  Bounds as for the planned sizes: FP32 1e-3 (sample points to 1e-4 px),
16-bit residuals 1e-2 and 3e-2."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
SIZES = [(16, 18), (18, 972), (20, 250), (24, 1350), (30, 1200), (54, 640), (50, 2304), (250, 486), (486, 54),
         (640, 30), (768, 60), (972, 32), (1000, 24), (1200, 20), (1250, 50), (1350, 36), (2304, 16), (64, 1250),
         (48, 1500), (2000, 40), (96, 96), (120, 1600), (1440, 128),
         (20, 1458), (18, 2000), (16, 2048), (18, 2430), (16, 2916), (18, 3456), (16, 3750), (20, 4000), (18, 4050),
         (16, 4096), (1458, 18), (1500, 16), (1536, 20), (1600, 18), (1944, 16), (2250, 16), (2400, 18), (2592, 16),
         (2916, 18), (3000, 16)]


@pytest.fixture(scope="module")
def ctx():
    import paper_2207_14507_gb300 as p
    p.build()
    c = p.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("H,W", SIZES)
def test_runtime_plans_match_the_oracle(ctx, H, W):
    import paper_2207_14507_gb300 as prnu
    rng = np.random.default_rng(H * 5000 + W)
    K = [synth.fingerprint_field(H, W, np.random.default_rng(s)) for s in (1, 2)]
    grid = synth.Grid(0.97, 0.03, 3, -1.0, 1.0, 3)
    R = (100 * np.roll(K[0], (3, -2), (0, 1)) + rng.standard_normal((H, W))).astype(np.float32)
    for dtype, store, tol in ((torch.float32, prnu.PRNU_F32, 1e-3), (torch.float16, prnu.PRNU_F16, 1e-2),
                              (torch.bfloat16, prnu.PRNU_F32, 3e-2)):
        dev = torch.from_numpy(R).to(DEV).to(dtype)[None].contiguous()
        hs = [ctx.prnu_fingerprint_term(torch.from_numpy(k).to(DEV), store) for k in K]
        ap = torch.empty((1, 2, grid.size), dtype=torch.float64, device=DEV)
        ctx.eis_grid_search(dev, hs, grid, all_pce=ap)
        got = ap.cpu().numpy()[0]
        _, ref = oracle.grid_search([dev[0].double().cpu().numpy()], [oracle.fingerprint_term(k) for k in K], grid)
        rel = np.abs(got / ref[0] - 1)
        assert rel.max() <= tol
        for h in hs:
            ctx.prnu_fingerprint_release(h)
    h = ctx.prnu_fingerprint_term(torch.from_numpy(K[0]).to(DEV))
    one = ctx.pce_score(torch.from_numpy(R).to(DEV), h)
    two = prnu.pce_score_noalloc(torch.from_numpy(R).to(DEV), torch.from_numpy(K[0]).to(DEV))
    ctx.prnu_fingerprint_release(h)
    assert (one["dy"], one["dx"]) == (two["dy"], two["dx"])
    assert abs(one["pce"] / two["pce"] - 1) <= 1e-4
