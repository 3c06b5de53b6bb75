"""prnu_tuning: what is reported is accepted, every row plan and the autotuner's
choice can be set, and the plan changes no bit of a result."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DEV = "cuda:0"
# row pairs per block with planned kernels, the default first
PLANS = {(256, 256): (8, 4), (720, 1280): (2, 4), (1080, 1920): (1, 2), (2160, 3840): (1, 2)}


@pytest.fixture(scope="module")
def prnu():
    import paper_2207_14507_gb300 as p
    p.build()
    return p


def _set(ctx, H, W, t, **kw):
    t = dict(t, **kw)
    ctx.prnu_set_tuning(H, W, t["col_width"], t["pairs_per_block"], t["wave"], t["variant"], t["persistent"],
                        t["streams"], t["share_forward"])


@pytest.mark.parametrize("H,W", sorted(PLANS))
def test_every_row_plan_can_be_set(prnu, H, W):
    wl = synth.make_workload(2, H=H, W=W, F=1, on_grid=True, s_max=8)
    win = synth.snap_windows(wl.grid, wl.planted[:, :2], np.array([1]))
    with prnu.Context(0) as ctx:
        R = torch.empty(wl.frames.shape, dtype=torch.float32, device=DEV)
        ctx.prnu_residual(torch.from_numpy(wl.frames).to(DEV), R)
        h = ctx.prnu_fingerprint_term(torch.from_numpy(wl.fingerprints[0]).to(DEV))
        t = ctx.prnu_get_tuning(H, W)
        assert t["pairs_per_block"] == PLANS[(H, W)][0]
        assert t["variant"] == 0   # the binding's default argument
        _set(ctx, H, W, t)
        out = []
        for ppb in sorted({*PLANS[(H, W)], 1, 2}):   # 1 and 2 were always taken
            _set(ctx, H, W, t, pairs_per_block=ppb)
            assert ctx.prnu_get_tuning(H, W)["pairs_per_block"] == ppb
            ap = torch.empty((1, 1, wl.grid.size), dtype=torch.float64, device=DEV)
            ctx.eis_grid_search(R, [h], wl.grid, windows=win, all_pce=ap)
            out.append(ap.cpu().numpy())
        for o in out[1:]:
            np.testing.assert_array_equal(o, out[0])
        for ppb in (0, -1, 3, 16):
            with pytest.raises(prnu.PrnuError) as e:
                _set(ctx, H, W, t, pairs_per_block=ppb)
            assert e.value.code == prnu.PRNU_EINVAL


@pytest.mark.parametrize("H,W", [(256, 256), (720, 1280), (480, 640)])
def test_the_autotuned_choice_can_be_set(prnu, H, W):
    with prnu.Context(0) as ctx:
        best = ctx.prnu_autotune(H, W, budget_ms=300.0)
        _set(ctx, H, W, best)
        assert ctx.prnu_get_tuning(H, W) == best


@pytest.mark.parametrize("H,W", [(16, 4096), (480, 640), (1440, 2560)])
def test_sizes_without_plans_take_1_2_and_4(prnu, H, W):
    with prnu.Context(0) as ctx:
        t = ctx.prnu_get_tuning(H, W)
        for ppb in (t["pairs_per_block"], 1, 2, 4):
            _set(ctx, H, W, t, pairs_per_block=ppb)
        with pytest.raises(prnu.PrnuError):
            _set(ctx, H, W, t, pairs_per_block=8)
