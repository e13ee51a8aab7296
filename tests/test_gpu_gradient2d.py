"""2-D table gradients whose contributions fill the fixed-point range (steady
dL/dI at its maximum, nearly opaque entries), over the forms of the shared-memory
accumulators: one slot per entry, a cache of tagged slots, and their edges."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
GMAX = 1500.0
DIMS, SPACING = (40, 33, 29), (1.0, 1.0, 1.5)


@pytest.fixture(scope="module")
def rc():
    import paper_1211_5595_gb300 as m
    m.lib()
    return m


# K + 4 columns of slots, M rows: the smallest table, one row below and one
# above the 10240 slots that fit, and tables that need the tagged cache
@pytest.mark.parametrize("K,M", [(2, 2), (64, 3), (252, 40), (253, 40), (512, 32), (1000, 9), (4096, 2)])
@pytest.mark.parametrize("sign", ["one", "mixed"])
@pytest.mark.parametrize("alpha", [0.05, 1.0])
def test_steady_gradient_matches_oracle(rc, orc, K, M, sign, alpha):
    import torch
    ph = synth.head_phantom(DIMS, SPACING, seed=9, tumor_radius_vox=3)
    W, H = 61, 45
    cam = synth.orbit_camera(DIMS, SPACING, 33.0, width=W, height=H)
    tab = synth.noise_tf(K * M, 21, alpha_max=alpha).reshape(M, K, 4)
    sc = orc.Scene(ph.vol, SPACING, tab, cam, step=0.5, term=0.99, gmax=GMAX)
    pix = np.arange(W * H)
    keep = pix[~orc.render(sc, pixels=pix)["tie"]]
    g = np.zeros((W * H, 4))
    g[keep] = 1.0 if sign == "one" else np.where(((keep // 7) % 2 == 0)[:, None], 1.0, -1.0)
    want, _ = orc.render_grad(sc, g[keep], pixels=keep)
    ctx = rc.rc_context_create(0)
    vol = rc.rc_volume_create(ctx, DIMS, SPACING, 4095, rc.RC_STORE_F32)
    try:
        rc.rc_volume_upload(ctx, vol, ph.vol)
        rc.rc_tf2d_set(ctx, tab, GMAX)
        rc.rc_camera_set(ctx, cam)
        gd = torch.from_numpy(g.astype(np.float32).reshape(H, W, 4)).cuda()
        p = rc.RenderParams(step_vox=0.5, term=0.99, shade=False, skip=True)
        got = torch.empty((M, K, 4), device="cuda")
        rc.rc_render_backward(ctx, vol, p, gd, got)
        # sixty views of it at once: many chunks per group of warps, and sums
        # beyond 32 bits in every word
        many = torch.empty_like(got)
        rc.rc_render_backward_views(ctx, vol, p, [cam] * 60, gd[None].expand(60, H, W, 4).contiguous(), many)
        again = torch.empty_like(got)
        rc.rc_render_backward_views(ctx, vol, p, [cam] * 60, gd[None].expand(60, H, W, 4).contiguous(), again)
        rc.rc_context_sync(ctx)
        assert torch.equal(many, again)
        scale = np.abs(want).max()
        assert scale > 0
        assert np.abs(got.cpu().numpy() - want).max() / scale < 2e-4
        assert np.abs(many.cpu().numpy() - 60.0 * want).max() / (60.0 * scale) < 2e-4
    finally:
        torch.cuda.synchronize()
        rc.rc_volume_destroy(ctx, vol)
        rc.rc_context_destroy(ctx)
