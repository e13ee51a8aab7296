"""Table gradients at the ends of dL/dI's range: all zero, and so small that
2^32 / max|dL/dI| is past FP32's largest number."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
DIMS, SPACING = (96, 80, 64), (1.0, 1.0, 1.0)


@pytest.fixture(scope="module")
def rc():
    import paper_1211_5595_gb300 as m
    m.lib()
    return m


def _time(torch, fn):
    ts = []
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        fn()
        b.record()
        b.synchronize()
        ts.append(a.elapsed_time(b))
    return sorted(ts)[3]


# 1-D tables with per-warp and with per-CTA accumulators, 2-D tables with a slot
# per entry and with the tagged cache
@pytest.mark.parametrize("K,M", [(64, 0), (1000, 0), (64, 16), (1000, 32)])
@pytest.mark.parametrize("given", [True, False])
def test_zero_and_tiny_gradients(rc, K, M, given):
    import torch
    ph = synth.head_phantom(DIMS, SPACING, seed=9, tumor_radius_vox=3)
    cams = [synth.orbit_camera(DIMS, SPACING, a, width=256, height=192) for a in (33.0, 200.0)]
    ctx = rc.rc_context_create(0)
    vol = rc.rc_volume_create(ctx, DIMS, SPACING, 4095, rc.RC_STORE_F32)
    try:
        rc.rc_volume_upload(ctx, vol, ph.vol)
        if M:
            rc.rc_tf2d_set(ctx, synth.tf2d_table(K, M, gmax=1500.0), 1500.0)
        else:
            rc.rc_tf_set(ctx, synth.tf_table(K))
        p = rc.RenderParams(step_vox=0.5, term=0.99, shade=False, skip=True)
        images = torch.empty((2, 192, 256, 4), device="cuda")
        rc.rc_render_views(ctx, vol, p, cams, images)

        def gradient(d):
            t = torch.empty((M, K, 4) if M else (K, 4), device="cuda")
            if given:
                call = lambda: rc.rc_render_backward_views_with_forward(ctx, vol, p, cams, images, d, t)  # noqa: E731
            else:
                call = lambda: rc.rc_render_backward_views(ctx, vol, p, cams, d, t)  # noqa: E731
            ms = _time(torch, call)
            rc.rc_context_sync(ctx)
            return t, ms

        ones = torch.ones_like(images)
        want, ms_ones = gradient(ones)
        top = float(want.abs().max())
        assert np.isfinite(top) and top > 3.0
        # nothing to march: exact zeros, in a fraction of the time
        zero, ms_zero = gradient(torch.zeros_like(images))
        assert (zero == 0).all()
        assert ms_zero < 0.5 * ms_ones, (ms_zero, ms_ones)
        # one pixel of all: its own rays only
        one = torch.zeros_like(images)
        one[0, 96, 128] = 1.0
        g, ms_one = gradient(one)
        assert torch.isfinite(g).all() and g.abs().max() > 0
        # linear in dL/dI. At 1e-30 a unit of the fixed point is 1 / 3.3e8 of the
        # gradient; at most 98304 rays x 250 samples / 8 per group of lanes round
        # by half a unit each: 4.7e-3 of 1e-30, less than 2e-3 of the largest entry
        tiny, _ = gradient(ones * 1e-30)
        err = float((tiny.double() * 1e30 - want.double()).abs().max())
        assert err < 2e-3 * top, (err, top)
    finally:
        torch.cuda.synchronize()
        rc.rc_volume_destroy(ctx, vol)
        rc.rc_context_destroy(ctx)
