"""The time of a set of views does not depend on which of them comes first: the
form of a launch is chosen by all of its views."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rc():
    import paper_1211_5595_gb300 as m
    m.lib()
    return m


# the first view looks past the volume, or stands far away
@pytest.mark.parametrize("eye,target", [((650.0, 80.0, 60.0), (300.0, 700.0, 60.0)), ((7000.0, 80.0, 60.0), (80.0, 80.0, 60.0))])
@pytest.mark.parametrize("form", [dict(shade=False), dict(shade=True)])
def test_view_order_does_not_change_the_time(rc, eye, target, form):
    import torch
    dims, spacing, n, w = (160, 160, 120), (1.0, 1.0, 1.0), 8, 768
    ph = synth.head_phantom(dims, spacing, seed=5, tumor_radius_vox=5)
    ctx = rc.rc_context_create(0)
    vol = rc.rc_volume_create(ctx, dims, spacing, 4095, rc.RC_STORE_F32)
    try:
        rc.rc_volume_upload(ctx, vol, ph.vol)
        rc.rc_tf_set(ctx, synth.tf_table(256))
        odd = rc.make_camera(dict(eye=eye, target=target, up=(0.0, 0.0, 1.0), fovy_deg=30.0, width=w, height=w))
        views = [rc.make_camera(synth.orbit_camera(dims, spacing, 45.0 * i, width=w, height=w)) for i in range(n)]
        p = rc.RenderParams(step_vox=0.5, term=0.99, **form)
        images, ms = [], []
        for order in ([odd] + views, views + [odd]):
            out = torch.empty((n + 1, w, w, 4), device="cuda")
            ts = []
            for _ in range(9):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                rc.rc_render_views(ctx, vol, p, order, out)
                b.record()
                b.synchronize()
                ts.append(a.elapsed_time(b))
            ms.append(sorted(ts)[4])
            images.append(out)
        assert torch.equal(images[0][1:], images[1][:-1]) and torch.equal(images[0][0], images[1][-1])
        assert ms[0] < 1.25 * ms[1], ms
    finally:
        torch.cuda.synchronize()
        rc.rc_volume_destroy(ctx, vol)
        rc.rc_context_destroy(ctx)
