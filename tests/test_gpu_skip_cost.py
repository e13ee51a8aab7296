"""Skipping by block maxima may not cost: a render with skip=1 takes no longer
than one that evaluates every sample."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rc():
    import paper_1211_5595_gb300 as m
    m.lib()
    return m


def _time(torch, fn):
    ts = []
    for _ in range(15):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(4):
            fn()
        b.record()
        b.synchronize()
        ts.append(a.elapsed_time(b))
    return sorted(ts)[4]


# small views and noise, where the maxima of neighbouring blocks are alike
@pytest.mark.parametrize("kind", ["phantom", "noise", "constant"])
@pytest.mark.parametrize("size", [128, 512])
@pytest.mark.parametrize("filt", [0, 1])
def test_mip_with_skip_costs_no_more(rc, kind, size, filt):
    import torch
    dims, spacing = (128, 128, 96), (1.0, 1.0, 1.0)
    if kind == "phantom":
        v = synth.head_phantom(dims, spacing, seed=5, tumor_radius_vox=5).vol
    else:
        u = synth.uniform01(17, np.arange(int(np.prod(dims)))).reshape(dims[::-1])
        v = (u * 4095 if kind == "noise" else np.full(dims[::-1], 2000.0)).astype(np.uint16)
    ctx = rc.rc_context_create(0)
    vol = rc.rc_volume_create(ctx, dims, spacing, 4095, rc.RC_STORE_F32)
    try:
        rc.rc_volume_upload(ctx, vol, v)
        rc.rc_tf_set(ctx, synth.tf_table(64))
        rc.rc_camera_set(ctx, synth.orbit_camera(dims, spacing, 77.0, width=size, height=size))
        images, ms = [], []
        for skip in (True, False):
            p = rc.RenderParams(step_vox=0.5, func=rc.RC_FUNC_MIP, skip=skip, filter=filt)
            out = torch.empty((size, size, 4), device="cuda")
            ms.append(_time(torch, lambda: rc.rc_render(ctx, vol, p, out)))
            images.append(out)
        assert torch.equal(*images) and images[0].max() > 0.1
        assert ms[0] < 1.1 * ms[1], ms
    finally:
        torch.cuda.synchronize()
        rc.rc_volume_destroy(ctx, vol)
        rc.rc_context_destroy(ctx)
