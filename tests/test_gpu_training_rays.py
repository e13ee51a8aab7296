"""Edges of the training-ray kernels: profiles with and without empty-space
skipping, ragged and single-pixel images, large tables, unaligned outputs."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu
DIMS, SPACING = (50, 41, 37), (1.0, 1.0, 1.5)


@pytest.fixture(scope="module")
def rc():
    import paper_1211_5595_gb300 as m
    m.lib()
    return m


# 2815 and 3072 entries: the table and the staged rows pass 48 KB together
@pytest.mark.parametrize("size,entries", [((1, 1), 256), ((7, 3), 2), ((66, 45), 256), ((33, 18), 2815), ((33, 18), 3072),
                                          ((33, 18), 4096)])
@pytest.mark.parametrize("storage", ["F32", "F16", "U16"])
def test_profiles_and_features(rc, orc, size, entries, storage):
    import torch
    w, h = size
    ph = synth.head_phantom(DIMS, SPACING, seed=5, tumor_radius_vox=3)
    cam = synth.orbit_camera(DIMS, SPACING, 77.0, width=w, height=h)
    tf = synth.tf_table(entries)
    ctx = rc.rc_context_create(0)
    vol = rc.rc_volume_create(ctx, DIMS, SPACING, 4095, getattr(rc, "RC_STORE_" + storage))
    try:
        rc.rc_volume_upload(ctx, vol, ph.vol)
        rc.rc_tf_set(ctx, tf)
        rc.rc_camera_set(ctx, cam)
        got = {}
        for skip in (True, False):
            p = rc.RenderParams(step_vox=0.5, term=0.99, skip=skip)
            y = torch.full((h * w * 33 + 7,), -1.0, device="cuda")
            rc.rc_profiles_generate(ctx, vol, p, y)
            f = torch.full((h * w * 112 + 7,), -1.0, device="cuda")
            rc.rc_proposal_features(ctx, vol, p, f)
            g = torch.full((h * w * 112 + 8,), -1.0, device="cuda")
            rc.rc_proposal_features(ctx, vol, p, g[1:])             # 4-byte aligned
            rc.rc_context_sync(ctx)
            assert (y[h * w * 33:] == -1).all() and (f[h * w * 112:] == -1).all() and (g[1 + h * w * 112:] == -1).all()
            assert torch.equal(f[:h * w * 112], g[1:1 + h * w * 112])
            got[skip] = y[:h * w * 33].reshape(h * w, 33).cpu().numpy()
        assert np.array_equal(got[True], got[False])
        bins, tfin = orc.profiles(orc.Scene(ph.vol, SPACING, tf, cam))
        np.testing.assert_allclose(got[True][:, :32], bins, atol=2e-4)
        np.testing.assert_allclose(got[True][:, 32], tfin, atol=2e-4)
    finally:
        torch.cuda.synchronize()
        rc.rc_volume_destroy(ctx, vol)
        rc.rc_context_destroy(ctx)
