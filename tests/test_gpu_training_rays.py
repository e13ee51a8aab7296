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


# Edges of the training kernel's tiles and groups: one ray, a tile and its
# neighbours, one CTA per tile up to one per SM and around it (152 tiles), and
# two groups per CTA with an odd tile left over.
@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128, 152 * 128 + 1, 303 * 128 + 5, 305 * 128])
def test_training_gradient_sizes(rc, n):
    import torch
    import oracle.mlp as mlp
    p = synth.proposal_init_params(7)
    f, y = synth.proposal_batch(31, n)
    ctx = rc.rc_context_create(0)
    try:
        rc.rc_proposal_load(ctx, rc.pack_proposal_blob(p))
        fd, yd = torch.from_numpy(f).cuda(), torch.from_numpy(y).cuda()
        grad, loss = torch.empty(18152, device="cuda"), torch.empty(1, device="cuda")
        rc.rc_proposal_grad(ctx, fd, yd, n, grad, loss)
        again = torch.empty_like(grad)
        rc.rc_proposal_grad(ctx, fd, yd, n, again)
        rc.rc_context_sync(ctx)
        assert torch.equal(grad, again)
        wloss, want = mlp.loss_and_grad(p, f, y)
        assert np.abs(grad.cpu().numpy() - want).max() / np.abs(want).max() < 1e-2
        assert abs(float(loss) - wloss) / abs(wloss) < 1e-3
        # a training step from the same state makes Adam's first step of that gradient
        rc.rc_proposal_train_step(ctx, fd, yd, n, 1e-3, loss)
        s = rc.unpack_proposal_blob(rc.rc_proposal_save(ctx))
        g = grad.cpu().numpy().astype(np.float64)
        np.testing.assert_allclose(s["m"], 0.1 * g, rtol=1e-5, atol=1e-12)
        np.testing.assert_allclose(s["v"], 0.001 * g * g, rtol=1e-4, atol=1e-18)
        step = 1e-3 * g / (np.abs(g) + 1e-8)
        np.testing.assert_allclose(s["params"], p - step, rtol=0, atol=2e-6)
        # and the next forward uses the stepped weights
        out = torch.empty((min(n, 300), 33), device="cuda")
        rc.rc_proposal_forward(ctx, fd, min(n, 300), out)
        rc.rc_context_sync(ctx)
        o = mlp.forward(s["params"], f[:300])
        assert np.abs(out.cpu().numpy()[:, :32] - o["pdf"]).max() < 2e-3
    finally:
        torch.cuda.synchronize()
        rc.rc_context_destroy(ctx)
