"""Device buffers that the kernels access 16 bytes at a time are refused on the
host when their address is not a multiple of 16; nothing is launched."""
import pytest

import synth

pytestmark = pytest.mark.gpu
DIMS, SPACING, W, H = (40, 33, 29), (1.0, 1.0, 1.5), 20, 12


@pytest.fixture(scope="module")
def rc():
    import paper_1211_5595_gb300 as m
    m.lib()
    return m


@pytest.fixture()
def scene(rc):
    import torch
    ph = synth.head_phantom(DIMS, SPACING, seed=9, tumor_radius_vox=3)
    ctx = rc.rc_context_create(0)
    vol = rc.rc_volume_create(ctx, DIMS, SPACING, 4095, rc.RC_STORE_F32)
    rc.rc_volume_upload(ctx, vol, ph.vol)
    rc.rc_tf_set(ctx, synth.tf_table(64))
    cam = synth.orbit_camera(DIMS, SPACING, 33.0, width=W, height=H)
    rc.rc_camera_set(ctx, cam)
    rc.rc_proposal_load(ctx, rc.pack_proposal_blob(synth.proposal_init_params(3)))
    yield ctx, vol, cam
    torch.cuda.synchronize()
    rc.rc_volume_destroy(ctx, vol)
    rc.rc_context_destroy(ctx)


@pytest.mark.parametrize("off", [1, 2, 3])
def test_misaligned_buffers_are_refused(rc, scene, off):
    import torch
    ctx, vol, cam = scene
    p = rc.RenderParams(step_vox=0.5, term=0.99, shade=False)
    n = H * W
    flat = torch.zeros(n * 112 + 8, device="cuda")
    bad = flat[off:]
    img = torch.full((1, H, W, 4), 7.0, device="cuda")
    dtf = torch.full((64, 4), 7.0, device="cuda")
    out = torch.full((n, 33), 7.0, device="cuda")
    grad = torch.full((rc.RC_PROPOSAL_PARAMS,), 7.0, device="cuda")
    pdf, that = torch.full((1, H, W, 32), 1 / 32, device="cuda"), torch.zeros((1, H, W), device="cuda")
    assert bad.data_ptr() % 16 == 4 * off
    calls = [lambda: rc.rc_render(ctx, vol, p, bad),
             lambda: rc.rc_render_views(ctx, vol, p, [cam], bad),
             lambda: rc.rc_render_batch(ctx, [vol], p, [cam], bad),
             lambda: rc.rc_render_backward(ctx, vol, p, bad, dtf),
             lambda: rc.rc_render_backward_noalloc(ctx, vol, p, bad, dtf),
             lambda: rc.rc_render_backward_views(ctx, vol, p, [cam], bad, dtf),
             lambda: rc.rc_render_backward_views_with_forward(ctx, vol, p, [cam], bad, img, dtf),
             lambda: rc.rc_render_backward_views_with_forward(ctx, vol, p, [cam], img, bad, dtf),
             lambda: rc.rc_render_importance(ctx, vol, p, pdf, that, 16, 2.0, bad),
             lambda: rc.rc_render_importance_views(ctx, vol, p, [cam], rc.RC_SAMPLING_RANGE, 0.0, pdf, that, 16, 2.0, bad),
             lambda: rc.rc_render_proposal(ctx, vol, p, 16, 2.0, bad),
             lambda: rc.rc_render_proposal_views(ctx, vol, p, [cam], 16, 2.0, bad),
             lambda: rc.rc_render_proposal_sampled(ctx, vol, p, [cam], rc.RC_SAMPLING_INVCDF, 0.5, 16, 2.0, bad),
             lambda: rc.rc_proposal_forward(ctx, bad, n, out),
             lambda: rc.rc_proposal_grad(ctx, bad, out, n, grad),
             lambda: rc.rc_proposal_train_step(ctx, bad, out, n, 1e-3)]
    for i, call in enumerate(calls):
        with pytest.raises(rc.RCError) as e:
            call()
        assert e.value.status == rc.RC_ERR_INVALID_ARG and "16-byte aligned" in str(e.value), i
    rc.rc_context_sync(ctx)
    assert (flat == 0).all() and (dtf == 7).all() and (out == 7).all() and (grad == 7).all()
    # buffers read and written by words keep their 4-byte alignment
    rc.rc_proposal_features(ctx, vol, p, flat[off:])
    rc.rc_profiles_generate(ctx, vol, p, flat[off:])
    feat = torch.zeros((n, 112), device="cuda")
    rc.rc_proposal_forward(ctx, feat, n, flat[off:])
    rc.rc_proposal_grad(ctx, feat, flat[off:], n, torch.zeros(rc.RC_PROPOSAL_PARAMS + off, device="cuda")[off:])
    host = torch.zeros(n * 4 + off)
    rc.rc_render_views_host(ctx, vol, p, [cam], host[off:])
    rc.rc_context_sync(ctx)
    assert host[off:].abs().max() > 0


def test_autograd_takes_a_gradient_at_any_offset(rc, scene):
    """The gradient of a concatenation is a view at the image's place in it."""
    import torch

    from paper_1211_5595_gb300.autograd import render_tf
    ctx, vol, cam = scene
    p = rc.RenderParams(step_vox=0.5, term=0.99, shade=False)
    w = torch.linspace(-1.0, 1.0, W * H * 4, device="cuda")
    grads = []
    for lead in (0, 3):
        tf = torch.tensor(synth.tf_table(64), dtype=torch.float32, device="cuda").requires_grad_()
        img = render_tf(tf, ctx, vol, p, cam)
        whole = torch.cat([torch.zeros(lead, device="cuda"), img.flatten()])
        (whole * torch.cat([torch.zeros(lead, device="cuda"), w])).sum().backward()
        grads.append(tf.grad)
    assert grads[0].abs().max() > 0
    assert torch.equal(grads[0], grads[1])
