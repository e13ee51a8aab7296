"""Edges of the march's coordinate split and of its launch forms against the
FP64 oracle."""
import numpy as np
import pytest

import synth
from gpu_helpers import TOL_FP32, GPURenderer, compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rc():
    import paper_1211_5595_gb300 as m
    m.lib()
    return m


# A camera so far away that FP32 positions round to either side of the box:
# the clamped coordinates (weight 0 below the first voxel, 1 on the last cell)
# decide. The smallest volume has one cell; entries 2 is the smallest table.
@pytest.mark.parametrize("dims", [(2, 2, 2), (18, 17, 33)])
@pytest.mark.parametrize("distance", [40.0, 3.0e4, 1.0e6])
@pytest.mark.parametrize("entries", [2, 256])
@pytest.mark.parametrize("filt", [0, 1])
def test_positions_outside_the_box_clamp(rc, orc, dims, distance, entries, filt):
    nx, ny, nz = dims
    vol = (500 + 3000 * synth.uniform01(3, np.arange(nx * ny * nz))).astype(np.uint16).reshape(nz, ny, nx)
    tf = synth.noise_tf(entries, 11, alpha_max=0.2)
    c = [(n - 1) / 2.0 for n in dims]
    d = np.array([0.64, -0.6, 0.48])
    extent = max(2.0, float(max(dims)))
    cam = dict(eye=tuple(synth.f32(a + distance * b) for a, b in zip(c, d)), target=tuple(synth.f32(a) for a in c),
               up=(0.0, 0.0, 1.0), fovy_deg=synth.f32(max(2.0e-4, np.degrees(2 * np.arctan(extent / distance)))),
               width=40, height=28)
    r = GPURenderer(rc, vol, (1.0, 1.0, 1.0))
    try:
        r.set_tf(tf)
        img = r.render(cam, step_vox=0.5, term=0.99, shade=False, filter=filt)
        o = orc.render(orc.Scene(vol, (1.0, 1.0, 1.0), tf, cam, step=0.5, term=0.99, shade=False, filter=filt))
        assert o["rgba"][..., 3].max() > 0
        compare(img, o, TOL_FP32)
    finally:
        r.close()


# The launch form depends on the number of rays: one small view marches with
# several lanes per ray, a hundred copies of it with one. The images and the
# sample counts are the same. Ragged image sizes; a camera inside the box; a
# table whose opacities end rays after a few samples.
@pytest.mark.parametrize("storage", ["F32", "F16", "U16"])
@pytest.mark.parametrize("form", [dict(shade=False), dict(shade=True), dict(shade=True, filter=1), dict(shade=False, tf2=True)])
@pytest.mark.parametrize("size,views", [((37, 21), 1200), ((97, 75), 130), ((260, 201), 18)])
def test_lanes_per_ray_change_nothing(rc, storage, form, size, views):
    import torch
    form = dict(form)
    dims, spacing = (50, 41, 37), (1.0, 1.0, 1.5)
    ph = synth.head_phantom(dims, spacing, seed=5, tumor_radius_vox=3)
    r = GPURenderer(rc, ph.vol, spacing, getattr(rc, "RC_STORE_" + storage))
    try:
        w, h = size
        inside = dict(eye=(20.0, 18.0, 25.0), target=(40.0, 20.0, 30.0), up=(0.0, 0.0, 1.0), fovy_deg=50.0, width=w, height=h)
        tf2 = form.pop("tf2", False)
        for alpha, step in ((1.0, 0.5), (8.0, 0.3)):
            tab = synth.tf2d_table(64, 8) if tf2 else synth.tf_table(200)
            tab[..., 3] = np.minimum(1.0, tab[..., 3] * alpha)
            if tf2:
                rc.rc_tf2d_set(r.ctx, tab, 1200.0)
            else:
                r.set_tf(tab)
            for cam in (synth.orbit_camera(dims, spacing, 77.0, width=w, height=h), inside):
                P = dict(step_vox=step, term=0.95, **form)
                one, st = r.render(cam, stats=True, **P)
                many = torch.empty((views, h, w, 4), device="cuda")
                sm = rc.rc_render_views(r.ctx, r.vol, P, [cam] * views, many, stats=True)
                assert (many == torch.from_numpy(one).cuda()[None]).all()
                for key in ("dense_samples", "evaluated_samples", "rays_hit", "rays_total"):
                    assert sm[key] == views * st[key], key
                assert st["evaluated_samples"] > 0
    finally:
        r.close()


# Codes on both sides of the line where value+gradient entries take 8 bytes
# (vmax 32767 | 32768): every form that reads gradients, against the oracle.
@pytest.mark.parametrize("storage", ["F32", "U16"])
@pytest.mark.parametrize("vmax", [32767, 32768, 65535])
def test_gradient_forms_by_code_width(rc, orc, storage, vmax):
    import torch
    dims, spacing, gmax = (38, 33, 29), (1.0, 0.9, 1.3), 20000.0
    n = dims[0] * dims[1] * dims[2]
    u = synth.uniform01(5, np.arange(n)).reshape(dims[2], dims[1], dims[0])
    ph = synth.head_phantom(dims, spacing, seed=12, tumor_radius_vox=3).vol.astype(np.float64)
    vol = np.clip(ph * (vmax / 4095.0) + 0.02 * vmax * u, 0, vmax).astype(np.uint16)
    vol[10, 10, 8:20] = vmax                         # full-scale steps: the largest differences
    vol[10, 12, 8:20] = 0
    cam = synth.orbit_camera(dims, spacing, 140.0, width=61, height=45)
    r = GPURenderer(rc, vol, spacing, getattr(rc, "RC_STORE_" + storage), vmax)
    try:
        tab, tab2 = synth.tf_table(200, vmax=vmax), synth.tf2d_table(64, 8, gmax=gmax, vmax=vmax)
        for tf, kw in ((tab, dict(shade=True)), (tab2, dict(shade=False)), (tab2, dict(shade=True))):
            two = tf.ndim == 3
            if two:
                rc.rc_tf2d_set(r.ctx, tf, gmax)
            else:
                r.set_tf(tf)
            sc = orc.Scene(vol, spacing, tf, cam, step=0.5, term=0.99, vmax=vmax, gmax=gmax if two else None, **kw)
            o = orc.render(sc)
            compare(r.render(cam, step_vox=0.5, term=0.99, **kw), o, TOL_FP32)
            keep = np.nonzero(~o["tie"].reshape(-1))[0]
            g = np.zeros((61 * 45, 4))
            g[keep] = 1.0
            want, _ = orc.render_grad(sc, g[keep], pixels=keep)
            got = torch.empty(tf.shape, device="cuda")
            rc.rc_render_backward(r.ctx, r.vol, rc.RenderParams(step_vox=0.5, term=0.99, **kw),
                                  torch.from_numpy(g.astype(np.float32).reshape(45, 61, 4)).cuda(), got)
            torch.cuda.synchronize()
            assert np.abs(got.cpu().numpy() - want).max() / np.abs(want).max() < 2e-4
        r.set_tf(tab)
        img = r.render(cam, step_vox=0.5, term=0.99, shade=True, func=rc.RC_FUNC_ISO, iso=0.4 * vmax)
        o = orc.render(orc.Scene(vol, spacing, tab, cam, step=0.5, term=0.99, shade=True, vmax=vmax, func=orc.ISO,
                                 iso=0.4 * vmax))
        a, b = img.reshape(-1, 4).astype(np.float64), o["rgba"].reshape(-1, 4)
        same = (a[:, 3] == b[:, 3]) & (a[:, 2] == b[:, 2])
        assert same.mean() > 0.99 and b[:, 3].sum() > 100
        np.testing.assert_allclose(a[same][:, 1], b[same][:, 1], atol=2e-4)
        # the importance march over the whole chord reads the same entries
        out = torch.empty((1, 45, 61, 4), device="cuda")
        rc.rc_render_importance_views(r.ctx, r.vol, rc.RenderParams(step_vox=0.5, term=0.99, shade=True), [cam],
                                      rc.RC_SAMPLING_INVCDF, 1.0, None, None, 64, 2.0, out)
        torch.cuda.synchronize()
        assert torch.isfinite(out).all() and out[..., 3].max() > 0.2
    finally:
        r.close()


# Average and x-ray sums: a small launch (several lanes per ray) gives the sums
# of a large one (one lane per ray) bit for bit, and matches the oracle.
@pytest.mark.parametrize("storage", ["F32", "F16", "U16"])
@pytest.mark.parametrize("filt", [0, 1])
@pytest.mark.parametrize("size,views", [((37, 21), 1200), ((97, 75), 130), ((260, 201), 18)])
def test_sums_by_lanes(rc, orc, storage, filt, size, views):
    import torch
    dims, spacing = (50, 41, 37), (1.0, 1.0, 1.5)
    ph = synth.head_phantom(dims, spacing, seed=5, tumor_radius_vox=3)
    tf = synth.tf_table(64)
    r = GPURenderer(rc, ph.vol, spacing, getattr(rc, "RC_STORE_" + storage))
    try:
        r.set_tf(tf)
        w, h = size
        cam = synth.orbit_camera(dims, spacing, 77.0, width=w, height=h)
        for func, name in ((rc.RC_FUNC_AVERAGE, "AVERAGE"), (rc.RC_FUNC_XRAY, "XRAY")):
            P = dict(step_vox=0.4, func=func, filter=filt)
            one, st = r.render(cam, stats=True, **P)
            many = torch.empty((views, h, w, 4), device="cuda")
            sm = rc.rc_render_views(r.ctx, r.vol, P, [cam] * views, many, stats=True)
            assert (many == torch.from_numpy(one).cuda()[None]).all()
            assert sm["dense_samples"] == sm["evaluated_samples"] == views * st["dense_samples"] == views * st["evaluated_samples"]
            o = orc.render(orc.Scene(ph.vol, spacing, tf, cam, step=0.4, term=0.99, func=getattr(orc, name), filter=filt))
            np.testing.assert_allclose(one.reshape(-1, 4), o["rgba"].reshape(-1, 4), rtol=2e-5, atol=1e-5)
    finally:
        r.close()
