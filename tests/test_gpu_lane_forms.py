"""Every number of lanes per ray gives the images and the sample counts of one
lane, bit for bit. The launch sizes are chosen on both sides of the rules' lines,
and the rules themselves say which form each launch takes."""
import pytest

import synth
from gpu_helpers import GPURenderer
from launch_rules import camera_view, compile_rules, launch_size

pytestmark = pytest.mark.gpu
DIMS, SPACING = (50, 41, 37), (1.0, 1.0, 1.5)


@pytest.fixture(scope="module")
def rc():
    import paper_1211_5595_gb300 as m
    m.lib()
    return m


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    return compile_rules(tmp_path_factory.mktemp("rules"))


def _views(rc, r, P, cam, n):
    import torch
    out = torch.empty((n, cam["height"], cam["width"], 4), device="cuda")
    st = rc.rc_render_views(r.ctx, r.vol, P, [cam] * n, out, stats=True)
    return out, {k: st[k] for k in ("dense_samples", "evaluated_samples", "rays_hit", "rays_total")}


def _compare(rc, r, P, cam, launches):
    """launches: (lanes, views); the last one, of one lane, is what the others have to equal."""
    want, ws = _views(rc, r, P, cam, launches[-1][1])
    assert (want == want[0]).all() and want[..., 3].max() > 0
    for lanes, n in launches[:-1]:
        got, gs = _views(rc, r, P, cam, n)
        assert (got == want[0]).all(), lanes
        for key in ws:
            assert gs[key] * launches[-1][1] == ws[key] * n, (lanes, key)


@pytest.mark.parametrize("storage,vmax", [("F32", 4095), ("F16", 4095), ("U16", 4095), ("F32", 40000), ("U16", 65535)])
@pytest.mark.parametrize("form", [dict(shade=False), dict(shade=True), dict(shade=True, filter=1),
                                  dict(shade=False, tf2=True), dict(shade=False, tf2=True, filter=1)])
def test_compositing(rc, rules, storage, vmax, form):
    form = dict(form)
    heavy = (form["shade"] and vmax >= 32768) or "tf2" in form or "filter" in form
    cam = synth.orbit_camera(DIMS, SPACING, 77.0, width=97, height=75)
    launches = [(8, 1), (4, 20), (2, 60), (1, 100)]
    for lanes, n in launches:
        hits, steps, _ = launch_size(rules, DIMS, SPACING, 0.1, [camera_view(cam, SPACING)] * n)
        assert rules.lanes_per_ray(hits, steps, int(heavy)) == lanes
    v = synth.head_phantom(DIMS, SPACING, seed=5, tumor_radius_vox=3).vol.astype("float64") * (vmax / 4095.0)
    r = GPURenderer(rc, v.astype("uint16"), SPACING, getattr(rc, "RC_STORE_" + storage), vmax)
    try:
        if form.pop("tf2", False):
            gmax = 1200.0 * vmax / 4095
            rc.rc_tf2d_set(r.ctx, synth.tf2d_table(64, 8, gmax=gmax, vmax=vmax), gmax)
        else:
            r.set_tf(synth.tf_table(200, vmax=vmax))
        for skip in (True, False):
            _compare(rc, r, dict(step_vox=0.1, term=0.95, skip=skip, **form), cam, launches)
    finally:
        r.close()


@pytest.mark.parametrize("storage", ["F32", "F16", "U16"])
@pytest.mark.parametrize("filt", [0, 1])
@pytest.mark.parametrize("func", ["AVERAGE", "XRAY", "MIP"])
def test_sums_and_maxima(rc, rules, storage, filt, func):
    cam = synth.orbit_camera(DIMS, SPACING, 77.0, width=260, height=201)
    launches = [(4, 1), (2, 7), (1, 24)]
    rule = rules.lanes_per_max if func == "MIP" else rules.lanes_per_sum
    for lanes, n in launches:
        assert rule(*launch_size(rules, DIMS, SPACING, 1.0, [camera_view(cam, SPACING)] * n), filt) == lanes
    r = GPURenderer(rc, synth.head_phantom(DIMS, SPACING, seed=5, tumor_radius_vox=3).vol, SPACING,
                    getattr(rc, "RC_STORE_" + storage))
    try:
        r.set_tf(synth.tf_table(64))
        _compare(rc, r, dict(step_vox=1.0, func=getattr(rc, "RC_FUNC_" + func), filter=filt), cam, launches)
    finally:
        r.close()
