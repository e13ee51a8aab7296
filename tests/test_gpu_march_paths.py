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
