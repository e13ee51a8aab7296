"""MIP, isosurface and threshold renders that jump over blocks by their maxima
give the images of the march that evaluates every sample, bit for bit."""
import numpy as np
import pytest

import synth
from gpu_helpers import GPURenderer

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rc():
    import paper_1211_5595_gb300 as m
    m.lib()
    return m


def _volume(kind, dims, vmax):
    nx, ny, nz = dims
    if kind == "phantom":
        v = synth.head_phantom(dims, (1.0, 1.0, 1.5), seed=5, tumor_radius_vox=3).vol.astype(np.int64)
        return np.clip(v * vmax // 4095, 0, vmax).astype(np.uint16)
    u = synth.uniform01(17, np.arange(nx * ny * nz)).reshape(nz, ny, nx)
    if kind == "sparse":                       # mostly zero with isolated full-scale voxels
        return np.where(u > 0.995, vmax, np.where(u > 0.6, u * 0.1 * vmax, 0)).astype(np.uint16)
    return (u * vmax).astype(np.uint16)        # noise: neighbouring blocks of nearly equal maxima


# the smallest volume, a block border (17 and 33 voxels), ragged sizes
@pytest.mark.parametrize("dims", [(2, 2, 2), (17, 33, 5), (50, 41, 37)])
@pytest.mark.parametrize("kind", ["phantom", "sparse", "noise"])
@pytest.mark.parametrize("storage,vmax", [("F32", 4095), ("U16", 65535), ("F16", 4095), ("F16", 65535)])
def test_block_maxima_skip_is_exact(rc, dims, kind, storage, vmax):
    if kind == "phantom" and min(dims) < 5:
        pytest.skip("no room for a phantom")
    vol = _volume(kind, dims, vmax)
    r = GPURenderer(rc, vol, (1.0, 1.0, 1.5), getattr(rc, "RC_STORE_" + storage), vmax)
    try:
        r.set_tf(synth.tf_table(200, vmax=vmax))
        cam = synth.orbit_camera(dims, (1.0, 1.0, 1.5), 77.0, width=61, height=45)
        hits = 0
        for filt in (0, 1):
            for func in ("MIP", "ISO", "THRESHOLD"):
                for iso in (0.0, 0.3 * vmax, 0.72 * vmax, float(vmax)) if func != "MIP" else (0.0,):
                    P = dict(step_vox=0.4, func=getattr(rc, "RC_FUNC_" + func), iso=iso, filter=filt)
                    on, st = r.render(cam, stats=True, skip=True, **P)
                    off, so = r.render(cam, stats=True, skip=False, **P)
                    assert np.array_equal(on, off), (filt, func, iso, np.abs(on - off).max())
                    assert st["dense_samples"] == so["dense_samples"] == so["evaluated_samples"]
                    assert st["evaluated_samples"] <= so["evaluated_samples"]
                    hits += int(on[..., 3].sum())
        assert hits > 0
    finally:
        r.close()
