"""The host-side rules of csrc/rc_rules.h compiled by themselves, for the tests
that call them or need to know which form a launch takes."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1211_5595_gb300", "csrc")
SHIM = r"""
#include "rc_rules.h"
extern "C" {
int persistent_ctas(int chunks, int sms) { return rc::persistent_ctas(chunks, sms); }
// rays and samples of `n` views (records of 16 doubles: eye, basis, tangents, size)
void launch_size(const int *dims, const double *spacing, double step, const double *views, int n, double *out) {
    rc::BoxGeom b;
    for (int i = 0; i < 3; i++) { b.n[i] = dims[i]; b.s[i] = spacing[i]; }
    rc::LaunchSizer z(b, step);
    for (int i = 0; i < n; i += rc::sized_stride(n)) {
        const double *q = views + 16 * i;
        rc::ViewGeom c;
        for (int a = 0; a < 3; a++) { c.o[a] = q[a]; c.f[a] = q[3 + a]; c.r[a] = q[6 + a]; c.u[a] = q[9 + a]; }
        c.tx = q[12]; c.ty = q[13]; c.W = (int)q[14]; c.H = (int)q[15];
        z.add(c);
    }
    const rc::LaunchSize s = z.size(n);
    out[0] = s.hits;
    out[1] = s.steps;
    out[2] = s.density;
}
int lanes_per_ray(double hits, double steps, int heavy) {
    rc::LaunchSize z;
    z.hits = hits;
    z.steps = steps;
    return rc::lanes_per_ray(z, heavy != 0);
}
int lanes_per_sum(double hits, double steps, double density, int cubic) {
    rc::LaunchSize z;
    z.hits = hits;
    z.steps = steps;
    z.density = density;
    return rc::lanes_per_sum(z, cubic != 0);
}
int lanes_per_max(double hits, double steps, double density, int cubic) {
    rc::LaunchSize z;
    z.hits = hits;
    z.steps = steps;
    z.density = density;
    return rc::lanes_per_max(z, cubic != 0);
}
}
"""


def compile_rules(d):
    """The rules as a shared library in directory d (a pathlib.Path)."""
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-ffp-contract=off", "-shared", "-fPIC", "-I", CSRC,
                    "-o", str(d / "shim.so"), str(d / "shim.cpp")], check=True)
    lib = C.CDLL(str(d / "shim.so"))
    lib.lanes_per_ray.argtypes = [C.c_double, C.c_double, C.c_int]
    lib.lanes_per_sum.argtypes = lib.lanes_per_max.argtypes = [C.c_double, C.c_double, C.c_double, C.c_int]
    return lib


def view(dims, spacing, eye, target, size, fovy=30.0, up=(0.0, 0.0, 1.0)):
    f = np.subtract(target, eye)
    f = f / np.linalg.norm(f)
    r = np.cross(f, up)
    r = r / np.linalg.norm(r)
    th = np.tan(np.radians(fovy) / 2)
    return np.concatenate([np.divide(eye, spacing), f, r, np.cross(r, f), [th * size[0] / size[1], th, *size]])


def launch_size(rules, dims, spacing, step, views):
    v = np.ascontiguousarray(np.stack(views), dtype=np.float64)
    out = (C.c_double * 3)()
    rules.launch_size((C.c_int * 3)(*dims), (C.c_double * 3)(*spacing), C.c_double(step),
                      v.ctypes.data_as(C.POINTER(C.c_double)), len(views), out)
    return tuple(out)


def camera_view(cam, spacing):
    """The view record of a camera dict."""
    return view(None, spacing, cam["eye"], cam["target"], (cam["width"], cam["height"]), cam["fovy_deg"], cam["up"])
