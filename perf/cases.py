"""Performance cases of the raycaster: what a user's program calls, over the
range of sizes, storages and forms it calls it with.

Kinds of case (key "kind"):
  frame     one interactive frame: a table edit, a camera move, one render
  orbit     several views of one volume in one call, any ray function,
            reconstruction filter or table form
  scan      a new scan of the same shape arrives on the device, and its first
            frame is rendered
  fit       one iteration of fitting a transfer function to images of several
            views: forward, loss gradient, table gradient
  proposal  views rendered with the learned sampling proposal
  train     one round of the proposal's training: features and opacity profiles
            of a view's rays, then the network's gradient on them

Volumes are seeded head phantoms (nested ellipsoids of tissue classes, a tumor
sphere, Rician noise; 12-bit codes), tables are a tissue table with seeded
changes (or the seeded noise a fit starts from), cameras lie on an orbit.
exact() restates the method in FP64 torch on the FP32 sample positions that
the interface specifies.
"""
import math

import numpy as np
import torch

import paper_1211_5595_gb300 as rc

VMAX = 4095
STORAGES = {"f32": rc.RC_STORE_F32, "f16": rc.RC_STORE_F16, "u16": rc.RC_STORE_U16}
FUNCS = {"composite": rc.RC_FUNC_COMPOSITE, "mip": rc.RC_FUNC_MIP, "average": rc.RC_FUNC_AVERAGE,
         "xray": rc.RC_FUNC_XRAY, "iso": rc.RC_FUNC_ISO, "threshold": rc.RC_FUNC_THRESHOLD}
GMAX = 1200.0


def _case(kind, dims, size, views=1, spacing=(1.0, 1.0, 1.0), storage="f32", func="composite", filter="trilinear",
          shade=True, step=0.5, term=0.99, entries=256, rows=0, fp16=False, iso=0.0, nimp=0, name=None):
    """A case as plain values. rows > 0: a 2-D table of that many gradient rows."""
    c = dict(kind=kind, nx=dims[0], ny=dims[1], nz=dims[2], sx=spacing[0], sy=spacing[1], sz=spacing[2],
             width=size[0], height=size[1], views=views, storage=storage, func=func, filter=filter, shade=shade,
             step=step, term=term, entries=entries, rows=rows, fp16=fp16, iso=iso, nimp=nimp)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: dragging a table's control point over a small preview volume
        _case("frame", (64, 64, 32), (256, 256), spacing=(1.0, 1.0, 3.0), shade=False, name="frame_preview_64"),
        # the ordinary job: a shaded orbit of one head scan for a review video
        _case("orbit", (256, 256, 180), (1024, 1024), views=12, name="orbit_shaded_256"),
        # the largest volume and image: a still at print size from 16-bit storage, quarter steps
        _case("orbit", (512, 512, 256), (2048, 2048), storage="u16", step=0.25, entries=1024, fp16=True,
              name="still_u16_512"),
        # an odd-shaped scan in FP16 storage, unshaded, in a window of ragged size
        _case("orbit", (181, 217, 157), (901, 703), views=4, spacing=(1.0, 1.0, 1.2), storage="f16", shade=False,
              fp16=True, name="views_f16_ragged"),
        # a time series or a queue of patients: every step is a new volume and its first picture
        _case("scan", (256, 256, 180), (1024, 1024), name="scan_256"),
        # the higher-quality reconstruction for publication views
        _case("orbit", (256, 256, 180), (1024, 1024), views=4, filter="bspline", name="orbit_bspline_256"),
        # maximum intensity projections, the usual look at vessels and bright lesions
        _case("orbit", (256, 256, 180), (1024, 1024), views=8, func="mip", shade=False, name="orbit_mip_256"),
        # an isosurface view of the same scan
        _case("orbit", (256, 256, 180), (1024, 1024), views=4, func="iso", iso=2200.0, name="orbit_iso_256"),
        # fitting a table to reference images: the differentiable path
        _case("fit", (128, 128, 96), (512, 512), views=8, shade=False, name="fit_table_128"),
        # the same for a table over value and gradient magnitude
        _case("fit", (128, 128, 96), (512, 512), views=4, shade=False, rows=32, name="fit_table2d_128"),
        # the learned proposal at 64 samples a ray
        _case("proposal", (256, 256, 180), (1024, 1024), views=6, nimp=64, name="proposal_256"),
        # training the proposal on the rays of one view
        _case("train", (256, 256, 180), (512, 512), name="train_proposal_256"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: any kind, sizes over their whole range, odd ones too."""
    kind = rng.choice(["frame", "orbit", "orbit", "orbit", "scan", "fit", "fit", "proposal", "train"])
    dims = (_log_int(rng, 48, 320), _log_int(rng, 48, 320), _log_int(rng, 32, 256))
    spacing = rng.choice([(1.0, 1.0, 1.0), (1.0, 1.0, 1.2), (1.0, 1.0, 3.0), (0.5, 0.5, 2.0)])
    size = (_log_int(rng, 128, 1100), _log_int(rng, 128, 1100))
    views = rng.randint(1, 6)
    storage = rng.choice(["f32", "f32", "f16", "u16"])
    step = rng.choice([0.5, 0.5, 0.5, 0.25, 1.0, 0.4])
    entries = rng.choice([256, 256, 512, 200, 1024])
    fp16 = storage != "f32" and rng.random() < 0.5
    shade = rng.random() < 0.7
    if kind == "frame":
        return _case(kind, dims, (min(size[0], 640), min(size[1], 640)), spacing=spacing, storage=storage, shade=shade,
                     step=step, entries=entries, fp16=fp16)
    if kind == "scan":
        return _case(kind, dims, size, spacing=spacing, storage=storage, shade=shade, step=step, entries=entries,
                     fp16=fp16)
    if kind == "fit":
        rows = rng.choice([0, 0, 16, 32])
        dims = tuple(min(d, 160) for d in dims)
        size = tuple(min(s, 512) for s in size)
        return _case(kind, dims, size, views=min(views, 4), spacing=spacing, storage=storage, shade=rng.random() < 0.4,
                     step=max(step, 0.4), term=rng.choice([0.99, 1.0]), entries=min(entries, 512), rows=rows,
                     filter=rng.choice(["trilinear", "trilinear", "bspline"]))
    if kind == "proposal":
        return _case(kind, dims, size, views=views, spacing=spacing, storage=storage, shade=shade, entries=entries,
                     nimp=rng.choice([16, 32, 64, 100, 128]))
    if kind == "train":
        return _case(kind, dims, (min(size[0], 640), min(size[1], 640)), spacing=spacing, storage=storage, shade=shade,
                     entries=entries)
    func = rng.choice(["composite", "composite", "composite", "mip", "average", "xray", "iso", "threshold"])
    filt = rng.choice(["trilinear", "trilinear", "bspline"])
    rows = rng.choice([0, 0, 24]) if func == "composite" else 0
    return _case(kind, dims, size, views=min(views, 3) if filt == "bspline" else views, spacing=spacing,
                 storage=storage, func=func, filter=filt, shade=shade, step=step, entries=min(entries, 256) if rows
                 else entries, rows=rows, fp16=fp16, iso=float(rng.choice([350, 900, 1600, 2200, 2900])))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
_LAYERS = ((0.92, 3000.0), (0.80, 400.0), (0.74, 1400.0), (0.58, 1800.0))
_POINTS = np.array([(0.0, 0.0, 0.0, 0.0, 0.0), (300.0, 0.0, 0.0, 0.0, 0.0), (400.0, 0.25, 0.45, 1.0, 0.02),
                    (900.0, 0.6, 0.55, 0.7, 0.02), (1400.0, 0.9, 0.7, 0.6, 0.04), (1800.0, 1.0, 0.92, 0.82, 0.06),
                    (2400.0, 1.0, 0.8, 0.7, 0.06), (2600.0, 1.0, 0.12, 0.1, 0.8), (2800.0, 1.0, 0.9, 0.9, 0.1),
                    (3000.0, 1.0, 1.0, 1.0, 0.1), (4095.0, 1.0, 1.0, 1.0, 0.1)])


def _dims(case):
    return (case["nx"], case["ny"], case["nz"]), (case["sx"], case["sy"], case["sz"])


def _codes(case, seed):
    """Head phantom, int16 codes 0..4095 of shape (nz, ny, nx) on the GPU."""
    (nx, ny, nz), sp = _dims(case)
    g = torch.Generator(device="cuda").manual_seed(1000003 * (seed + 1))
    ax = [(torch.arange(n, device="cuda", dtype=torch.float32) * (2.0 / (n - 1)) - 1.0) for n in (nx, ny, nz)]
    r = np.random.default_rng(seed)
    q = r.uniform(-0.25, 0.25, 3)
    half = [(n - 1) * s / 2.0 for n, s in zip((nx, ny, nz), sp)]
    rad = 0.12 * min(half)
    rho = torch.sqrt(ax[2][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[0][None, None, :] ** 2)
    v = torch.zeros_like(rho)
    for radius, value in _LAYERS:
        v = torch.where(rho <= radius, value, v)
    d2 = sum(((a - float(qi)) * float(h)).reshape(shape) ** 2
             for a, qi, h, shape in zip(ax, q, half, ((1, 1, -1), (1, -1, 1), (-1, 1, 1))))
    v = torch.where(d2 <= rad * rad, 2600.0, v)
    n1 = torch.randn(v.shape, generator=g, device="cuda") * 40.0
    n2 = torch.randn(v.shape, generator=g, device="cuda") * 40.0
    return torch.sqrt((v + n1) ** 2 + n2 ** 2).round().clamp(0, VMAX).to(torch.int16)


def _table(case, seed):
    """(K, 4) or (M, K, 4) float32 numpy table."""
    r = np.random.default_rng(7919 * (seed + 1))
    K, M = case["entries"], case["rows"]
    if case["kind"] == "fit":
        t = r.random((K, 4))
        t[:, 3] *= 0.1
    else:
        p = _POINTS.copy()
        p[2:, 1:4] = np.clip(p[2:, 1:4] + r.uniform(-0.1, 0.1, (len(p) - 2, 3)), 0.0, 1.0)
        p[2:, 4] = np.clip(p[2:, 4] * r.uniform(0.8, 1.2, len(p) - 2), 0.0, 1.0)
        xs = np.arange(K) * (VMAX / (K - 1))
        t = np.stack([np.interp(xs, p[:, 0], p[:, c]) for c in range(1, 5)], axis=1)
    if M:
        x = np.clip(np.arange(M) / (M - 1) / 0.5, 0.0, 1.0)
        w = 0.3 + 0.7 * x * x * (3.0 - 2.0 * x)
        t = np.repeat(t[None], M, axis=0)
        t[..., 3] *= w[:, None]
    return np.clip(t, 0.0, 1.0).astype(np.float32)


def _camera(case, i):
    (nx, ny, nz), sp = _dims(case)
    e = [(n - 1) * s for n, s in zip((nx, ny, nz), sp)]
    dist = 1.1 * math.sqrt(sum(x * x for x in e)) / 2.0 / math.sin(math.radians(15.0))
    az, el = math.radians(12.0 + 360.0 * i / case["views"]), math.radians(20.0)
    off = (dist * math.cos(el) * math.cos(az), dist * math.cos(el) * math.sin(az), dist * math.sin(el))
    f = lambda x: float(np.float32(x))  # noqa: E731
    return dict(eye=tuple(f(a / 2 + b) for a, b in zip(e, off)), target=tuple(f(a / 2) for a in e), up=(0.0, 0.0, 1.0),
                fovy_deg=30.0, width=case["width"], height=case["height"])


def _params(case):
    return rc.RenderParams(step_vox=case["step"], term=case["term"], shade=case["shade"], func=FUNCS[case["func"]],
                           iso=case["iso"], skip=True,
                           filter=rc.RC_FILTER_BSPLINE if case["filter"] == "bspline" else rc.RC_FILTER_TRILINEAR)


def _network(seed):
    """Network parameters: He-uniform weights, and output biases that favour
    the near bins as a trained network's PDFs do."""
    r = np.random.default_rng(104729 * (seed + 1))
    out = []
    for li, (k, n) in enumerate(((112, 64), (64, 64), (64, 64), (64, 40))):
        w = r.uniform(-1.0, 1.0, (k, n)) * math.sqrt(6.0 / k)
        b = np.zeros(n)
        if li == 0:
            w[110:] = 0.0
        if li == 3:
            w[:, 33:] = 0.0
            b[:32] = 1.5 - 0.12 * np.arange(32)
        out += [w.reshape(-1), b]
    return np.concatenate(out).astype(np.float32)


def _target(case, seed):
    """The images a table is fitted to: smooth colours, (views, H, W, 4)."""
    g = torch.Generator(device="cuda").manual_seed(seed + 5)
    low = torch.rand((case["views"], 4, 9, 9), generator=g, device="cuda")
    return torch.nn.functional.interpolate(low, (case["height"], case["width"]), mode="bilinear",
                                           align_corners=True).permute(0, 2, 3, 1).contiguous()


class _State:
    """A context, a volume on the device and the buffers of one user's program."""

    def __init__(self, case, seed):
        dims, spacing = _dims(case)
        self.kind, self.case = case["kind"], case
        self.params = _params(case)
        self.cams = [rc.make_camera(_camera(case, i)) for i in range(case["views"])]
        self.codes = _codes(case, seed)
        self.table = _table(case, seed)
        self.ctx = rc.rc_context_create(0)
        self.vol = rc.rc_volume_create(self.ctx, dims, spacing, VMAX, STORAGES[case["storage"]])
        rc.rc_volume_upload(self.ctx, self.vol, self.codes)
        n, px = case["views"], case["width"] * case["height"]
        f32 = dict(device="cuda", dtype=torch.float32)
        if self.kind == "fit":
            self.table_dev = torch.from_numpy(self.table).cuda()
            self.dtf = torch.empty(self.table.shape, **f32)
            self.target = _target(case, seed)
        else:
            self.set_table()
        if self.kind in ("proposal", "train"):
            rc.rc_proposal_load(self.ctx, rc.pack_proposal_blob(_network(seed)))
        if self.kind == "train":
            self.features = torch.empty((px, rc.RC_PROPOSAL_FEATURES), **f32)
            self.profiles = torch.empty((px, rc.RC_PROPOSAL_OUTPUTS), **f32)
            self.grad = torch.empty(rc.RC_PROPOSAL_PARAMS, **f32)
            self.loss = torch.empty(1, **f32)
            rc.rc_camera_set(self.ctx, self.cams[0])
        else:
            self.out = torch.empty((n, case["height"], case["width"], 4), **f32)
        rc.rc_context_sync(self.ctx)

    def set_table(self):
        if self.case["rows"]:
            rc.rc_tf2d_set(self.ctx, self.table, GMAX, self.case["fp16"])
        else:
            rc.rc_tf_set(self.ctx, self.table, self.case["fp16"])

    def __del__(self):
        try:
            torch.cuda.synchronize()
            rc.rc_volume_destroy(self.ctx, self.vol)
            rc.rc_context_destroy(self.ctx)
        except Exception:
            pass


def prepare(case, seed):
    return _State(case, seed)


def run(s):
    c = s.case
    if s.kind == "frame":
        s.set_table()
        rc.rc_camera_set(s.ctx, s.cams[0])
        rc.rc_render(s.ctx, s.vol, s.params, s.out)
        return s.out
    if s.kind == "orbit":
        rc.rc_render_views(s.ctx, s.vol, s.params, s.cams, s.out)
        return s.out
    if s.kind == "scan":
        rc.rc_volume_upload(s.ctx, s.vol, s.codes)
        rc.rc_camera_set(s.ctx, s.cams[0])
        rc.rc_render(s.ctx, s.vol, s.params, s.out)
        return s.out
    if s.kind == "fit":
        if c["rows"]:
            rc.rc_tf2d_set_device(s.ctx, s.table_dev, GMAX, c["fp16"])
        else:
            rc.rc_tf_set_device(s.ctx, s.table_dev, c["fp16"])
        rc.rc_render_views(s.ctx, s.vol, s.params, s.cams, s.out)
        dimg = (s.out - s.target) * (2.0 / s.out.numel())
        rc.rc_render_backward_views_with_forward(s.ctx, s.vol, s.params, s.cams, s.out, dimg, s.dtf)
        return {"images": s.out, "dtf": s.dtf}
    if s.kind == "proposal":
        rc.rc_render_proposal_views(s.ctx, s.vol, s.params, s.cams, c["nimp"], 2.0, s.out)
        return s.out
    rc.rc_proposal_features(s.ctx, s.vol, s.params, s.features)
    rc.rc_profiles_generate(s.ctx, s.vol, s.params, s.profiles)
    rc.rc_proposal_grad(s.ctx, s.features, s.profiles, s.features.shape[0], s.grad, s.loss)
    return {"features": s.features, "profiles": s.profiles, "grad": s.grad, "loss": s.loss}


def work(case):
    """Bytes: the volume's codes as stored (as uploaded for a new scan) read
    once, images and gradients read or written once. Flops: an estimate from
    the number of samples that carry opacity before a ray ends (about 3% of
    the box diagonal's samples per pixel with a tissue table, 12% with a fit's
    opaque table) and the arithmetic of one sample."""
    dims, spacing = _dims(case)
    vox = dims[0] * dims[1] * dims[2]
    px = case["views"] * case["width"] * case["height"]
    diag = math.sqrt(sum(((n - 1) * s / min(spacing)) ** 2 for n, s in zip(dims, spacing)))
    esz = 4 if case["storage"] == "f32" and case["kind"] != "scan" else 2
    per = (400 if case["filter"] == "bspline" else 90) + (60 if case["shade"] else 0) + (40 if case["rows"] else 0)
    frac = 0.12 if case["kind"] == "fit" else 0.028
    samples = px * (frac * diag / case["step"])
    b, f = vox * esz + px * 16, samples * per
    if case["kind"] == "fit":
        b += px * 32
        f *= 3
    if case["kind"] == "proposal":
        f = px * 0.4 * (case["nimp"] * 0.4 * per + 2 * 17920)
    if case["kind"] == "train":
        b = vox * esz + 2 * px * (112 + 33) * 4
        f = px * 0.4 * (200 * 100) + px * 2 * 46592
    return {"bytes": float(b), "flops": float(f)}


# ---------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------
F32, F64 = torch.float32, torch.float64
_BATCH = 1 << 21            # samples evaluated at once


def _t32(x):
    return torch.tensor(np.float32(x), device="cuda")


def _fma(a, b, c):
    """FP32 fused multiply-add (the product is exact in FP64)."""
    return (a.double() * b.double() + c.double()).float()


class _Rays:
    """Rays of one view in the FP32 specification of the interface; hits only."""

    def __init__(self, case, i):
        dims, sp = _dims(case)
        cam = _camera(case, i)
        W, H = cam["width"], cam["height"]
        eye, tgt, up = (np.array([np.float32(x) for x in cam[k]], dtype=np.float64) for k in ("eye", "target", "up"))
        f = tgt - eye
        f /= math.sqrt(f[0] * f[0] + f[1] * f[1] + f[2] * f[2])
        r = np.array([f[1] * up[2] - f[2] * up[1], f[2] * up[0] - f[0] * up[2], f[0] * up[1] - f[1] * up[0]])
        r /= math.sqrt(r[0] * r[0] + r[1] * r[1] + r[2] * r[2])
        u = np.array([r[1] * f[2] - r[2] * f[1], r[2] * f[0] - r[0] * f[2], r[0] * f[1] - r[1] * f[0]])
        th = math.tan(cam["fovy_deg"] * math.pi / 360.0)
        x = torch.arange(W, device="cuda", dtype=F32)[None, :].expand(H, W).reshape(-1)
        y = torch.arange(H, device="cuda", dtype=F32)[:, None].expand(H, W).reshape(-1)
        ndcx = ((x + 0.5) / _t32(W) * 2.0 - 1.0) * _t32(th * W / H)
        ndcy = (1.0 - (y + 0.5) / _t32(H) * 2.0) * _t32(th)
        v = [(_t32(f[a]) + ndcx * _t32(r[a])) + ndcy * _t32(u[a]) for a in range(3)]
        ln = torch.sqrt((v[0] * v[0] + v[1] * v[1]) + v[2] * v[2])
        tn = torch.zeros_like(x)
        tf = torch.full_like(x, math.inf)
        hit = torch.ones_like(x, dtype=torch.bool)
        o, d, dr = [], [], []
        for a in range(3):
            da = v[a] / ln
            dd = da / _t32(sp[a])
            oa = _t32(float(eye[a]) / float(np.float32(sp[a])))
            hi = _t32(dims[a] - 1)
            t0, t1 = (0.0 - oa) / dd, (hi - oa) / dd
            flat = dd == 0
            tn = torch.where(flat, tn, torch.maximum(tn, torch.minimum(t0, t1)))
            tf = torch.where(flat, tf, torch.minimum(tf, torch.maximum(t0, t1)))
            hit &= ~(flat & ((oa < 0) | (oa > hi)))
            o.append(oa)
            d.append(dd)
            dr.append(da)
        hit &= tf >= tn
        self.pixels = W * H
        self.idx = torch.nonzero(hit).squeeze(1)
        self.tn, self.tf = tn[hit], tf[hit]
        self.d, self.dir = torch.stack(d, 1)[hit], torch.stack(dr, 1)[hit]
        self.o = torch.stack(o)
        self.smin = np.float32(min(sp))
        self.ds = np.float32(np.float32(case["step"]) * self.smin)
        self.n = (torch.floor((self.tf - self.tn) / _t32(self.ds)).clamp(max=16777215.0)).long() + 1

    def position(self, sel, t):
        """FP32 index-space positions at distances t (rays sel x samples)."""
        return _fma(t[..., None], self.d[sel][:, None, :], self.o)


class _Field:
    """The scalar field of a case in FP64 and its classification."""

    def __init__(self, case, seed):
        self.case = case
        self.dims, self.sp = _dims(case)
        v = _codes(case, seed).float()
        self.scalar = v.reshape(-1)
        self.vol = v
        self.table = torch.from_numpy(_table(case, seed)).cuda()
        if case["fp16"]:
            self.table = self.table.half().float()
        self.table = self.table.double()
        self.vg = None

    def _gradients(self):
        if self.vg is None:
            v, ch = self.vol, [self.vol]
            for dim in (2, 1, 0):
                n = v.shape[dim]
                up = torch.arange(n, device="cuda")
                hi, lo = (up + 1).clamp(max=n - 1), (up - 1).clamp(min=0)
                ch.append(v.index_select(dim, hi) - v.index_select(dim, lo))
            self.vg = torch.stack(ch, -1).reshape(-1, 4)
        return self.vg

    def cell(self, p):
        base, w = [], []
        for a in range(3):
            q = p[..., a].clamp(0.0, float(self.dims[a] - 1))
            b = q.floor().clamp(max=float(self.dims[a] - 2))
            base.append(b.long())
            w.append((q - b).double())
        return base, w

    def trilinear(self, p, grad):
        (i, j, k), w = self.cell(p)
        nx, ny = self.dims[0], self.dims[1]
        src = self._gradients() if grad else self.scalar[:, None]
        at = (k * ny + j) * nx + i
        acc = 0.0
        for oz in (0, 1):
            for oy in (0, 1):
                for ox in (0, 1):
                    wt = (w[0] if ox else 1 - w[0]) * (w[1] if oy else 1 - w[1]) * (w[2] if oz else 1 - w[2])
                    acc = acc + src[at + (oz * ny + oy) * nx + ox].double() * wt[..., None]
        g = None
        if grad:
            g = torch.stack([acc[..., 1 + a] * (0.5 / self.sp[a]) for a in range(3)], -1)
        return acc[..., 0], g

    def bspline(self, p, grad):
        base, w = self.cell(p)
        nx, ny = self.dims[0], self.dims[1]
        wt, dw, ix = [], [], []
        for a in range(3):
            t = w[a]
            s = 1 - t
            wt.append([s ** 3 / 6, 0.5 * t ** 3 - t * t + 2.0 / 3, -0.5 * t ** 3 + 0.5 * t * t + 0.5 * t + 1.0 / 6,
                       t ** 3 / 6])
            dw.append([-0.5 * s * s, 1.5 * t * t - 2 * t, -1.5 * t * t + t + 0.5, 0.5 * t * t])
            ix.append([(base[a] + e).clamp(0, self.dims[a] - 1) for e in (-1, 0, 1, 2)])
        f, gx, gy, gz = 0.0, 0.0, 0.0, 0.0
        for z in range(4):
            fz, gxz, gyz = 0.0, 0.0, 0.0
            for y in range(4):
                row = (ix[2][z] * ny + ix[1][y]) * nx
                v = [self.scalar[row + ix[0][x]].double() for x in range(4)]
                fx = sum(a * b for a, b in zip(v, wt[0]))
                fz = fz + fx * wt[1][y]
                if grad:
                    gxz = gxz + sum(a * b for a, b in zip(v, dw[0])) * wt[1][y]
                    gyz = gyz + fx * dw[1][y]
            f = f + fz * wt[2][z]
            if grad:
                gx, gy, gz = gx + gxz * wt[2][z], gy + gyz * wt[2][z], gz + fz * dw[2][z]
        if not grad:
            return f, None
        return f, torch.stack([gx / self.sp[0], gy / self.sp[1], gz / self.sp[2]], -1)

    def value(self, p, grad=False):
        return self.bspline(p, grad) if self.case["filter"] == "bspline" else self.trilinear(p, grad)

    def cells_of_table(self, val, g):
        """Table entries around each sample and their weights: (indices, weights)."""
        K, M = self.case["entries"], self.case["rows"]
        u = (val * ((K - 1) / VMAX)).clamp(0, K - 1)
        i = u.floor().clamp(max=K - 2)
        a = u - i
        i = i.long()
        if not M:
            return [i, i + 1], [1 - a, a]
        w = (g.square().sum(-1).sqrt() * ((M - 1) / GMAX)).clamp(0, M - 1)
        j = w.floor().clamp(max=M - 2)
        b = w - j
        e = j.long() * K + i
        return [e, e + 1, e + K, e + K + 1], [(1 - a) * (1 - b), a * (1 - b), (1 - a) * b, a * b]

    def shading(self, g, dirs):
        g2 = g.square().sum(-1)
        ndl = ((g * dirs).sum(-1).abs() / g2.clamp(min=1e-300).sqrt()).clamp(max=1.0)
        flat = g2 < (1e-6 * VMAX) ** 2
        return torch.where(flat, 0.8, 0.1 + 0.7 * ndl), torch.where(flat, 0.0, 0.2 * ndl ** 16)

    def sample(self, p, dirs, shade):
        """Straight colour, opacity per reference step, and what the gradient needs."""
        val, g = self.value(p, shade or self.case["rows"] > 0)
        ent, wts = self.cells_of_table(val, g)
        flat = self.table.reshape(-1, 4)
        e = sum(flat[i] * w[..., None] for i, w in zip(ent, wts))
        col, al, k = e[..., :3], e[..., 3], 1.0
        if shade:
            sf, spec = self.shading(g, dirs[:, None, :].double())
            raw = col * sf[..., None] + spec[..., None]
            k = torch.where(raw < 1.0, sf[..., None], 0.0)
            col = raw.clamp(max=1.0)
        return col, al, k, ent, wts


def _corrected(al, ratio):
    return 1.0 - (1.0 - al) ** ratio


def _march(field, rays, times, count, ratio, term, shade):
    """Front-to-back composite of count[r] samples at times(rays, k): RGBA per hit ray."""
    n = rays.idx.numel()
    C = torch.zeros((n, 3), device="cuda", dtype=F64)
    T = torch.ones(n, device="cuda", dtype=F64)
    alive, k0, S = torch.arange(n, device="cuda"), 0, 8
    while alive.numel():
        keep = []
        for sel in alive.split(_BATCH // S):
            ks = torch.arange(k0, k0 + S, device="cuda")
            col, al, _, _, _ = field.sample(rays.position(sel, times(sel, ks)), rays.dir[sel], shade)
            r = ratio[sel][:, None] if torch.is_tensor(ratio) else ratio
            ap = torch.where(ks[None, :] < count[sel][:, None], _corrected(al, r), 0.0)
            t, c = T[sel], C[sel]
            for q in range(S):                  # a ray ends after the sample that reaches the limit
                on = (1.0 - t < term).double()
                c = c + (on * t * ap[:, q])[:, None] * col[:, q]
                t = t * (1.0 - on * ap[:, q])
            C[sel], T[sel] = c, t
            keep.append(sel[(1.0 - t < term) & (count[sel] > k0 + S)])
        alive = torch.cat(keep)
        k0 += S
    return torch.cat([C, (1.0 - T)[:, None]], 1)


def _step_times(rays):
    ds = _t32(rays.ds)
    return lambda sel, ks: _fma(ks.float()[None, :], ds, rays.tn[sel][:, None])


def _put(rays, rgba, case):
    out = torch.zeros((rays.pixels, 4), device="cuda", dtype=F64)
    out[rays.idx] = rgba
    return out.reshape(case["height"], case["width"], 4)


def _function(field, rays, case):
    """The ray functions other than compositing, per hit ray."""
    n, func = rays.idx.numel(), case["func"]
    times = _step_times(rays)
    acc = torch.full((n,), -1.0 if func == "mip" else 0.0, device="cuda", dtype=F64)
    first = torch.full((n,), -1, device="cuda", dtype=torch.long)
    prev, cross = torch.zeros(n, device="cuda", dtype=F64), torch.zeros(n, device="cuda", dtype=F64)
    found = torch.zeros(n, device="cuda", dtype=F64)
    iso = float(np.float32(case["iso"]))
    alive, k0, S = torch.arange(n, device="cuda"), 0, 8
    while alive.numel():
        keep = []
        for sel in alive.split(_BATCH // S):
            ks = torch.arange(k0, k0 + S, device="cuda")
            on = ks[None, :] < rays.n[sel][:, None]
            t = times(sel, ks)
            val, _ = field.value(rays.position(sel, t))
            if func == "mip":
                acc[sel] = torch.maximum(acc[sel], torch.where(on, val, -1.0).amax(1))
            elif func in ("average", "xray"):
                acc[sel] += torch.where(on, val, 0.0).sum(1)
            else:
                over = on & (val >= iso)
                at = torch.where(over.any(1), over.float().argmax(1), -1)
                h = at >= 0
                a, rows = at[h], torch.nonzero(h).squeeze(1)
                v1, t1 = val[rows, a], t[rows, a].double()
                v0 = torch.where(a > 0, val[rows, (a - 1).clamp(min=0)], prev[sel[h]])
                t0 = _fma((a + k0 - 1).clamp(min=0).float(), _t32(rays.ds), rays.tn[sel[h]]).double()
                cross[sel[h]] = torch.where(a + k0 > 0, t0 + (t1 - t0) * ((iso - v0) / (v1 - v0)), t1)
                first[sel[h]] = a + k0
                found[sel[h]] = v1
                prev[sel] = val[:, -1]
                sel = sel[~h]
            keep.append(sel[rays.n[sel] > k0 + S])
        alive = torch.cat(keep)
        k0 += S
    if func == "mip":
        m = acc / VMAX
    elif func == "average":
        m = acc / rays.n / VMAX
    elif func == "xray":
        m = acc * float(rays.ds) / VMAX
    else:
        out = torch.zeros((n, 4), device="cuda", dtype=F64)
        h = torch.nonzero(first >= 0).squeeze(1)
        if func == "threshold":
            ent, wts = field.cells_of_table(found[h], None)
            out[h, :3] = sum(field.table[i] * w[:, None] for i, w in zip(ent, wts))[:, :3]
            out[h, 3] = 1.0
            return out
        for sel in h.split(_BATCH):
            p = rays.position(sel, _fma(first[sel].float(), _t32(rays.ds), rays.tn[sel])[:, None])
            sf, spec = field.shading(field.value(p, True)[1][:, 0], rays.dir[sel].double())
            out[sel] = torch.stack([cross[sel], (sf + spec).clamp(max=1.0), first[sel].double(),
                                    torch.ones_like(sf)], 1)
        return out
    return torch.stack([m, m, m, torch.ones_like(m)], 1)


def _table_gradient(field, rays, dimg, ratio, term, shade, out):
    """Adds the table gradient of one view to out (entries x 4)."""
    dimg = dimg.reshape(-1, 4).double()
    times = _step_times(rays)
    order = torch.argsort(rays.n)
    N = int(rays.n.max())
    for sel in order.split(max(1, _BATCH // N)):
        m = int(rays.n[sel].max())
        ks = torch.arange(m, device="cuda")
        col, al, dcol, ent, wts = field.sample(rays.position(sel, times(sel, ks)), rays.dir[sel], shade)
        on = ks[None, :] < rays.n[sel][:, None]
        ap = torch.where(on, _corrected(al, ratio), 0.0)
        T = torch.cumprod(1.0 - ap, 1)
        before = torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
        on &= 1.0 - before < term
        ap = torch.where(on, ap, 0.0)
        T = torch.cumprod(1.0 - ap, 1)
        before = torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
        wgt = before * ap
        part = wgt[..., None] * col
        after = part.sum(1, keepdim=True) - torch.cumsum(part, 1)
        g = dimg[rays.idx[sel]]
        inv = torch.where(ap < 1.0, 1.0 / (1.0 - ap).clamp(min=1e-300), 0.0)
        dap = ((before[..., None] * col - after * inv[..., None]) * g[:, None, :3]).sum(-1) + \
            g[:, None, 3] * T[:, -1:] * inv
        dal = dap if ratio == 1.0 else dap * ratio * (1.0 - al.clamp(max=1.0 - 1e-6)) ** (ratio - 1.0)
        d = torch.cat([g[:, None, :3] * wgt[..., None] * dcol, dal[..., None]], -1)
        d = torch.where(on[..., None], d, 0.0).reshape(-1, 4)
        for i, w in zip(ent, wts):
            out.index_add_(0, i.reshape(-1), d * w.reshape(-1, 1))


def _occupied(field):
    """Which 16^3 cell-bricks may hold opacity (bz, by, bx), for a 1-D table."""
    K = field.case["entries"]
    cb = [(n - 1 + 15) // 16 for n in field.dims]
    v = field.vol
    for dim, n in ((0, cb[2]), (1, cb[1]), (2, cb[0])):
        idx = (torch.arange(n, device="cuda")[:, None] * 16 + torch.arange(17, device="cuda")).clamp(
            max=v.shape[dim] - 1)
        if dim == 0:
            lo = hi = v
        lo = lo.index_select(dim, idx.reshape(-1)).unflatten(dim, (n, 17)).amin(dim + 1)
        hi = hi.index_select(dim, idx.reshape(-1)).unflatten(dim, (n, 17)).amax(dim + 1)
    coef = _t32(np.float32(K - 1) / np.float32(VMAX))
    lo = (lo * coef).floor().long().clamp(max=K - 1)
    hi = ((hi * coef).floor().long() + 1).clamp(max=K - 1)
    seen = torch.cat([torch.zeros(1, device="cuda", dtype=torch.long), torch.cumsum(field.table[:, 3] != 0, 0)])
    return (seen[hi + 1] - seen[lo]) > 0


def _occupied_at(field, occ, p):
    (i, j, k), _ = field.cell(p)
    return occ[k >> 4, j >> 4, i >> 4]


def _features(field, rays):
    """The 112 features of every hit ray, in FP64, and the occupancy bits of the bins."""
    occ = _occupied(field)
    n = rays.idx.numel()
    everything = torch.arange(n, device="cuda")
    size = torch.tensor([float(d - 1) for d in field.dims], device="cuda")
    x = torch.cat([_fma(rays.tn[:, None], rays.d, rays.o) / size, rays.dir], 1)
    ang = x.double()[:, :, None] * (math.pi * 2.0 ** torch.arange(6, device="cuda", dtype=F64))
    enc = torch.stack([torch.sin(ang), torch.cos(ang)], -1).reshape(n, 72)
    bw = (rays.tf - rays.tn) / _t32(32.0)
    t = _fma(torch.arange(32, device="cuda").float()[None, :] + 0.5, bw[:, None], rays.tn[:, None])
    bits = _occupied_at(field, occ, rays.position(everything, t))
    return torch.cat([x.double(), enc, bits.double(), torch.zeros((n, 2), device="cuda", dtype=F64)], 1), bits, occ


def _bf16(x):
    return x.float().bfloat16().double()


def _layers(seed):
    p, off, out = torch.from_numpy(_network(seed)).cuda().double(), 0, []
    for k, n in ((112, 64), (64, 64), (64, 64), (64, 40)):
        out.append((p[off:off + k * n].reshape(k, n), p[off + k * n:off + k * n + n]))
        off += k * n + n
    return out


def _forward(layers, x):
    """Layer inputs (rounded to BF16) and the logits."""
    hs = [_bf16(x)]
    for w, b in layers[:3]:
        hs.append(_bf16((hs[-1] @ _bf16(w) + b).clamp(min=0.0)))
    return hs, hs[-1] @ _bf16(layers[3][0]) + layers[3][1]


def _exact_proposal(case, seed):
    field, layers, images = _Field(case, seed), _layers(seed), []
    for i in range(case["views"]):
        rays = _Rays(case, i)
        x, mid, occ = _features(field, rays)
        pdf = torch.cat([torch.softmax(_forward(layers, part)[1][:, :32], 1) for part in x.split(1 << 18)])
        n = rays.idx.numel()
        everything = torch.arange(n, device="cuda")
        bw = (rays.tf - rays.tn) / _t32(32.0)
        edge = _fma(torch.arange(33, device="cuda").float()[None, :], bw[:, None], rays.tn[:, None])
        edge[:, 0] = rays.tn
        at = _occupied_at(field, occ, rays.position(everything, edge))
        any_bin = at[:, :-1] | mid | at[:, 1:]
        some = any_bin.any(1)
        b0 = torch.where(some, any_bin.float().argmax(1), 0)
        reach = (torch.cumsum(pdf, 1) >= 1.0 - 1.0 / 64.0) & (torch.arange(32, device="cuda")[None, :] >= b0[:, None])
        b1 = torch.where(reach.any(1) & some, (reach.float().argmax(1) + 1).clamp(max=31), 31)
        ta = torch.where(b0 == 0, rays.tn, _fma(b0.float(), bw, rays.tn))
        tb = torch.where(b1 == 31, rays.tf, _fma((b1 + 1).float(), bw, rays.tn))
        seg = (tb - ta) / _t32(case["nimp"])
        ratio = (seg / _t32(rays.smin)).double()
        rgba = _march(field, rays, lambda sel, ks: _fma(ks.float()[None, :] + 0.5, seg[sel][:, None], ta[sel][:, None]),
                      torch.full((n,), case["nimp"], device="cuda"), ratio, case["term"], case["shade"])
        images.append(_put(rays, rgba, case))
    return torch.stack(images)


def _exact_train(case, seed):
    field, layers, rays = _Field(case, seed), _layers(seed), _Rays(case, 0)
    n = rays.pixels
    x = torch.zeros((n, 112), device="cuda", dtype=F64)
    x[rays.idx] = _features(field, rays)[0]
    y = torch.zeros((n, 33), device="cuda", dtype=F64)
    y[:, 32] = 1.0
    delta = (rays.tf - rays.tn) / _t32(512.0)
    ratio = (delta / _t32(rays.smin)).double()
    for sel in torch.arange(rays.idx.numel(), device="cuda").split(_BATCH // 512):
        t = _fma(torch.arange(512, device="cuda").float()[None, :] + 0.5, delta[sel][:, None], rays.tn[sel][:, None])
        ap = _corrected(field.sample(rays.position(sel, t), rays.dir[sel], False)[1], ratio[sel][:, None])
        T = torch.cumprod(1.0 - ap, 1)
        before = torch.cat([torch.ones_like(T[:, :1]), T[:, :-1]], 1)
        y[rays.idx[sel]] = torch.cat([(before * ap).reshape(-1, 32, 16).sum(-1), T[:, -1:]], 1)
    grads = [torch.zeros_like(w) for w, _ in layers], [torch.zeros_like(b) for _, b in layers]
    loss = 0.0
    for xs, ys in zip(x.split(1 << 18), y.split(1 << 18)):
        hs, z = _forward(layers, xs)
        w = ys[:, :32].sum(1, keepdim=True)
        q = ys[:, :32] / w.clamp(min=1e-300)
        logp = torch.log_softmax(z[:, :32], 1)
        th = torch.sigmoid(z[:, 32:33])
        dt = th - ys[:, 32:]
        loss = loss + (torch.where(q > 0, w * q * (q.clamp(min=1e-300).log() - logp), 0.0)).sum() + dt.square().sum()
        dz = torch.zeros_like(z)
        dz[:, :32] = w * (logp.exp() - q) / n
        dz[:, 32:33] = 2.0 * dt * th * (1.0 - th) / n
        for li in (3, 2, 1, 0):
            grads[0][li] += hs[li].t() @ dz
            grads[1][li] += dz.sum(0)
            if li:
                dz = torch.where(hs[li] > 0, dz @ _bf16(layers[li][0]).t(), 0.0)
    grad = torch.cat([t.reshape(-1) for w, b in zip(*grads) for t in (w, b)])
    return {"features": x, "profiles": y, "grad": grad, "loss": (loss / n).reshape(1)}


def exact(case, seed):
    if case["kind"] == "proposal":
        return _exact_proposal(case, seed)
    if case["kind"] == "train":
        return _exact_train(case, seed)
    field, images = _Field(case, seed), []
    ratio = float(np.float32(np.float32(case["step"]) * np.float32(min(_dims(case)[1]))) /
                  np.float32(min(_dims(case)[1])))
    term = float(np.float32(case["term"]))
    dtf = torch.zeros((field.table.numel() // 4, 4), device="cuda", dtype=F64)
    target = _target(case, seed) if case["kind"] == "fit" else None
    for i in range(case["views"]):
        rays = _Rays(case, i)
        if case["func"] != "composite":
            images.append(_put(rays, _function(field, rays, case), case))
            continue
        images.append(_put(rays, _march(field, rays, _step_times(rays), rays.n, ratio, term, case["shade"]), case))
        if target is not None:
            dimg = (images[-1] - target[i].double()) * (2.0 / target.numel())
            _table_gradient(field, rays, dimg, ratio, term, case["shade"], dtf)
    images = torch.stack(images)
    if target is not None:
        return {"images": images, "dtf": dtf.reshape(field.table.shape)}
    return images
