"""The work that users of this framework have it do, as cases that can be timed.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges,
``prepare(case, seed)`` builds what a program has in hand before the call,
``run(state)`` is one pass through the public entry points, ``work(case)`` the bytes
and operations the pass cannot do without, and ``exact(case, seed)`` the pass's
outputs in 64 bits by plain torch.

Kinds of case (``kind``):

* ``frame``   one ``Context.render`` of one or more cameras; with ``slider`` the
  transfer function is uploaded from host memory first (a viewer's slider drag);
* ``batch``   a registered batch of views over several volumes, replayed as a graph;
* ``grad``    forward and backward with the gradients of table, uniforms and voxels:
  through ``Context.render`` / ``render_backward``, or (``autograd``) through the
  torch binding, which also replaces the volume's intensities on every pass;
* ``fit``     one transfer-function fit step through the torch binding;
* ``open``    a study opened from host memory: load, morphology, table, first frame,
  volume freed again;
* ``vessels`` the multi-scale vesselness of a loaded volume;
* ``clean``   a loaded volume's intensities replaced, pre-filtered and its tissue
  histogram taken.

Volumes are head-like (nested tissue ellipsoids; 12-bit with a scalp and a skull
for ``t1``) or angiography-like (a branching tube tree) with seeded noise.
"""

import math

import numpy as np
import torch

import paper_2605_19737_gb300 as pkg
from paper_2605_19737_gb300 import autograd as ag

DEV = "cuda:0"
TABLE_W = 256
COHORT = ((96, 96, 96), (128, 160, 128), (181, 217, 181), (256, 256, 176))
# share of a frame's sample points that carry opacity (arithmetic that cannot be left out)
VISIBLE = {"head": 0.30, "t1": 0.33, "vessel": 0.03}


def _case(kind, name=None, **kw):
    c = dict(kind=kind, phantom="head", dtype="f32", nx=64, ny=64, nz=64, sz=1.0, W=128, H=128, cams=1, mode=0,
             rows=1, second=False, gamma=0.0, step=0.5, brick=8, derived=True, slider=False, autograd=False,
             volumes=1, cohort=False, sigmas="", filter="")
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: a thumbnail of a 64^3 volume, bound by latency
        _case("frame", "thumbnail_head64_128"),
        # the headline: a full-HD frame of a BrainWeb-sized T1 with curvature-modulated opacity
        _case("frame", "frame_t1_1080p", phantom="t1", dtype="u16", nx=181, ny=217, nz=181, W=1920, H=1080, mode=1,
              rows=64, gamma=0.5),
        # the same frame size over the vesselness channel of an angiography, at the tuned brick edge
        _case("frame", "frame_vessel_1080p", phantom="vessel", nx=256, ny=256, nz=176, W=1920, H=1080, mode=2,
              rows=64, sigmas="1,2,3", brick=16),
        # a slider drag in a viewer: new table from the host, then a quarter-size frame
        _case("frame", "slider_t1_540p", phantom="t1", dtype="u16", nx=181, ny=217, nz=181, W=960, H=540, mode=1,
              rows=64, gamma=0.5, brick=16, slider=True),
        # a context without the memory for derived bricks, odd sizes, thick slices
        _case("frame", "frame_stencil_odd", phantom="t1", dtype="u16", nx=151, ny=173, nz=97, sz=1.7, W=641, H=361,
              gamma=0.5, derived=False),
        # data-set rendering: many views of several volumes in one launch
        _case("batch", "batch_4vol_8cam_512", W=512, H=512, cams=8, volumes=4, cohort=True),
        # the smallest gradient: a thumbnail through autograd, table + uniforms + voxels
        _case("grad", "grad_head64_128", autograd=True),
        # the largest: full-HD forward and backward with every gradient
        _case("grad", "grad_t1_1080p", phantom="t1", dtype="u16", nx=181, ny=217, nz=181, W=1920, H=1080, mode=1,
              rows=64, gamma=0.5, brick=16),
        # one step of a transfer-function fit over 8 views
        _case("fit", "fit_head128_8x512", nx=128, ny=128, nz=128, W=512, H=512, cams=8),
        # time to first picture of a study in host memory
        _case("open", "open_t1_720p", phantom="t1", dtype="u16", nx=181, ny=217, nz=181, W=1280, H=720, mode=1,
              rows=64, gamma=0.5),
        # the vesselness stage of an angiography
        _case("vessels", "vessels_256x256x176", phantom="vessel", nx=256, ny=256, nz=176, sigmas="1,2,3"),
        # a noisy scan cleaned and its tissue peaks found
        _case("clean", "clean_t1_median", phantom="t1", dtype="u16", nx=181, ny=217, nz=181, filter="median"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame"] * 5 + ["batch", "grad", "grad", "fit", "open", "vessels", "clean"])
    phantom = rng.choice(["head", "t1", "vessel"])
    c = _case(kind, phantom=phantom, dtype="u16" if phantom == "t1" else "f32")
    for a in ("nx", "ny", "nz"):
        c[a] = _log_int(rng, 40, 230)
    c["sz"] = rng.choice([1.0, 1.0, 1.25, 2.0])
    c["W"] = _log_int(rng, 90, 1920)
    c["H"] = max(60, min(1080, int(c["W"] * rng.choice([0.5625, 0.75, 1.0]))))
    c["mode"] = rng.choice([0, 1, 2])
    c["gamma"] = rng.choice([0.0, 0.5])
    c["step"] = rng.choice([0.5, 0.5, 0.35, 1.0])
    c["brick"] = rng.choice([4, 8, 8, 16])
    if kind in ("grad", "fit", "batch"):
        c["cams"] = rng.choice([1, 2, 4])
        c["W"], c["H"] = min(c["W"], 700), min(c["H"], 600)
        c["step"] = 0.5
    if kind == "batch":
        c["volumes"] = rng.choice([1, 2, 4])
        c["brick"] = 8
    if kind == "frame":
        c["cams"] = rng.choice([1, 1, 1, 3])
        if c["cams"] > 1:
            c["W"], c["H"] = min(c["W"], 960), min(c["H"], 720)
        c["derived"] = rng.random() < 0.8
        c["slider"] = rng.random() < 0.4
    if kind == "grad":
        c["autograd"] = rng.random() < 0.5
    if kind in ("vessels", "clean"):
        c["mode"] = 0
    if kind == "clean":
        c["filter"] = rng.choice(["median", "gauss"])
    if kind == "batch" or kind == "fit":
        c["mode"] = min(c["mode"], 1)
    if c["mode"] == 2:
        c["second"] = rng.random() < 0.5
    if kind == "vessels" or (c["mode"] == 2 and not c["second"]):
        c["sigmas"] = rng.choice(["1", "1,2", "1,2,3", "1.5,2.5"])
    c["rows"] = 1 if c["mode"] == 0 else rng.choice([32, 64])
    return c


# ------------------------------------------------------------------ inputs

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) & 0x7FFFFFFF)


def _randn(shape, g):
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float32)


def _axes(dims):
    return [(torch.arange(n, device=DEV, dtype=torch.float32) + 0.5) / n * 2.0 - 1.0 for n in dims]


def _head(dims, g, classes, noise):
    """Nested ellipsoids (first class outermost), two ventricles of the class 'csf'."""
    x, y, z = _axes(dims)
    vol = torch.zeros(dims[::-1], device=DEV)

    def put(r, value, cx=0.0):
        q = (((z / r[2]) ** 2)[:, None, None] + ((y / r[1]) ** 2)[None, :, None] + (((x - cx) / r[0]) ** 2)[None, None])
        vol.masked_fill_(q <= 1.0, value)

    for r, name in (((0.97, 0.97, 0.95), "fat"), ((0.91, 0.92, 0.89), "bone"), ((0.86, 0.88, 0.84), "csf"),
                    ((0.81, 0.84, 0.79), "gm"), ((0.58, 0.63, 0.54), "wm")):
        if name in classes:
            put(r, classes[name])
    for cx in (-0.15, 0.15):
        put((0.11, 0.22, 0.10), classes["csf"], cx)
    return vol


def _volume(phantom, dtype, dims, g, rnd):
    if phantom == "head":
        return _head(dims, g, {"csf": 0.15, "gm": 0.45, "wm": 0.75}, 0.02) + 0.02 * _randn(dims[::-1], g)
    if phantom == "t1":
        v = _head(dims, g, {"fat": 3600.0, "bone": 90.0, "csf": 300.0, "gm": 560.0, "wm": 890.0}, 0.0)
        x, y, z = _axes(dims)
        f, p = rnd.uniform(0.5, 1.5, 3), rnd.uniform(0.0, 2 * math.pi, 3)
        b = [torch.cos(math.pi * f[q] * a + p[q]) for q, a in enumerate((x, y, z))]
        v = v * (1.0 + 0.1 * b[2][:, None, None] * b[1][None, :, None] * b[0][None, None])
        v = torch.sqrt((v + 27.0 * _randn(dims[::-1], g)) ** 2 + (27.0 * _randn(dims[::-1], g)) ** 2)
        v = v.round().clamp(0, 4095)
        return v.to(torch.int16) if dtype == "u16" else v
    v = torch.full(dims[::-1], 0.2, device=DEV)
    ext = np.array(dims, np.float64)
    stack = []
    for _ in range(4):
        d = rnd.normal(size=3)
        stack.append((ext * rnd.uniform(0.2, 0.8, 3), d / np.linalg.norm(d), 4.0, 0))
    while stack:
        p0, d, r, gen = stack.pop()
        p1 = np.clip(p0 + d * rnd.uniform(18.0, 40.0) * 0.9 ** gen, 2.0, ext - 2.0)
        lo = np.maximum(np.floor(np.minimum(p0, p1) - r - 2).astype(int), 0)
        hi = np.minimum(np.ceil(np.maximum(p0, p1) + r + 2).astype(int), np.array(dims) - 1)
        ax = [torch.arange(lo[q], hi[q] + 1, device=DEV, dtype=torch.float32) + 0.5 - float(p0[q]) for q in range(3)]
        X, Y, Z = ax[0][None, None], ax[1][None, :, None], ax[2][:, None, None]
        e = p1 - p0
        t = ((X * e[0] + Y * e[1] + Z * e[2]) / max(float(e @ e), 1e-12)).clamp(0.0, 1.0)
        dist = ((X - t * e[0]) ** 2 + (Y - t * e[1]) ** 2 + (Z - t * e[2]) ** 2).sqrt()
        sub = v[lo[2]:hi[2] + 1, lo[1]:hi[1] + 1, lo[0]:hi[0] + 1]
        torch.maximum(sub, 0.2 + 0.6 * (r + 0.5 - dist).clamp(0.0, 1.0), out=sub)
        if gen + 1 < 5:
            for _ in range(2):
                nd = d + 0.6 * rnd.normal(size=3)
                stack.append((p1, nd / np.linalg.norm(nd), max(1.0, 0.8 * r), gen + 1))
    return v + 0.03 * _randn(dims[::-1], g)


WINDOWS = {
    "t1": (((0.05, 0.12), 0.02, (0.30, 0.55, 1.00)), ((0.12, 0.18), 0.05, (0.95, 0.62, 0.52)),
           ((0.18, 0.35), 0.08, (1.00, 0.95, 0.85))),
    "head": (((0.19, 0.34), 0.04, (0.30, 0.55, 1.00)), ((0.50, 0.67), 0.08, (0.95, 0.62, 0.52)),
             ((0.82, 1.00), 0.15, (1.00, 0.95, 0.85))),
    "vessel": (((0.45, 1.00), 0.20, (1.00, 0.30, 0.25)),),
}


def _table(phantom, mode, rows, rnd):
    """(rows, 256, 4) RGBA: one trapezoid per tissue window, scaled along the second axis."""
    x = np.arange(TABLE_W) / (TABLE_W - 1.0)
    tf = np.zeros((rows, TABLE_W, 4))
    for (lo, hi), a, rgb in WINDOWS[phantom]:
        a = a * rnd.uniform(0.9, 1.1)
        trap = np.clip(np.minimum(x - lo, hi - x) / 0.02, 0.0, 1.0) * a
        take = trap > tf[0, :, 3]
        tf[:, take, :3] = rgb
        tf[:, take, 3] = trap[take]
    if rows > 1:
        v = np.arange(rows) / (rows - 1.0)
        tf[:, :, 3] *= (np.clip(0.2 + 16.0 * v, 0, 1) if mode == 1 else 0.15 + 0.85 * np.clip(v / 0.33, 0, 1))[:, None]
    return tf.astype(np.float32)


def _camera(dims, sp, az, el, W, H):
    """Orbit camera at twice the largest extent, 30 degrees high, in FP64, rounded once."""
    ext = np.asarray(dims, np.float64) * sp
    a, e = math.radians(az), math.radians(el)
    c = ext / 2.0
    eye = c + 2.0 * ext.max() * np.array([math.cos(e) * math.sin(a), math.sin(e), math.cos(e) * math.cos(a)])
    fwd = (c - eye) / np.linalg.norm(c - eye)
    r = np.cross(fwd, [0.0, 1.0, 0.0])
    r /= np.linalg.norm(r)
    th = math.tan(math.radians(15.0))
    return np.concatenate([eye, fwd, r * th * W / H, np.cross(r, fwd) * th]).astype(np.float32)


def _scene(case, seed, index=0):
    """Seeded inputs of one volume of the case: volume, cameras, table, uniforms."""
    g, rnd = _gen(seed * 16 + index), np.random.default_rng([int(seed), index])
    k = (1.0, 0.75, 1.25, 0.5)[index]
    dims = tuple(max(24, int(case[a] * k)) for a in ("nx", "ny", "nz"))
    if case["cohort"]:
        dims = COHORT[index]
    sp = (1.0, 1.0, case["sz"])
    az, el = rnd.uniform(0, 360), rnd.uniform(-30, 30)
    cams = np.stack([_camera(dims, sp, az + 360.0 * i / case["cams"], el, case["W"], case["H"])
                     for i in range(case["cams"])])
    mode = case["mode"]
    fixed = dict(tf_mode=mode, grad_mod=1 if mode == 0 else 0, shading=1, kappa_ref=0.02, w_max=3.0,
                 et_threshold=0.99, step_vox=case["step"])
    s = dict(dims=dims, sp=sp, cams=cams, fixed=fixed, tf=_table(case["phantom"], mode, case["rows"], rnd),
             par=np.array([case["gamma"], 0.3, 0.7, 0.2, 1.0], np.float32),
             vol=_volume(case["phantom"], case["dtype"], dims, g, rnd))
    if case["second"]:
        s["second"] = _volume("head", "f32", dims, g, rnd)
    if case["kind"] in ("grad", "fit"):
        s["dl"] = _randn((case["cams"], case["H"], case["W"], 4), g)
        s["target"] = torch.rand((case["cams"], case["H"], case["W"], 4), generator=g, device=DEV)
    return s


def _sigmas(case):
    return tuple(float(x) for x in case["sigmas"].split(",")) if case["sigmas"] else ()


def _uniforms(s):
    return dict(s["fixed"], **dict(zip(ag.PARAM_NAMES, (float(x) for x in s["par"]))))


def _norm32(vol):
    """I_norm as the loader defines it: float32 (x - min) / (max - min)."""
    v = vol.to(torch.float32)
    return (v - v.min()) / (v.max() - v.min())


def _ready(ctx, case, s, tissue=True):
    """The volume loaded and its morphology (and second channel) built."""
    vid = ctx.load_volume(s["vol"], s["sp"])
    if case["brick"] != 8:
        ctx.set_brick_size(vid, case["brick"])
    if not case["derived"]:
        ctx.set_derived_budget(0)
    ctx.precompute_morphology(vid, () if case["kind"] == "vessels" else _sigmas(case))
    if case["second"]:
        ctx.load_second_channel(vid, s["second"])
    if tissue:
        ctx.set_tissue_params(vid, s["tf"], **_uniforms(s))
    return vid


def prepare(case, seed):
    kind, W, H, n = case["kind"], case["W"], case["H"], case["cams"]
    ctx = pkg.Context(0)
    st = dict(case=case, ctx=ctx)
    if kind == "batch":
        views, st["out"] = [], []
        for i in range(case["volumes"]):
            s = _scene(case, seed, i)
            vid = _ready(ctx, case, s)
            out = torch.empty((n, H, W, 4), device=DEV)
            st["out"].append(out)
            views += [(vid, s["cams"][k], out[k], W, H) for k in range(n)]
        st["batch"] = ctx.batch_create(views)
        return st
    s = _scene(case, seed)
    st["s"] = s
    if kind == "open":
        v = s["vol"].cpu().numpy()
        st["host"] = v.view(np.uint16) if case["dtype"] == "u16" else v
        if case["second"]:
            st["host2"] = s["second"].cpu().numpy()
        st["out"] = torch.empty((n, H, W, 4), device=DEV)
        del s["vol"]
        return st
    st["vid"] = _ready(ctx, case, s, tissue=kind not in ("vessels", "clean"))
    if kind == "frame":
        st["out"] = torch.empty((n, H, W, 4), device=DEV)
    if kind == "clean" or (kind == "grad" and case["autograd"]):
        st["norm"] = _norm32(s["vol"])
    if kind in ("grad", "fit"):
        st["tf"] = torch.from_numpy(s["tf"]).to(DEV).requires_grad_(True)
        st["par"] = torch.from_numpy(s["par"]).requires_grad_(kind == "grad")
        if "norm" in st:
            st["norm"].requires_grad_(True)
        if kind == "grad" and not case["autograd"]:
            st["image"] = torch.empty((n, H, W, 4), device=DEV)
            st["rays"] = torch.empty((n, H, W, 2), device=DEV)
    s.pop("vol")
    return st


def run(st):
    case, ctx, kind = st["case"], st["ctx"], st["case"]["kind"]
    W, H = case["W"], case["H"]
    if kind == "batch":
        ctx.batch_render(st["batch"], packet_w=4, warps_per_block=4, graph=True)
        return st["out"]
    s = st["s"]
    if kind == "frame":
        if case["slider"]:
            ctx.set_tissue_params(st["vid"], s["tf"], **_uniforms(s))
        return ctx.render(st["vid"], s["cams"], W, H, out=st["out"])
    if kind == "grad" and not case["autograd"]:
        img = ctx.render(st["vid"], s["cams"], W, H, out=st["image"], ray_state=st["rays"])
        dtf, dpar, dvol = ctx.render_backward(st["vid"], s["cams"], W, H, s["dl"], ray_state=st["rays"])
        return {"image": img, "dtf": dtf, "dpar": dpar, "dvol": dvol}
    if kind == "grad":
        img = ag.render(ctx, st["vid"], st["tf"], st["par"], s["cams"], W, H, s["fixed"], norm_volume=st["norm"])
        dtf, dpar, dvol = torch.autograd.grad(img, (st["tf"], st["par"], st["norm"]), s["dl"])
        return {"image": img.detach(), "dtf": dtf, "dpar": dpar, "dvol": dvol}
    if kind == "fit":
        img = ag.render(ctx, st["vid"], st["tf"], st["par"], s["cams"], W, H, s["fixed"])
        loss = ((img - s["target"]) ** 2).sum()
        (dtf,) = torch.autograd.grad(loss, (st["tf"],))
        return {"image": img.detach(), "dtf": dtf}
    if kind == "open":
        vid = ctx.load_volume(st["host"], s["sp"])
        if case["brick"] != 8:
            ctx.set_brick_size(vid, case["brick"])
        ctx.precompute_morphology(vid, _sigmas(case))
        if case["second"]:
            ctx.load_second_channel(vid, st["host2"])
        ctx.set_tissue_params(vid, s["tf"], **_uniforms(s))
        img = ctx.render(vid, s["cams"], W, H, out=st["out"])
        ctx.free_volume(vid)
        return img
    if kind == "vessels":
        ctx.precompute_morphology(st["vid"], _sigmas(case))
        return ctx.get_vesselness(st["vid"])
    ctx.set_normalized(st["vid"], st["norm"])
    ctx.prefilter(st["vid"], case["filter"], 1.2)
    hist, peaks = ctx.tissue_histogram(st["vid"], 8, 200)
    return {"norm": ctx.get_normalized(st["vid"]), "hist": hist, "peaks": peaks}


# ------------------------------------------------------------------ work

def _dense(case, dims):
    """Sample points of one view: rays through the volume's box, from a coarse grid of pixels."""
    sp = (1.0, 1.0, case["sz"])
    W, H, g = case["W"], case["H"], 48
    cam = _camera(dims, sp, 30.0, 20.0, W, H).astype(np.float64)
    a = 2 * (np.arange(g) + 0.5) / g - 1
    d = cam[3:6] + a[:, None, None] * cam[6:9] + a[None, :, None] * cam[9:12]
    d /= np.linalg.norm(d, axis=-1, keepdims=True)
    with np.errstate(divide="ignore"):
        t = np.stack([-cam[:3] / d, (np.asarray(dims) * sp - cam[:3]) / d])
    chord = np.maximum(t.max(0).min(-1) - t.min(0).max(-1), 0.0)
    return float(chord.mean()) / (case["step"] * min(sp)) * W * H


def work(case):
    dims = (case["nx"], case["ny"], case["nz"])
    vox = dims[0] * dims[1] * dims[2]
    px = case["W"] * case["H"] * case["cams"]
    raw = vox * (2 if case["dtype"] == "u16" else 4)
    table = 16 * TABLE_W * case["rows"]
    kind, channels = case["kind"], 2 if case["mode"] == 2 else 1
    samples = VISIBLE[case["phantom"]] * _dense(case, dims) * case["cams"]
    frame = {"bytes": 4 * vox * channels + table + 16 * px, "flops": 303 * samples}
    n_sig = len(_sigmas(case))
    vessel = sum((2 * math.ceil(4 * x) + 1) * 6 + 200 for x in _sigmas(case)) * vox
    if kind == "frame":
        return frame
    if kind == "batch":
        if case["cohort"]:
            boxes = COHORT[:case["volumes"]]
        else:
            boxes = [tuple(int(x * k) for x in dims) for k in (1.0, 0.75, 1.25, 0.5)[:case["volumes"]]]
        return {"bytes": sum(4 * b[0] * b[1] * b[2] + table + 16 * px for b in boxes),
                "flops": sum(303 * VISIBLE[case["phantom"]] * _dense(case, b) * case["cams"] for b in boxes)}
    if kind == "grad":
        return {"bytes": frame["bytes"] + 4 * vox + table + 16 * px, "flops": 3 * frame["flops"]}
    if kind == "fit":
        return {"bytes": frame["bytes"] + table + 32 * px, "flops": 2.5 * frame["flops"]}
    if kind == "open":
        return {"bytes": raw + frame["bytes"], "flops": frame["flops"] + vessel}
    if kind == "vessels":
        return {"bytes": 8 * vox, "flops": vessel}
    return {"bytes": 8 * vox, "flops": (27 if case["filter"] == "median" else 66) * vox}


# ------------------------------------------------------------------ 64-bit statement

def _shift(v, axis, k):
    """v at index i + k along `axis`, clamped to the edge."""
    n = v.shape[axis]
    return v.index_select(axis, (torch.arange(n, device=v.device) + k).clamp(0, n - 1))


def _channels(I, sp):
    """(nvox, 10): I, its central differences and second differences, mm units."""
    ax = (2, 1, 0)
    g = [(_shift(I, ax[q], 1) - _shift(I, ax[q], -1)) / (2 * sp[q]) for q in range(3)]
    h = [(_shift(I, ax[q], 1) - 2 * I + _shift(I, ax[q], -1)) / sp[q] ** 2 for q in range(3)]
    for p, q in ((0, 1), (0, 2), (1, 2)):
        d = _shift(I, ax[p], 1) - _shift(I, ax[p], -1)
        h.append((_shift(d, ax[q], 1) - _shift(d, ax[q], -1)) / (4 * sp[p] * sp[q]))
    return torch.stack([I] + g + h, -1).reshape(-1, 10)


def _gauss(v, sigma):
    R = math.ceil(4 * sigma)
    w = np.exp(-np.arange(-R, R + 1) ** 2 / (2.0 * sigma * sigma))
    w /= w.sum()
    for axis in (2, 1, 0):
        v = sum(float(w[t + R]) * _shift(v, axis, t) for t in range(-R, R + 1))
    return v


def _eig3(H):
    """Eigenvalues of symmetric 3x3 matrices (xx yy zz xy xz yz) by cyclic Jacobi rotations."""
    a = {(0, 0): H[0], (1, 1): H[1], (2, 2): H[2], (0, 1): H[3], (0, 2): H[4], (1, 2): H[5]}
    key = lambda p, q: (p, q) if p <= q else (q, p)  # noqa: E731
    for _ in range(7):
        for p, q, r in ((0, 1, 2), (0, 2, 1), (1, 2, 0)):
            apq = a[(p, q)]
            safe = torch.where(apq == 0, torch.ones_like(apq), apq)
            th = (a[(q, q)] - a[(p, p)]) / (2 * safe)
            t = torch.where(th >= 0, 1.0, -1.0) / (th.abs() + (th * th + 1).sqrt())
            t = torch.where(apq == 0, torch.zeros_like(t), t)
            c = 1 / (t * t + 1).sqrt()
            s = t * c
            rp, rq = a[key(r, p)], a[key(r, q)]
            a[(p, p)], a[(q, q)] = a[(p, p)] - t * apq, a[(q, q)] + t * apq
            a[(p, q)] = torch.zeros_like(apq)
            a[key(r, p)], a[key(r, q)] = c * rp - s * rq, s * rp + c * rq
    return torch.stack([a[(0, 0)], a[(1, 1)], a[(2, 2)]])


def _vesselness(I, sigmas):
    """Multi-scale bright-vessel response (Frangi 1998), alpha = beta = 1/2, c = max S / 2."""
    V = torch.zeros_like(I)
    for sg in sigmas:
        C = _channels(_gauss(I, sg), (1.0, 1.0, 1.0))
        H = [C[:, q].reshape(I.shape) * (sg * sg) for q in range(4, 10)]
        S2 = H[0] ** 2 + H[1] ** 2 + H[2] ** 2 + 2 * (H[3] ** 2 + H[4] ** 2 + H[5] ** 2)
        lam = _eig3(H)
        lam = lam.gather(0, lam.abs().argsort(0))
        l1, l2, l3 = lam
        ok = (l2 < 0) & (l3 < 0)
        l2s, l3s = torch.where(ok, l2, torch.full_like(l2, -1.0)), torch.where(ok, l3, torch.full_like(l3, -1.0))
        c2 = S2.max() / 4
        v = ((1 - torch.exp(-2 * (l2s / l3s) ** 2)) * torch.exp(-2 * l1 * l1 / (l2s * l3s))
             * (1 - torch.exp(-S2 / (2 * c2))))
        V = torch.maximum(V, torch.where(ok, v, torch.zeros_like(v)))
    return V


def _rays(cam, W, H, dims, sp, dt):
    cam = torch.from_numpy(cam.astype(np.float64)).to(DEV)
    a = 2 * (torch.arange(W, device=DEV, dtype=torch.float64) + 0.5) / W - 1
    b = 1 - 2 * (torch.arange(H, device=DEV, dtype=torch.float64) + 0.5) / H
    d = cam[3:6] + a[None, :, None] * cam[6:9] + b[:, None, None] * cam[9:12]
    d = (d / (d * d).sum(-1, keepdim=True).sqrt()).reshape(-1, 3)
    box = torch.tensor([n * s for n, s in zip(dims, sp)], device=DEV, dtype=torch.float64)
    ta, tb = -cam[:3] / d, (box - cam[:3]) / d
    t0 = torch.minimum(ta, tb).max(-1).values.clamp(min=0.0)
    t1 = torch.maximum(ta, tb).min(-1).values
    ns = torch.where(t0 < t1, torch.ceil((t1 - t0) / dt - 0.5), torch.zeros_like(t0)).clamp(min=0).to(torch.int64)
    return cam[:3], d, t0, ns


def _image(F, V, tf, par, s, W, H, gmax, dl=None, most=3 << 20):
    """(n, H, W, 4) of the scene in 64 bits; with `dl` the gradients of (image * dl).sum() in
    the leaves among F, tf and par are accumulated on the way."""
    dims, sp, fx = s["dims"], s["sp"], s["fixed"]
    dt = fx["step_vox"] * min(sp)
    nx, ny, nz = dims
    size = torch.tensor(dims, device=DEV, dtype=torch.float64)
    spt = torch.tensor(sp, device=DEV, dtype=torch.float64)
    h, w = tf.shape[:2]
    images = []
    for v in range(s["cams"].shape[0]):
        eye, d, t0, ns = _rays(s["cams"][v], W, H, dims, sp, dt)
        img = torch.zeros((W * H, 4), device=DEV, dtype=torch.float64)
        order = torch.argsort(ns)
        lens = ns[order].cpu().numpy()
        at = int(np.searchsorted(lens, 1))
        while at < len(lens):
            end = min(len(lens), at + max(256, most // max(int(lens[min(len(lens) - 1, at + most // int(lens[-1]))]), 1)))
            sel, K = order[at:end], int(lens[end - 1])
            at = end
            kk = torch.arange(K, device=DEV, dtype=torch.float64)
            inside = kk[None] < ns[sel][:, None]
            with torch.no_grad():
                t = t0[sel][:, None] + (kk[None] + 0.5) * dt
                u = ((eye + t[..., None] * d[sel][:, None]) / spt - 0.5)[inside]
                u = torch.minimum(u.clamp(min=0.0), size - 1)
                i0 = torch.minimum(u.floor(), size - 2)
                f, i0 = u - i0, i0.to(torch.int64)
                base = (i0[:, 2] * ny + i0[:, 1]) * nx + i0[:, 0]
                dirs = d[sel][:, None].expand(-1, K, -1)[inside]
            fld, vv = 0.0, 0.0
            for c in range(8):
                b = (c & 1, (c >> 1) & 1, c >> 2)
                wt = 1.0
                for q in range(3):
                    wt = wt * (f[:, q] if b[q] else 1 - f[:, q])
                idx = base + (b[2] * ny + b[1]) * nx + b[0]
                fld = fld + wt[:, None] * F[idx]
                if V is not None:
                    vv = vv + wt * V.reshape(-1)[idx]
            I, g = fld[:, 0], fld[:, 1:4]
            gg = (g * g).sum(-1)
            some = gg > 0
            ggs = torch.where(some, gg, torch.ones_like(gg))
            gmag = torch.where(some, ggs.sqrt(), torch.zeros_like(gg))
            gn = gmag / gmax
            xs = I.clamp(0, 1) * (w - 1)
            j = xs.detach().floor().clamp(max=w - 2).to(torch.int64)
            tx = (xs - j)[:, None]
            if h == 1:
                rgba = tf[0][j] * (1 - tx) + tf[0][j + 1] * tx
            else:
                ys = (gn if fx["tf_mode"] == 1 else vv).clamp(0, 1) * (h - 1)
                k = ys.detach().floor().clamp(max=h - 2).to(torch.int64)
                ty = (ys - k)[:, None]
                flat, e = tf.reshape(-1, 4), k * w + j
                rgba = ((flat[e] * (1 - tx) + flat[e + 1] * tx) * (1 - ty)
                        + (flat[e + w] * (1 - tx) + flat[e + w + 1] * tx) * ty)
            gx, gy, gz = g[:, 0], g[:, 1], g[:, 2]
            hs = [fld[:, 4 + q] for q in range(6)]
            ghg = (hs[0] * gx * gx + hs[1] * gy * gy + hs[2] * gz * gz
                   + 2 * (hs[3] * gx * gy + hs[4] * gx * gz + hs[5] * gy * gz))
            kappa = torch.where(some, ghg / ggs, torch.zeros_like(gg))
            wk = (1 + par[0] * kappa / fx["kappa_ref"]).clamp(0.0, fx["w_max"])
            raw = par[4] * rgba[:, 3] * wk
            if fx["grad_mod"]:
                raw = raw * gn.clamp(max=1.0)
            alpha = raw.clamp(0.0, 1.0)
            cosv = torch.where(some, (g * dirs).sum(-1) / ggs.sqrt(), torch.zeros_like(gg)).abs()
            col = rgba[:, :3] * (par[1] + par[2] * cosv)[:, None] + (par[3] * cosv ** 16)[:, None]
            al = torch.zeros(inside.shape, device=DEV, dtype=torch.float64).masked_scatter(inside, alpha)
            with torch.no_grad():
                acc = 1 - torch.cumprod(1 - al, 1)
                before = torch.cat([torch.zeros_like(acc[:, :1]), acc[:, :-1]], 1)
                live = before < fx["et_threshold"]  # samples up to the stopping one
            al = torch.where(live, al, torch.zeros_like(al))
            trans = torch.cumprod(1 - al, 1)
            front = torch.cat([torch.ones_like(trans[:, :1]), trans[:, :-1]], 1)
            wgt = front * al
            rows = inside.nonzero()[:, 0]
            C = torch.zeros((len(sel), 3), device=DEV, dtype=torch.float64).index_add(0, rows, wgt[inside][:, None] * col)
            px = torch.cat([C, 1 - trans[:, -1:]], 1)
            img[sel] = px.detach()
            if dl is not None:
                (px * dl[v].reshape(-1, 4)[sel]).sum().backward()
        images.append(img.reshape(H, W, 4))
    return torch.stack(images)


def _exact_scene(case, seed, index=0):
    s = _scene(case, seed, index)
    I = s["vol"].to(torch.float64)
    I = (I - I.min()) / (I.max() - I.min())
    V = None
    if case["second"]:
        V = s["second"].to(torch.float64)
        V = (V - V.min()) / (V.max() - V.min())
    elif case["mode"] == 2:
        V = _vesselness(I, _sigmas(case))
    F = _channels(I, s["sp"])
    gmax = (F[:, 1:4] ** 2).sum(-1).max().sqrt()
    return s, I, F, V, gmax


def exact(case, seed):
    kind, W, H = case["kind"], case["W"], case["H"]
    par64 = lambda s: torch.from_numpy(s["par"].astype(np.float64)).to(DEV)  # noqa: E731
    tf64 = lambda s: torch.from_numpy(s["tf"].astype(np.float64)).to(DEV)  # noqa: E731
    if kind == "batch":
        out = []
        for i in range(case["volumes"]):
            s, _, F, V, gmax = _exact_scene(case, seed, i)
            out.append(_image(F, V, tf64(s), par64(s), s, W, H, gmax))
        return out
    if kind == "vessels":
        v = _scene(case, seed)["vol"].to(torch.float64)
        return _vesselness((v - v.min()) / (v.max() - v.min()), _sigmas(case))
    if kind == "clean":
        n = _norm32(_scene(case, seed)["vol"]).to(torch.float64)
        if case["filter"] == "gauss":
            return {"norm": _gauss(n, float(np.float32(1.2))), "hist": None, "peaks": None}
        near = torch.stack([_shift(_shift(_shift(n, 0, a), 1, b), 2, c)
                            for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)])
        return {"norm": near.median(0).values, "hist": None, "peaks": None}
    s, I, F, V, gmax = _exact_scene(case, seed)
    if kind in ("frame", "open"):
        return _image(F, V, tf64(s), par64(s), s, W, H, gmax)
    tf, par = tf64(s).requires_grad_(True), par64(s)
    if kind == "fit":
        with torch.no_grad():
            img = _image(F, V, tf, par, s, W, H, gmax)
        _image(F, V, tf, par, s, W, H, gmax, dl=2 * (img - s["target"].to(torch.float64)))
        return {"image": img, "dtf": tf.grad}
    par.requires_grad_(True)
    F = F.detach().requires_grad_(True)
    img = _image(F, V, tf, par, s, W, H, gmax, dl=s["dl"].to(torch.float64), most=1 << 20)
    I = I.detach().requires_grad_(True)
    _channels(I, s["sp"]).backward(F.grad)
    return {"image": img, "dtf": tf.grad, "dpar": par.grad, "dvol": I.grad}
