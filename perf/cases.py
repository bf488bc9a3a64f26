"""Timed cases of the volume renderer, through its public entry points.

The cubes are what the renderer is for: HI-like spectral cubes of unit noise with
compact Gaussian sources (5-20 sigma) and a continuum ripple along the channel axis,
made on the GPU from a seed.  Sizes are those of the workloads of this repository
(the 128^3 and 256^3 cubes, the 1024 x 1024 x 2048 survey, the 1721 x 1721 x 1025
static render, the 2048 x 2048 x 1024 cube on a 5 x 5 wall) and of its tests.

Kinds of case:
  frame    a viewer's frame: new camera(s), then a render of a loaded cube;
  load     a cube already on the device is loaded and its first frame rendered;
  step     a gradient step: forward render of several views, loss, gradients of the
           transfer function and the voxels, through autograd;
  pyramid  zoom levels of a finished high-resolution render.
"""
import math

import numpy as np
import torch

import paper_1012_2909_gb300 as vr

STEP, ERT, VMIN, VMAX = 0.5, 0.99, -1.0, 20.0
DEV = "cuda"
STORE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


# ------------------------------------------------------------------ the cases
def _frame(name, dims, image, mode, storage, path="auto", view="orbit", az=10.0, brick=128, cols=1, rows=1):
    return dict(name=name, kind="frame", nx=dims[0], ny=dims[1], nz=dims[2], width=image[0], height=image[1],
                mode=mode, storage=storage, path=path, view=view, az=az, brick=brick, cols=cols, rows=rows)


SURVEY, HIPASS, WALL = (1024, 1024, 2048), (1721, 1721, 1025), (2048, 2048, 1024)


def listed():
    return [
        # a quick look at a sub-cube around one source: ragged, two small views; launches are all there is
        _frame("thumbnail_mip_f16", (96, 80, 72), (64, 48), "mip", "f16", az=35.0, brick=32, cols=2),
        # the small interactive view: a 128^3 cut-out in a 512 x 512 window
        _frame("small_composite_f32", (128, 128, 128), (512, 512), "composite", "f32", view="ortho", az=30.0),
        # the survey cube in a full-HD viewer: the composite view and the MIP view of an orbit frame
        _frame("survey_composite_f16", SURVEY, (1920, 1080), "composite", "f16", az=30.0),
        _frame("survey_mip_f16", SURVEY, (1920, 1080), "mip", "f16", az=30.0),
        # the same frame by parts: per-brick partial images folded, and brick layers with carried state
        _frame("survey_sortlast_f16", SURVEY, (1920, 1080), "composite", "f16", path="sortlast", az=30.0),
        _frame("survey_layered_bf16", SURVEY, (1920, 1080), "composite", "bf16", path="layered", az=60.0),
        # a high-resolution static render of a full-precision cube, ragged on every axis
        _frame("static_composite_f32", HIPASS, (3000, 3000), "composite", "f32", az=30.0),
        _frame("static_mip_f32", HIPASS, (3000, 3000), "mip", "f32", az=30.0),
        # the tiled display: 25 off-axis panels of 1920 x 1080 in one call
        _frame("wall_mip_f16", WALL, (1920, 1080), "mip", "f16", az=20.0, cols=5, rows=5),
        # opening a cube that another program left on the device, up to its first frame
        dict(name="load_survey_f16", kind="load", nx=1024, ny=1024, nz=2048, width=1920, height=1080,
             mode="composite", storage="f16", path="auto", view="orbit", az=0.0, brick=128, cols=1, rows=1),
        # fitting a transfer function (and the voxels) to images: 16 views at 512 x 512, forward and backward
        dict(name="fit_step_f32", kind="step", nx=256, ny=256, nz=256, width=512, height=512, views=16,
             mode="composite", storage="f32", brick=128),
        # zoom levels of the 8000 x 8000 static render, cut into 256 x 256 tiles
        dict(name="pyramid_8000", kind="pyramid", width=8000, height=8000, tile=256),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("frame", "frame", "frame", "parts", "wall", "load", "step", "pyramid"))
    if kind == "pyramid":
        return dict(kind="pyramid", width=_log(rng, 300, 8000), height=_log(rng, 300, 8000),
                    tile=rng.choice((0, 0, 256, 512)))
    if kind == "step":
        n = [_log(rng, 64, 256) for _ in range(3)]
        return dict(kind="step", nx=n[0], ny=n[1], nz=n[2], width=_log(rng, 100, 512), height=_log(rng, 100, 512),
                    views=_log(rng, 1, 16), mode=rng.choice(("composite", "composite", "mip")),
                    storage=rng.choice(("f32", "f32", "f16")), brick=rng.choice((32, 64, 128)))
    n = [_log(rng, 64, 1500) for _ in range(3)]
    while n[0] * n[1] * n[2] > SURVEY[0] * SURVEY[1] * SURVEY[2]:
        n[rng.randrange(3)] //= 2
    c = dict(kind="load" if kind == "load" else "frame", nx=n[0], ny=n[1], nz=n[2], width=_log(rng, 64, 3000),
             height=_log(rng, 48, 2200), mode=rng.choice(("composite", "mip")),
             storage=rng.choice(("f32", "f16", "f16", "bf16")), path="auto",
             view=rng.choice(("orbit", "orbit", "ortho")), az=round(rng.uniform(0.0, 360.0), 2),
             brick=128 if max(n) > 256 else rng.choice((32, 64, 128)), cols=1, rows=1)
    if kind == "parts":
        c.update(mode="composite", path=rng.choice(("sortlast", "layered")), width=min(c["width"], 1920),
                 height=min(c["height"], 1200))
    if kind == "wall":
        c.update(cols=rng.randint(2, 5), rows=rng.randint(1, 5), width=_log(rng, 64, 960), height=_log(rng, 48, 540))
    return c


# ------------------------------------------------------------------ inputs
def _cube(c, seed):
    """Unit noise + ripple along z + Gaussian sources, float32 (nz, ny, nx) on the device."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    vol = torch.randn((nz, ny, nx), generator=g, device=DEV)
    rng = np.random.default_rng(int(seed))
    z = torch.arange(nz, device=DEV, dtype=torch.float32)
    vol += (0.5 * torch.sin((z + 0.5) * (2 * math.pi / 256.0) + float(rng.uniform(0, 2 * math.pi))))[:, None, None]
    nsrc = max(20, round(nx * ny * nz * 2000 / 2 ** 31))
    amp = rng.uniform(5.0, 20.0, nsrc)
    centre = rng.uniform(0.0, 1.0, (nsrc, 3)) * np.array([nx, ny, nz])
    sig = np.stack([rng.uniform(2.0, 6.0, nsrc)] * 2 + [rng.uniform(4.0, 20.0, nsrc)], 1) / 2.3548
    prof, spans = [], []
    for a, n in enumerate((nx, ny, nz)):
        half = int(math.ceil(4 * sig[:, a].max()))
        off = np.floor(centre[:, a, None]) + np.arange(-half, half + 1)
        p = np.exp(-0.5 * ((off + 0.5 - centre[:, a, None]) / sig[:, a, None]) ** 2)
        if a == 0:
            p *= amp[:, None]
        prof.append(torch.from_numpy(p.astype(np.float32)).to(DEV))
        first = off[:, 0].astype(int)
        lo = np.maximum(first, 0)
        hi = np.minimum(first + 2 * half + 1, n)
        spans.append(list(zip(lo.tolist(), hi.tolist(), (lo - first).tolist())))
    for s in range(nsrc):  # one by one: overlapping sources add in a fixed order
        (x0, x1, xo), (y0, y1, yo), (z0, z1, zo) = (spans[a][s] for a in range(3))
        if x0 >= x1 or y0 >= y1 or z0 >= z1:
            continue
        px, py = prof[0][s, xo:xo + x1 - x0], prof[1][s, yo:yo + y1 - y0]
        pz = prof[2][s, zo:zo + z1 - z0]
        vol[z0:z1, y0:y1, x0:x1] += pz[:, None, None] * (py[:, None] * px)
    return vol


def _table(n=256):
    """The viewer's default table: an opacity ramp with dark purple - teal - yellow colours."""
    x = np.linspace(0.0, 1.0, n)
    anchors = np.array([[0.267, 0.005, 0.329], [0.229, 0.322, 0.546], [0.128, 0.567, 0.551],
                        [0.369, 0.789, 0.383], [0.993, 0.906, 0.144]])
    rgb = [np.interp(x, np.linspace(0.0, 1.0, len(anchors)), anchors[:, k]) for k in range(3)]
    return np.stack(rgb + [x], axis=1).astype(np.float32)


def _cam(t, eye, right, up, fwd, win, w, h):
    return dict(type=t, eye=[float(v) for v in eye], right=[float(v) for v in right], up=[float(v) for v in up],
                fwd=[float(v) for v in fwd], win=[float(v) for v in win], width=w, height=h)


def _look(dims, fwd, w, h):
    """Perspective view of the whole cube: eye two half-diagonals before its centre, 60 degrees."""
    d = np.array(dims, float)
    f = np.asarray(fwd, float) / np.linalg.norm(fwd)
    hint = np.array([0.0, 1.0, 0.0]) if abs(f[1]) <= 0.99 else np.array([1.0, 0.0, 0.0])
    right = np.cross(hint, f)
    right /= np.linalg.norm(right)
    t = math.tan(math.radians(30.0))
    return _cam(1, d / 2 - np.linalg.norm(d) * f, right, np.cross(f, right), f, (-t * w / h, t * w / h, -t, t), w, h)


def _cameras(c):
    """The case's views; several columns and rows are the off-axis panels of one view."""
    dims, w, h = (c["nx"], c["ny"], c["nz"]), c["width"] * c["cols"], c["height"] * c["rows"]
    a = math.radians(c["az"])
    if c["view"] == "orbit":
        full = _look(dims, (math.sin(a), 0.0, math.cos(a)), w, h)
    else:  # orthographic, turned by az about y and 20 degrees about x
        b = math.radians(20.0)
        m = (np.array([[1, 0, 0], [0, math.cos(b), -math.sin(b)], [0, math.sin(b), math.cos(b)]]) @
             np.array([[math.cos(a), 0, math.sin(a)], [0, 1, 0], [-math.sin(a), 0, math.cos(a)]]))
        d = np.array(dims, float)
        r = np.linalg.norm(d) / 2
        full = _cam(0, d / 2 - 2 * r * m[:, 2], m[:, 0], m[:, 1], m[:, 2], (-r * w / h, r * w / h, -r, r), w, h)
    l, r, b, t = full["win"]
    return [dict(full, width=c["width"], height=c["height"],
                 win=[l + (r - l) * i / c["cols"], l + (r - l) * (i + 1) / c["cols"],
                      t - (t - b) * (j + 1) / c["rows"], t - (t - b) * j / c["rows"]])
            for j in range(c["rows"]) for i in range(c["cols"])]


def _step_cameras(c, seed):
    rng = np.random.default_rng(int(seed) + 7)
    return [_look((c["nx"], c["ny"], c["nz"]), rng.normal(size=3), c["width"], c["height"])
            for _ in range(c["views"])]


def _target(c, seed):
    """Smooth seeded images to fit."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) + 3)
    low = torch.rand((c["views"], 4, 8, 8), generator=g, device=DEV)
    up = torch.nn.functional.interpolate(low, size=(c["height"], c["width"]), mode="bilinear", align_corners=True)
    return up.permute(0, 2, 3, 1).contiguous()


def _image(c, seed):
    """A finished render: premultiplied, smooth with pixel noise."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    img = torch.rand((c["height"], c["width"], 4), generator=g, device=DEV)
    img[..., :3] *= img[..., 3:]
    return img


def prepare(case, seed):
    c = case
    if c["kind"] == "pyramid":
        return dict(kind="pyramid", r=vr.Renderer(0), image=_image(c, seed), tile=c["tile"])
    if c["kind"] == "step":
        r = vr.VolumeRenderer(0, brick=c["brick"], step=STEP, ert=ERT, vmin=VMIN, vmax=VMAX, storage=c["storage"])
        r.set_camera(_step_cameras(c, seed))
        return dict(kind="step", r=r, mode=c["mode"], target=_target(c, seed),
                    tf=torch.from_numpy(_table()).to(DEV).requires_grad_(),
                    volume=_cube(c, seed).requires_grad_())
    r = vr.Renderer(0, brick=c["brick"], step=STEP, ert=ERT)
    vol = _cube(c, seed)
    r.set_transfer_function(_table(), VMIN, VMAX)
    r.set_path(c["path"])
    s = dict(kind=c["kind"], r=r, mode=c["mode"], cams=_cameras(c), storage=c["storage"])
    if c["kind"] == "load":
        s["volume"] = vol
    else:
        r.load_cube(vol, c["storage"])
    return s


# ------------------------------------------------------------------ one pass
def run(state):
    s, r = state, state["r"]
    if s["kind"] == "pyramid":
        return r.pyramid(s["image"], tile=s["tile"])
    if s["kind"] == "step":
        image = r.render(s["mode"], tf=s["tf"], volume=s["volume"])
        loss = (image - s["target"]).square().mean()
        dtf, dvol = torch.autograd.grad(loss, (s["tf"], s["volume"]))
        return {"image": image.detach(), "dtf": dtf, "dvol": dvol}
    if s["kind"] == "load":
        r.load_cube(s["volume"], s["storage"])
    r.set_camera(s["cams"])
    if s["mode"] == "mip":
        rgba, largest = r.render("mip", with_max=True)
        return {"rgba": rgba, "max": largest}
    return {"rgba": r.render("composite")}


# ------------------------------------------------------------------ what a pass cannot do without
def _mean_samples(cams, dims, most):
    """Mean number of samples a pixel's ray takes in the cube (`most` at most), from a grid of its rays."""
    total, rays = 0.0, 0
    for cam in cams[::max(1, len(cams) // 8)]:
        w, h = cam["width"], cam["height"]
        px = np.arange(0, w, max(1, w // 40)) + 0.5
        py = np.arange(0, h, max(1, h // 40)) + 0.5
        l, r, b, t = cam["win"]
        u, v = np.meshgrid(l + px * (r - l) / w, t - py * (t - b) / h)
        off = u[..., None] * np.array(cam["right"]) + v[..., None] * np.array(cam["up"])
        o = np.array(cam["eye"]) + (off if cam["type"] == 0 else 0 * off)
        d = np.array(cam["fwd"]) + (0 * off if cam["type"] == 0 else off)
        d = d / np.linalg.norm(d, axis=-1, keepdims=True)
        d = np.where(np.abs(d) < 1e-12, 1e-12, d)
        t1, t2 = -o / d, (np.array(dims) - o) / d
        near = np.maximum(np.minimum(t1, t2).max(-1), 0.0)
        total += float(np.minimum(np.maximum(np.maximum(t1, t2).min(-1) - near, 0.0) / STEP, most).sum())
        rays += near.size
    return total / rays


def work(case):
    c = case
    px = c["width"] * c["height"]
    if c["kind"] == "pyramid":
        return {"bytes": 16 * px * (1 + 1 / 3), "flops": 4 * px * (1 + 1 / 3)}
    dims = (c["nx"], c["ny"], c["nz"])
    vox, size = dims[0] * dims[1] * dims[2], STORE[c["storage"]].itemsize
    if c["kind"] == "step":
        cams = _step_cameras(c, 0)
    else:
        cams = _cameras(c)
    # a composite ray ends after about 100 samples of noise (opacity 0.05 each) at ert 0.99
    ends = c["mode"] == "composite" and c.get("path") != "sortlast"
    samples = _mean_samples(cams, dims, 100.0 if ends else math.inf) * px * len(cams)
    # a sample half a voxel on reads about 3.3 voxels that its ray has not read; rays share voxels
    read = vox * (1 - math.exp(-3.3 * samples / vox)) * size
    out = 16 * px * len(cams) + (4 * px * len(cams) if c["mode"] == "mip" else 0)
    if c["kind"] == "load":  # read the cube, write the store, render
        return {"bytes": vox * (4 + size) + read + out, "flops": 40 * samples}
    if c["kind"] == "step":  # forward, backward (recomputed), image gradient read, voxel gradients written
        return {"bytes": 2 * read + 3 * out + 4 * vox, "flops": 200 * samples}
    return {"bytes": read + out, "flops": (28 if c["mode"] == "mip" else 40) * samples}


# ------------------------------------------------------------------ the same in 64 bits, by torch alone
class _Rays:
    """Rays of some pixel rows of a camera in float64: origin, step vector, sample range."""

    def __init__(self, cam, dims, y0, y1):
        f = dict(dtype=torch.float64, device=DEV)
        w, h = cam["width"], cam["height"]
        l, r, b, t = cam["win"]
        u = l + (torch.arange(w, **f) + 0.5) * ((r - l) / w)
        v = t - (torch.arange(y0, y1, **f) + 0.5) * ((t - b) / h)
        off = [(u * cam["right"][a] + (v * cam["up"][a])[:, None]).reshape(-1) for a in range(3)]
        if cam["type"] == 1:
            d = [off[a] + cam["fwd"][a] for a in range(3)]
            inv = 1.0 / torch.sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2])
            d = [x * inv for x in d]
            o = [torch.full_like(off[0], cam["eye"][a]) for a in range(3)]
        else:
            length = math.sqrt(sum(x * x for x in cam["fwd"]))
            d = [torch.full_like(off[0], cam["fwd"][a] / length) for a in range(3)]
            o = [off[a] + cam["eye"][a] for a in range(3)]
        near, far = torch.zeros_like(off[0]), torch.full_like(off[0], math.inf)
        for a in range(3):
            t1, t2 = -o[a] / d[a], (dims[a] - o[a]) / d[a]
            flat = d[a] == 0
            inside = (o[a] >= 0) & (o[a] <= dims[a])
            lo = torch.where(flat, torch.where(inside, -math.inf, math.inf), torch.minimum(t1, t2))
            hi = torch.where(flat, torch.where(inside, math.inf, -math.inf), torch.maximum(t1, t2))
            near, far = torch.maximum(near, lo), torch.minimum(far, hi)
        k0, k1 = torch.ceil(near / STEP), torch.ceil(far / STEP)
        self.count = off[0].numel()
        self.at = torch.nonzero((near < far) & (k1 > k0)).reshape(-1)
        self.o = [x[self.at] for x in o]
        self.e = [x[self.at] * STEP for x in d]
        self.k0, self.k1 = k0[self.at], k1[self.at]


def _corners(dims, p):
    """Weights and clamped indices of the eight voxels around each position."""
    lo, hi, w = [], [], []
    for a in range(3):
        q = p[a] - 0.5
        f = torch.floor(q)
        w.append(q - f)
        i = f.long()
        hi.append((i + 1).clamp_(0, dims[a] - 1))
        lo.append(i.clamp_(0, dims[a] - 1))
    rows = [(z * dims[1] + y) * dims[0] for z in (lo[2], hi[2]) for y in (lo[1], hi[1])]
    return w, [(r + lo[0], r + hi[0]) for r in rows]


def _value(flat, w, idx):
    a = [torch.lerp(flat.index_select(0, i).double(), flat.index_select(0, j).double(), w[0]) for i, j in idx]
    return torch.lerp(torch.lerp(a[0], a[1], w[1]), torch.lerp(a[2], a[3], w[1]), w[2])


def _lookup(tab, v):
    n = tab.shape[0]
    u0 = (v - VMIN) / (VMAX - VMIN)
    x = u0.clamp(0.0, 1.0) * (n - 1)
    i = x.long().clamp_(max=n - 2)
    w = x - i
    lo, hi = tab.index_select(0, i), tab.index_select(0, i + 1)
    return torch.lerp(lo, hi, w[:, None]), i, w, (u0 > 0) & (u0 < 1), hi - lo


def _march(flat, dims, tab, rays, mode, ert, visit=None):
    """Composite (C, A) or maximum and its sample index of every ray; `visit` sees each composite sample."""
    n = rays.at.numel()
    f = dict(dtype=torch.float64, device=DEV)
    state = torch.zeros((n, 4), **f) if mode == "composite" else torch.full((n,), -math.inf, **f)
    trans, best = torch.ones(n, **f), torch.zeros(n, **f)
    live = torch.arange(n, device=DEV)
    o, e, k, k1 = rays.o, rays.e, rays.k0, rays.k1
    st, tr = state.clone(), trans
    bk = best
    steps = 0
    while live.numel():
        p = [o[a] + e[a] * k for a in range(3)]
        w, idx = _corners(dims, p)
        v = _value(flat, w, idx)
        on = k < k1
        if mode == "mip":
            up = on & (v > st)
            st = torch.where(up, v, st)
            bk = torch.where(up, k, bk)
        else:
            c, i, tw, inside, rise = _lookup(tab, v)
            on = on & (1.0 - tr < ert)
            a = torch.where(on, c[:, 3], 0.0)
            if visit is not None:
                visit(live, w, idx, i, tw, inside, rise, c, a, tr, on)
            add = tr * a
            st[:, :3] += add[:, None] * c[:, :3]
            tr = tr * (1.0 - a)
        k = k + 1
        steps += 1
        if steps % 16 == 0:
            keep = k < k1
            if mode == "composite":
                keep &= 1.0 - tr < ert
            if bool((~keep).any()):
                if mode == "mip":
                    state[live], best[live] = st, bk
                    bk = bk[keep]
                else:
                    state[live], trans[live] = st, tr
                    tr = tr[keep]
                st, live, k, k1 = st[keep], live[keep], k[keep], k1[keep]
                o, e = [x[keep] for x in o], [x[keep] for x in e]
    if mode == "composite":
        state[:, 3] = 1.0 - trans
    return state, best


def _chunks(cams, most=6_000_000):
    for ci, cam in enumerate(cams):
        rows = max(1, most // cam["width"])
        for y0 in range(0, cam["height"], rows):
            yield ci, cam, y0, min(cam["height"], y0 + rows)


def _exact_frame(c, seed):
    dims, cams = (c["nx"], c["ny"], c["nz"]), _cameras(c)
    flat = _cube(c, seed).to(STORE[c["storage"]]).reshape(-1)
    tab = torch.from_numpy(_table()).to(DEV).double()
    ert = 2.0 if c["path"] == "sortlast" else ERT  # partial images start afresh: no termination
    h, w = c["height"], c["width"]
    rgba = torch.zeros((len(cams), h, w, 4), dtype=torch.float64, device=DEV)
    largest = torch.full((len(cams), h, w), -math.inf, dtype=torch.float64, device=DEV) if c["mode"] == "mip" else None
    for ci, cam, y0, y1 in _chunks(cams):
        rays = _Rays(cam, dims, y0, y1)
        if not rays.at.numel():
            continue
        got, _ = _march(flat, dims, tab, rays, c["mode"], ert)
        if c["mode"] == "mip":
            largest[ci, y0:y1].view(-1)[rays.at] = got
            got = _lookup(tab, got)[0]
        rgba[ci, y0:y1].view(-1, 4)[rays.at] = got
    return {"rgba": rgba, "max": largest} if c["mode"] == "mip" else {"rgba": rgba}


def _exact_step(c, seed):
    dims, cams = (c["nx"], c["ny"], c["nz"]), _step_cameras(c, seed)
    flat = _cube(c, seed).to(STORE[c["storage"]]).reshape(-1)
    tab = torch.from_numpy(_table()).to(DEV).double()
    target = _target(c, seed).double()
    n = tab.shape[0]
    image = torch.zeros_like(target)
    dvol = torch.zeros(flat.numel(), dtype=torch.float64, device=DEV)
    moments = torch.zeros((2, 4, n), dtype=torch.float64, device=DEV)  # sums of g and of w g per table interval

    def scatter(w, idx, dv):
        for q, (i, j) in enumerate(idx):
            wyz = (w[1] if q & 1 else 1.0 - w[1]) * (w[2] if q & 2 else 1.0 - w[2]) * dv
            dvol.index_add_(0, i, wyz * (1.0 - w[0]))
            dvol.index_add_(0, j, wyz * w[0])

    def to_table(i, tw, g):
        for ch in range(4):
            moments[0, ch] += torch.bincount(i, weights=g[:, ch], minlength=n)
            moments[1, ch] += torch.bincount(i, weights=tw * g[:, ch], minlength=n)

    scale = (n - 1) / (VMAX - VMIN)
    for ci, cam, y0, y1 in _chunks(cams):
        rays = _Rays(cam, dims, y0, y1)
        if not rays.at.numel():
            continue
        got, best = _march(flat, dims, tab, rays, c["mode"], ERT)
        rgba = got if c["mode"] == "composite" else _lookup(tab, got)[0]
        image[ci, y0:y1].view(-1, 4)[rays.at] = rgba
        gi = 2.0 / target.numel() * (rgba - target[ci, y0:y1].reshape(-1, 4)[rays.at])
        if c["mode"] == "mip":
            _, i, tw, inside, rise = _lookup(tab, got)
            to_table(i, tw, gi)
            w, idx = _corners(dims, [rays.o[a] + rays.e[a] * best for a in range(3)])
            scatter(w, idx, (gi * rise).sum(1) * scale * inside)
            continue
        front = torch.zeros((rays.at.numel(), 3), dtype=torch.float64, device=DEV)

        def visit(live, w, idx, i, tw, inside, rise, col, a, tr, on):
            add = tr * a
            f = front.index_select(0, live) + add[:, None] * col[:, :3]
            front[live] = f
            g = gi.index_select(0, live)
            tot = got.index_select(0, live)
            rest = 1.0 - a
            opaque = rest == 0.0  # the ray's last sample: nothing behind it
            rest = torch.where(opaque, 1.0, rest)
            behind = torch.where(opaque[:, None], 0.0, (tot[:, :3] - f) / rest[:, None])
            clear = torch.where(opaque, tr, (1.0 - tot[:, 3]) / rest)
            ga = g[:, 3] * clear + (g[:, :3] * (tr[:, None] * col[:, :3] - behind)).sum(1)
            gc = torch.cat([g[:, :3] * add[:, None], ga[:, None]], 1) * on[:, None]
            to_table(i, tw, gc)
            scatter(w, idx, (gc * rise).sum(1) * scale * inside)

        _march(flat, dims, tab, rays, "composite", ERT, visit)
    dtf = (moments[0] - moments[1]).T.contiguous()
    dtf[1:] += moments[1].T[:-1]
    return {"image": image, "dtf": dtf, "dvol": dvol.reshape(dims[2], dims[1], dims[0])}


def _exact_pyramid(c, seed):
    img, tile, out = _image(c, seed).double(), c["tile"], []
    while img.shape[0] > 1 or img.shape[1] > 1:
        h, w = img.shape[:2]
        h2, w2 = (h + 1) // 2, (w + 1) // 2
        both = torch.cat([img, torch.ones_like(img[..., :1])], -1)  # the fifth channel counts pixels
        both = torch.nn.functional.pad(both, (0, 0, 0, 2 * w2 - w, 0, 2 * h2 - h))
        both = both.reshape(h2, 2, w2, 2, 5).sum((1, 3))
        img = both[..., :4] / both[..., 4:]
        if not tile:
            out.append(img.reshape(-1))
        else:
            ty, tx = -(-h2 // tile), -(-w2 // tile)
            t = torch.nn.functional.pad(img, (0, 0, 0, tx * tile - w2, 0, ty * tile - h2))
            out.append(t.reshape(ty, tile, tx, tile, 4).transpose(1, 2).reshape(-1))
    return torch.cat(out) if out else torch.zeros(0, dtype=torch.float64, device=DEV)


def exact(case, seed):
    if case["kind"] == "pyramid":
        return _exact_pyramid(case, seed)
    if case["kind"] == "step":
        return _exact_step(case, seed)
    return _exact_frame(case, seed)
