"""Performance cases: the calls a program makes of this renderer, over the range of sizes, data
types and options it takes.

A case is a dict of plain values. Its `kind` says which call it makes:

  frame    Renderer.render of one view of a resident volume (a viewer that turns the camera)
  host     Renderer.render_host_batch: several views read back to pinned host memory
  edit     Renderer.update_tf, then a frame (a viewer whose user edits the palette)
  volume   Renderer.update_volume from a device tensor, build_bricks, a frame (a time series)
  train    DifferentiableRenderer: forward and backward of an L2 loss over some views, and a
           gradient step on the volume and the transfer function
  pieces   Renderer.render_sortlast of a plan of pieces (object-order rendering)
  serve    a burst of requests of mixed image sizes and transfer functions on a PlainServer

The volumes are synthetic CT and phantom data made on the GPU from the seed (the recipes and
value ranges of paper_2005_01442_gb300.synth); transfer functions and cameras come from synth.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2005_01442_gb300 import synth
from paper_2005_01442_gb300.autograd import DifferentiableRenderer
from paper_2005_01442_gb300.renderer import Renderer
from paper_2005_01442_gb300.serve import PlainServer, Request

PHONG = (0.3, 0.7, 0.25, 16.0)  # headlight Blinn-Phong: ambient, diffuse, specular, shininess
SEG_LEN = 64                    # DifferentiableRenderer's default checkpoint interval


def _case(kind, volume, dtype, image, *, name=None, tf="ct", step=0.5, ert=0.999, brick=8,
          variant="cubic", kernel=0, ortho=False, views=1, grid="2,2,2"):
    nx, ny, nz = volume
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "dtype": dtype, "width": image[0],
         "height": image[1], "tf": tf, "step": step, "ert": ert, "brick": brick,
         "variant": variant, "kernel": kernel, "ortho": ortho, "views": views, "grid": grid}
    if name is not None:
        c["name"] = name
    return c


def listed():
    ct = (512, 512, 400)  # the benchmark's CT
    return [
        # a thumbnail: the 64^3 phantom along z at 128^2, no brick table (latency and launches)
        _case("frame", (64, 64, 64), "uint16", (128, 128), name="preview_phantom_128",
              tf="random", ert=1.0, brick=0, ortho=True),
        # the benchmark's frame: a turning camera over a resident CT, bone and vessels visible
        _case("frame", ct, "int16", (1024, 1024), name="frame_ct_1024"),
        # soft tissue semi-transparent: long rays, nearly every sample resampled
        _case("frame", ct, "int16", (1024, 1024), name="frame_dense_1024", tf="dense"),
        # shaded view of a ragged crop in a window of a user's size, coarse bricks
        _case("frame", (253, 187, 250), "int16", (777, 613), name="frame_phong_odd",
              variant="phong", brick=16),
        # a turntable end to end: each frame lands in pinned host memory
        _case("host", ct, "int16", (1024, 1024), name="host_views_1024", views=4),
        # dragging a control point of the palette: every edit redraws the frame
        _case("edit", ct, "int16", (512, 512), name="edit_palette_512"),
        # the next volume of a time series: upload from the device, brick table, first frame
        _case("volume", ct, "int16", (1024, 1024), name="next_volume_1024"),
        # the differentiation workload: 256^3 float32 CT, 512^2 targets
        _case("train", (256, 256, 256), "float32", (512, 512), name="train_256_512", ert=1.0,
              views=2),
        # a small fit on a ragged crop without bricks
        _case("train", (61, 53, 47), "float32", (97, 80), name="train_ragged_small", ert=1.0,
              brick=0),
        # object-order rendering in 2 x 2 x 2 pieces
        _case("pieces", ct, "int16", (1024, 1024), name="pieces_2x2x2_1024"),
        # several clients at once: a burst of small and middling requests on one stream
        _case("serve", (256, 256, 256), "int16", (512, 512), name="serve_burst", views=12),
        # the largest: 512^2 x 2000 at 4096^2, quarter-voxel steps, 16^3 bricks
        _case("frame", (512, 512, 2000), "int16", (4096, 4096), name="large_4096", step=0.25,
              brick=16),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    while True:
        kind = rng.choice(["frame"] * 5 + ["host", "edit", "volume", "train", "pieces", "serve"])
        volume = (spread(40, 512), spread(40, 512), spread(40, 640))
        image = (spread(64, 1600), spread(64, 1600))
        step = rng.choice([0.25, 0.37, 0.5, 0.5, 0.5, 0.75, 1.0])
        ert = rng.choice([0.999, 0.999, 0.99, 1.0])
        brick = rng.choice([8, 8, 16])
        dtype = rng.choice(["int16", "int16", "uint16", "float32"])
        tf, variant, kernel, views, grid = "ct", "cubic", 0, 1, "2,2,2"
        if dtype == "uint16":
            tf = "random"
        elif rng.random() < 0.35:
            tf = "dense"
        if kind == "frame":
            variant = rng.choice(["cubic"] * 4 + ["linear", "phong", "cubic_pre", "linear_pre",
                                                  "preint"])
            if variant == "preint" or rng.random() < 0.1:
                brick = 0
            if variant == "cubic" and tf == "dense" and rng.random() < 0.2:
                kernel = 7  # the staged kernel, for dense transfer functions
        elif kind == "host":
            views = rng.randint(2, 6)
        elif kind == "train":
            dtype, ert = "float32", 1.0
            tf = rng.choice(["ct", "ct", "dense"])
            volume = (spread(32, 256), spread(32, 256), spread(32, 256))
            image = (spread(48, 512), spread(48, 512))
            brick = rng.choice([0, 8, 8, 16])
            views = rng.randint(1, 3)
        elif kind == "pieces":
            grid = rng.choice(["2,2,2", "3,1,2", "1,1,4"])
        elif kind == "serve":
            views = rng.randint(4, 12)
        c = _case(kind, volume, dtype, image, tf=tf, step=step, ert=ert, brick=brick,
                  variant=variant, kernel=kernel, ortho=rng.random() < 0.15, views=views,
                  grid=grid)
        visited = _nominal(c) * (1.0 if brick == 0 or tf != "ct" else 0.05)
        if visited <= 3.0e8:
            return c


# ------------------------------------------------------------------------------ inputs ------
def _window(case):
    return ((synth.PHANTOM_LO, synth.PHANTOM_HI) if case["tf"] == "random"
            else (synth.CT_LO, synth.CT_HI))


def _table(case, seed):
    if case["tf"] == "random":
        return synth.tf_random(seed)
    if case["tf"] == "dense":
        t = synth.tf_ct_dense()
        t[:, 3] *= np.float32(0.8 + 0.4 * np.random.Generator(np.random.PCG64(seed)).random())
        return np.clip(t, 0.0, 1.0)
    return synth.tf_ct(seed)


def _rotation(rng):
    q, r = np.linalg.qr(rng.standard_normal((3, 3)))
    return q * np.sign(np.diag(r))


def _axes(lo, hi, center):
    """Offsets from `center` (x, y, z) of the voxels of a box, broadcast over (z, y, x)."""
    return [torch.arange(lo[k], hi[k], device="cuda", dtype=torch.float32).view(
        [(1, 1, -1), (1, -1, 1), (-1, 1, 1)][k]) - center[k] for k in range(3)]


def _ellipsoid(vol, center, semi, rot, value, add):
    n = vol.shape[::-1]
    ext = float(max(semi)) + 1.0
    lo = [max(0, int(center[k] - ext)) for k in range(3)]
    hi = [min(n[k], int(center[k] + ext) + 2) for k in range(3)]
    if any(h <= l for l, h in zip(lo, hi)):
        return
    x = _axes(lo, hi, center)
    q = sum(((x[0] * rot[0, a] + x[1] * rot[1, a] + x[2] * rot[2, a]) / semi[a]) ** 2
            for a in range(3))
    sub = vol[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]]
    sub.copy_(torch.where(q <= 1.0, sub + value if add else torch.full_like(sub, value), sub))


def _capsule(vol, p0, p1, radius, value):
    n = vol.shape[::-1]
    lo = [max(0, int(min(p0[k], p1[k]) - radius) - 1) for k in range(3)]
    hi = [min(n[k], int(max(p0[k], p1[k]) + radius) + 2) for k in range(3)]
    if any(h <= l for l, h in zip(lo, hi)):
        return
    x = _axes(lo, hi, p0)
    s = [float(p1[k] - p0[k]) for k in range(3)]
    t = ((x[0] * s[0] + x[1] * s[1] + x[2] * s[2]) / max(sum(v * v for v in s), 1e-9)).clamp(0, 1)
    d2 = sum((x[k] - t * s[k]) ** 2 for k in range(3))
    sub = vol[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]]
    sub.masked_fill_(d2 <= radius * radius, value)


def _ct(nx, ny, nz, seed):
    """CT in Hounsfield units as float32 whole numbers: air, an elliptic body of noisy soft
    tissue, bone ellipsoids and contrast-filled vessels (synth.ct_volume's recipe)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 31)))
    cx = (nx - 1) / 2.0 + rng.uniform(-0.02, 0.02) * nx
    cy = (ny - 1) / 2.0 + rng.uniform(-0.02, 0.02) * ny
    ax, ay = 0.42 * nx * rng.uniform(0.95, 1.05), 0.33 * ny * rng.uniform(0.95, 1.05)
    x, y, _ = _axes((0, 0, 0), (nx, ny, 1), (cx, cy, 0.0))
    body = (x / ax) ** 2 + (y / ay) ** 2 <= 1.0
    vol = torch.empty((nz, ny, nx), device="cuda")
    coarse = torch.rand((1, 1, nz // 64 + 2, ny // 64 + 2, nx // 64 + 2), device="cuda",
                        generator=gen) * 80.0
    for z0 in range(0, nz, 128):
        z1 = min(nz, z0 + 128)
        f = torch.linspace(z0 / 64.0, (z1 - 1) / 64.0, z1 - z0, device="cuda")
        i, w = f.long(), (f - f.floor()).view(1, 1, -1, 1, 1)
        planes = coarse[:, :, i] * (1.0 - w) + coarse[:, :, i + 1] * w
        tissue = F.interpolate(planes, size=(z1 - z0, ny, nx), mode="trilinear",
                               align_corners=True)[0, 0]
        noise = torch.randn((z1 - z0, ny, nx), device="cuda", generator=gen) * 10.0
        vol[z0:z1] = torch.where(body, torch.round(tissue + noise),
                                 torch.full_like(noise, -1000.0))

    def point():
        a, r = rng.uniform(0.0, 2.0 * math.pi), math.sqrt(rng.uniform(0.0, 0.8))
        return cx + ax * r * math.cos(a), cy + ay * r * math.sin(a)

    scale = nx / 512.0
    for _ in range(30):
        c = (*point(), rng.uniform(0.05 * nz, 0.95 * nz))
        semi = np.array([rng.uniform(6, 24), rng.uniform(6, 24), rng.uniform(15, 60)]) * scale
        _ellipsoid(vol, c, semi, _rotation(rng), float(rng.integers(700, 1501)), False)
    for _ in range(40):
        p0 = np.array([*point(), rng.uniform(0.0, nz)])
        d = rng.standard_normal(3)
        p1 = p0 + d / np.linalg.norm(d) * rng.uniform(0.2, 0.6) * nz
        _capsule(vol, p0, p1, float(rng.uniform(2.0, 6.0)), 300.0)
    return vol


def _phantom(nx, ny, nz, seed):
    """12-bit phantom: a large ellipsoid and nine smaller ones with additive intensities."""
    rng = np.random.Generator(np.random.PCG64(seed))
    n = np.array([nx, ny, nz], np.float64)
    vol = torch.zeros((nz, ny, nx), device="cuda")
    _ellipsoid(vol, (n - 1) / 2.0, np.array([0.46, 0.40, 0.43]) * n, np.eye(3), 2000.0, True)
    for _ in range(9):
        semi = rng.uniform(0.08, 0.30, 3) * n.min()
        _ellipsoid(vol, rng.uniform(0.25, 0.75, 3) * n, semi, _rotation(rng),
                   float(rng.uniform(-600.0, 1500.0)), True)
    return vol.round_().clamp_(0.0, 4095.0)


def _volume(case, seed):
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    make = _phantom if case["tf"] == "random" else _ct
    if case["dtype"] == "float32":  # the mean of 2 x 2 x 2 voxels of a finer scan
        return F.avg_pool3d(make(2 * nx, 2 * ny, 2 * nz, seed)[None, None], 2)[0, 0].contiguous()
    v = make(nx, ny, nz, seed)
    if case["dtype"] == "int16":
        return v.to(torch.int16)
    return v.to(torch.int32).to(torch.uint16)


def _cameras(case, seed):
    dims = (case["nx"], case["ny"], case["nz"])
    w, h = case["width"], case["height"]
    if case["kind"] == "serve":  # a burst mixes halved, full and doubled images
        sizes = [(max(w // 2, 1), max(h // 2, 1)), (w, h), (2 * w, 2 * h)]
    else:
        sizes = [(w, h)]
    if case["ortho"]:
        return [synth.ortho_z_camera(dims, *sizes[k % len(sizes)]) for k in range(case["views"])]
    rng = np.random.Generator(np.random.PCG64(seed + 7919))
    return [synth.orbit_camera(rng, dims, *sizes[k % len(sizes)]) for k in range(case["views"])]


def _target(case, cam, seed, k):
    """The image a fit aims at: a smooth one, RGBA in [0, 0.6]."""
    gen = torch.Generator(device="cuda").manual_seed(seed * 16 + k)
    low = torch.rand((1, 4, 9, 9), device="cuda", generator=gen) * 0.6
    img = F.interpolate(low, size=(cam.height, cam.width), mode="bilinear", align_corners=True)
    return img[0].permute(1, 2, 0).contiguous()


# ------------------------------------------------------------------------ prepare, run ------
def prepare(case, seed):
    kind, brick = case["kind"], case["brick"]
    lo, hi = _window(case)
    vol = _volume(case, seed)
    cams = _cameras(case, seed)
    table = _table(case, seed + 1)
    R = Renderer(0)
    s = {"case": case, "R": R, "cams": cams, "window": (lo, hi)}
    opts = dict(step=case["step"], ert=case["ert"], brick=brick)
    if kind == "train":
        s["dr"] = DifferentiableRenderer(R, tuple(vol.shape), lo, hi)
        s["volume"] = vol.requires_grad_()
        s["tf"] = torch.from_numpy(table).cuda().requires_grad_()
        s["targets"] = [_target(case, c, seed, k) for k, c in enumerate(cams)]
        s["opts"] = opts
        torch.cuda.synchronize()
        return s
    s["vid"] = R.upload_volume(vol)
    s["tid"] = R.set_tf(table, lo, hi)
    if brick:
        R.build_bricks(s["vid"], brick)
        R.build_occupancy(s["vid"], s["tid"], brick)
    if kind in ("frame", "edit", "volume"):
        opts["kernel"] = case["kernel"]
        opts.update({"linear": {"interp": 1}, "cubic_pre": {"preclass": 1},
                     "linear_pre": {"interp": 1, "preclass": 1}, "phong": {"phong": PHONG},
                     "preint": {"preint": 1}}.get(case["variant"], {}))
    if kind == "host":
        s["out"] = [torch.empty((c.height, c.width, 4), dtype=torch.float32, pin_memory=True)
                    for c in cams]
    elif kind == "edit":
        s["table"] = _table(case, seed + 2)
    elif kind == "volume":
        s["next"] = _volume(case, seed + 3)
    elif kind == "pieces":
        s["plan"] = R.build_pieces(s["vid"], s["tid"], brick,
                                   [int(g) for g in case["grid"].split(",")])
    elif kind == "serve":
        tids = [s["tid"], R.set_tf(_table(case, seed + 2), lo, hi)]
        R.build_occupancy(s["vid"], tids[1], brick)
        s["server"] = PlainServer(R)
        s["requests"] = [Request(0.0, s["vid"], tids[k % 2], c, case["step"], case["ert"], brick)
                         for k, c in enumerate(cams)]
        s["out"] = [torch.empty((c.height, c.width, 4), device="cuda") for c in cams]
    s["opts"] = opts
    torch.cuda.synchronize()
    return s


def run(state):
    kind, R, cams, opts = state["case"]["kind"], state["R"], state["cams"], state["opts"]
    if kind == "frame":
        return R.render(state["vid"], state["tid"], cams[0], **opts)
    if kind == "host":
        return R.render_host_batch(state["vid"], state["tid"], cams, out=state["out"], **opts)
    if kind == "edit":
        R.update_tf(state["tid"], state["table"], *state["window"])
        return R.render(state["vid"], state["tid"], cams[0], **opts)
    if kind == "volume":
        R.update_volume(state["vid"], state["next"])
        R.build_bricks(state["vid"], opts["brick"])
        return R.render(state["vid"], state["tid"], cams[0], **opts)
    if kind == "pieces":
        return R.render_sortlast(state["plan"], cams[0], **opts)
    if kind == "serve":
        done = [state["server"].submit(r, o) for r, o in zip(state["requests"], state["out"])]
        for ev in done:
            torch.cuda.current_stream().wait_event(ev)
        return state["out"]
    vol, tf = state["volume"], state["tf"]
    vol.grad = tf.grad = None
    images = [state["dr"](vol, tf, c, seg_len=SEG_LEN, **opts) for c in cams]
    loss = sum(((im - t) ** 2).sum() for im, t in zip(images, state["targets"]))
    loss.backward()
    with torch.no_grad():  # a small gradient step: the next pass sees new parameters
        vol.sub_(vol.grad, alpha=1e-4)
        tf.sub_(tf.grad, alpha=1e-9).clamp_(0.0, 1.0)
    return {"images": [im.detach() for im in images], "grad_volume": vol.grad, "grad_tf": tf.grad}


# ------------------------------------------------------------------------------- work -------
def _nominal(case):
    """Samples of all rays of all views, skipped or not (about)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    px = sum(c.width * c.height for c in _cameras(case, 0))
    if case["ortho"]:
        return px * nz / case["step"]
    return px * 0.18 * math.sqrt(nx * nx + ny * ny + nz * nz) / case["step"]


def work(case):
    """Each visible voxel read once and each pixel (and gradient) written once; 230 flop per
    sample of non-zero opacity (64 taps, their weights, classification, compositing) and about
    400 more for its gradient. The visible shares are those of the benchmark's CT: 1.1% of the
    samples and 5% of the voxels for bone and vessels, 40% and 60% with soft tissue. Random
    tables are nearly opaque: with termination a ray ends after some 5% of its samples."""
    share, seen = {"ct": (0.011, 0.05), "dense": (0.40, 0.60),
                   "random": (1.0, 1.0) if case["ert"] >= 1.0 else (0.05, 0.10)}[case["tf"]]
    if case["variant"] == "preint" and case["tf"] != "random":
        share, seen = (0.6, 1.0) if case["tf"] == "dense" else (0.9, 1.0)
    voxels = case["nx"] * case["ny"] * case["nz"]
    size = 4 if case["dtype"] == "float32" else 2
    pixels = sum(c.width * c.height for c in _cameras(case, 0))
    samples = _nominal(case) * share
    out = {"bytes": voxels * size * seen + 16.0 * pixels, "flops": 230.0 * samples}
    if case["kind"] == "volume":
        out["bytes"] += voxels * size * (1.0 - seen)
    if case["kind"] == "edit":  # a new palette is held against every brick
        out["bytes"] += 2 * size * voxels / max(case["brick"], 1) ** 3
    if case["kind"] == "train":
        out["bytes"] += 4.0 * voxels + 16.0 * pixels
        out["flops"] += 400.0 * samples
    return out


# ------------------------------------------------------------------------------ exact -------
def _weights(f, derivative=False):
    """Uniform cubic B-spline weights of the four taps at fraction f, or their derivatives."""
    if derivative:
        return [-0.5 * (1 - f) ** 2, 1.5 * f * f - 2 * f, 0.5 + f - 1.5 * f * f, 0.5 * f * f]
    return [(1 - f) ** 3 / 6, (3 * f ** 3 - 6 * f ** 2 + 4) / 6,
            (-3 * f ** 3 + 3 * f ** 2 + 3 * f + 1) / 6, f ** 3 / 6]


class _Exact:
    """The renderer's definition in 64 bits: uniform cubic B-spline (or trilinear) resampling at
    the midpoints of the ray's segments, a 256-entry RGBA table, opacity corrected to the
    segment length, front-to-back compositing, early termination."""

    def __init__(self, case, vol, table):
        self.case = case
        self.n = (case["nx"], case["ny"], case["nz"])
        self.vol = vol.to(torch.float32).reshape(-1)
        self.lo, self.hi = _window(case)
        self.du = 255.0 / (self.hi - self.lo)
        self.tab = torch.from_numpy(table).cuda().double()
        self.slab = self._slabs() if case["variant"] == "preint" else None
        # cells all of whose taps are transparent: their samples have opacity zero
        nz, ny, nx = vol.shape
        p = F.pad(vol.to(torch.float32)[None, None], (2,) * 6, mode="replicate")

        def window(t):
            for k in ((1, 1, 4), (1, 4, 1), (4, 1, 1)):
                t = F.max_pool3d(t, k, 1)
            return t[0, 0]

        u1 = ((window(p) - self.lo) * self.du).clamp_(0, 255).ceil_().to(torch.int16)
        u0 = ((-window(-p) - self.lo) * self.du).clamp_(0, 255).floor_().to(torch.int16)
        pre = F.pad((self.tab[:, 3] > 0).int().cumsum(0), (1, 0)).to(torch.int16)
        self.open = (pre[(u1 + 1).int().clamp_(max=256)] > pre[u0.int()]).reshape(-1)

    def _slabs(self):
        """Slab colour and opacity between table coordinates i (front) and k (back): 32 equal
        sub-steps along the linear ramp."""
        i = torch.arange(256, device="cuda", dtype=torch.float64)
        front, back = i.view(-1, 1), i.view(1, -1)
        c = torch.zeros((256, 256, 3), device="cuda", dtype=torch.float64)
        T = torch.ones((256, 256), device="cuda", dtype=torch.float64)
        for m in range(32):
            rgba = self.lookup((front + (back - front) * (m + 0.5) / 32).reshape(-1))[0]
            rgba = rgba.view(256, 256, 4)
            a = self.opacity(rgba[..., 3], self.case["step"] / 32)
            c += (T * a)[..., None] * rgba[..., :3]
            T = T * (1 - a)
        return torch.cat([c, (1 - T)[..., None]], -1).reshape(-1, 4)

    def lookup(self, u):
        """Table value at coordinate u in [0, 255]; also the entry below and the slope."""
        i = u.floor().clamp_(max=254).long()
        d = self.tab[i + 1] - self.tab[i]
        return self.tab[i] + (u - i)[:, None] * d, i, d

    @staticmethod
    def opacity(a, delta):
        return -torch.expm1(delta * torch.log1p(-a.clamp(0, 1 - 2.0 ** -24)))

    def rays(self, cam):
        """Origins, unit directions, entry and exit parameters of all pixels, row by row."""
        f64 = dict(device="cuda", dtype=torch.float64)
        eye, center, up = (np.array(v, np.float64) for v in (cam.eye, cam.center, cam.up))
        f = (center - eye) / np.linalg.norm(center - eye)
        r = np.cross(f, up)
        r /= np.linalg.norm(r)
        u = np.cross(r, f)
        X = (2 * torch.arange(cam.width, **f64) + 1) / cam.width - 1
        Y = 1 - (2 * torch.arange(cam.height, **f64) + 1) / cam.height
        X, Y = X.view(1, -1, 1), Y.view(-1, 1, 1)
        f, r, u, eye = (torch.tensor(v, **f64) for v in (f, r, u, eye))
        if cam.ortho:
            hx, hy = (0.5 * e for e in cam.ortho_extent)
            o = (eye + X * hx * r + Y * hy * u).reshape(-1, 3)
            d = f.expand_as(o)
        else:
            th = math.tan(0.5 * math.radians(cam.fovy_deg))
            d = (f + X * th * cam.width / cam.height * r + Y * th * u).reshape(-1, 3)
            d = d / d.norm(dim=1, keepdim=True)
            o = eye.expand_as(d)
        size = torch.tensor(self.n, **f64)
        t0, t1 = (-0.5 - o) / d, (size - 0.5 - o) / d
        flat = d == 0
        inside = (o >= -0.5) & (o <= size - 0.5)
        near = torch.where(flat, -math.inf, torch.minimum(t0, t1)).amax(1).clamp_(min=0)
        far = torch.where(flat, math.inf, torch.maximum(t0, t1)).amin(1)
        hit = (far > near) & (inside | ~flat).all(1)
        return o, d, near, torch.where(hit, far, near)

    def taps(self, base, first, count):
        """Clamped tap indices of each axis: first .. first + count - 1 from the cell."""
        return [[(base[k] + first + m).clamp_(0, self.n[k] - 1) for m in range(count)]
                for k in range(3)]

    def sample(self, base, frac, dirs):
        """(rgba, table coordinate before clamping) of samples at cell `base`."""
        v = self.case["variant"]
        if v in ("linear", "linear_pre"):
            w, idx = [[1 - f, f] for f in frac], self.taps(base, 0, 2)
        else:
            w, idx = [_weights(f) for f in frac], self.taps(base, -1, 4)
        dw = [_weights(f, True) for f in frac] if v == "phong" else None
        nx, ny, _ = self.n
        acc = grad = 0
        for c, z in enumerate(idx[2]):
            for b, y in enumerate(idx[1]):
                row = (z * ny + y) * nx
                s = ds = 0
                for a, x in enumerate(idx[0]):
                    value = self.vol[row + x].double()
                    if v.endswith("_pre"):
                        u = ((value - self.lo) * self.du).clamp_(0, 255)
                        value, = self.lookup(u)[:1]
                        s = s + w[0][a][:, None] * value
                    else:
                        s = s + w[0][a] * value
                        if dw:
                            ds = ds + dw[0][a] * value
                wyz = w[1][b] * w[2][c]
                if v.endswith("_pre"):
                    acc = acc + wyz[:, None] * s
                    continue
                acc = acc + wyz * s
                if dw:
                    grad = grad + torch.stack([wyz * ds, dw[1][b] * w[2][c] * s,
                                               w[1][b] * dw[2][c] * s], 1)
        if v.endswith("_pre"):
            return acc, None
        u = (acc - self.lo) * self.du
        if v == "preint":
            return None, u
        rgba = self.lookup(u.clamp(0, 255))[0]
        if dw:
            ka, kd, ks, shine = PHONG
            eps = 0.01 * (self.hi - self.lo)
            nl = (grad * dirs).sum(1).abs() / ((grad ** 2).sum(1) + eps * eps).sqrt()
            rgba = torch.cat([rgba[:, :3] * (ka + kd * nl)[:, None]
                              + (ks * nl ** shine)[:, None], rgba[:, 3:]], 1)
        return rgba, u

    def chunks(self, cam, piece=1 << 22, most=1 << 25):
        """Runs of rays: (pixels, lengths, opacity and colour per sample, and the samples that
        were resampled as (ray, index, cell, fraction, u))."""
        step = self.case["step"]
        o, d, near, far = self.rays(cam)
        length = far - near
        nseg = (length / step).ceil().clamp_(min=1).long() * (length > 0)
        per = max(1, most // max(1, int(nseg.max())))
        for r0 in range(0, nseg.numel(), per):
            pix = torch.arange(r0, min(nseg.numel(), r0 + per), device="cuda")
            pix = pix[nseg[pix] > 0]
            if not pix.numel():
                continue
            S = int(nseg[pix].max())
            j = torch.arange(S, device="cuda")
            last = j[None] == nseg[pix, None] - 1
            start = j[None] * step
            delta = torch.where(last, length[pix, None] - start, torch.full_like(start, step))
            live = j[None] < nseg[pix, None]
            t = near[pix, None] + start + 0.5 * delta
            pos = [o[pix, k, None] + t * d[pix, k, None] for k in range(3)]
            cell = [torch.minimum(p.floor().long().clamp_(min=-1),
                                  torch.tensor(n - 1, device="cuda"))
                    for p, n in zip(pos, self.n)]
            if self.slab is None:
                nx, ny, _ = self.n
                live &= self.open[((cell[2] + 1) * (ny + 1) + cell[1] + 1) * (nx + 1)
                                  + cell[0] + 1]
            ray, idx = live.nonzero(as_tuple=True)
            base = [c[ray, idx] for c in cell]
            frac = [p[ray, idx] - b for p, b in zip(pos, base)]
            del pos, cell, t, live
            rgba, u = [], []
            for q in range(0, ray.numel(), piece):
                cut = slice(q, q + piece)
                a, b = self.sample([v[cut] for v in base], [v[cut] for v in frac],
                                   d[pix[ray[cut]]])
                rgba.append(a)
                u.append(b)
            yield pix, S, delta, (ray, idx, base, frac), rgba, u

    def image(self, cam, grad_of=None):
        """The image, and with grad_of(image) = dL/dimage the gradients of volume and table."""
        thr = self.case["ert"]
        out = torch.zeros((cam.height * cam.width, 4), device="cuda", dtype=torch.float64)
        kept = []
        for pix, S, delta, where, rgba, u in self.chunks(cam):
            ray, idx = where[:2]
            alpha = torch.zeros((pix.numel(), S), device="cuda", dtype=torch.float64)
            color = torch.zeros((pix.numel(), S, 3), device="cuda", dtype=torch.float64)
            if not ray.numel():
                continue
            u = torch.cat(u) if u[0] is not None else None
            if self.slab is not None:
                grid = torch.zeros_like(alpha)
                grid[ray, idx] = u.clamp(0, 255)
                valid = torch.zeros_like(alpha, dtype=torch.bool)
                valid[ray, idx] = True
                f0, f1 = grid[:, :-1], grid[:, 1:]
                i0, k0 = (g.floor().clamp_(max=254).long() for g in (f0, f1))
                fi, fk = (f0 - i0)[..., None], (f1 - k0)[..., None]
                at = i0 * 256 + k0
                e = ((1 - fi) * ((1 - fk) * self.slab[at] + fk * self.slab[at + 1])
                     + fi * ((1 - fk) * self.slab[at + 256] + fk * self.slab[at + 257]))
                span = 0.5 * (delta[:, :-1] + delta[:, 1:]) / self.case["step"]
                a2 = self.opacity(e[..., 3], span)
                ok = valid[:, 1:] & (e[..., 3] > 0)
                color[:, 1:] = torch.where(ok[..., None], e[..., :3] / e[..., 3:].clamp(min=1e-300),
                                           torch.zeros_like(e[..., :3]))
                alpha[:, 1:] = torch.where(ok, a2, torch.zeros_like(a2))
            else:
                rgba = torch.cat(rgba)
                alpha[ray, idx] = self.opacity(rgba[:, 3], delta[ray, idx])
                color[ray, idx] = rgba[:, :3]
            after = torch.cumprod(1 - alpha, 1)
            stop = (1 - after > thr) & (alpha > 0)
            alpha = torch.where(stop.cumsum(1) - stop.long() == 0, alpha, torch.zeros_like(alpha))
            after = torch.cumprod(1 - alpha, 1)
            before = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
            weight = before * alpha
            out[pix, :3] = (weight[..., None] * color).sum(1)
            out[pix, 3] = 1 - after[:, -1]
            if grad_of is not None:
                kept.append((pix, delta, where, u, alpha, color, before, weight, after[:, -1]))
        image = out.view(cam.height, cam.width, 4)
        if grad_of is None:
            return image
        g_all = grad_of(image).view(-1, 4)
        gtab = torch.zeros_like(self.tab)
        gvol = torch.zeros(self.vol.numel(), device="cuda", dtype=torch.float64)
        for pix, delta, (ray, idx, base, frac), u, alpha, color, before, weight, final in kept:
            g = g_all[pix]
            gc = (color * g[:, None, :3]).sum(-1)
            behind = (weight * gc).flip(1).cumsum(1).flip(1) - weight * gc
            dalpha = before * gc + (g[:, 3, None] * final[:, None] - behind) / (1 - alpha)
            rgba, i, slope = self.lookup(u.clamp(0, 255))
            a, dl = rgba[:, 3], delta[ray, idx]
            da = torch.where((a > 0) & (a <= 1 - 2.0 ** -24), dl * (1 - a).clamp(min=2.0 ** -24)
                             ** (dl - 1), torch.zeros_like(a))
            d = torch.cat([weight[ray, idx, None] * g[ray, :3],
                           (dalpha[ray, idx] * da)[:, None]], 1)
            f = (u.clamp(0, 255) - i)[:, None]
            gtab.index_add_(0, i, (1 - f) * d)
            gtab.index_add_(0, i + 1, f * d)
            ds = (d * slope).sum(1) * self.du * ((u > 0) & (u < 255))
            w = [_weights(x) for x in frac]
            tap = self.taps(base, -1, 4)
            for c in range(4):
                for b in range(4):
                    row = (tap[2][c] * self.n[1] + tap[1][b]) * self.n[0]
                    for k in range(4):
                        gvol.index_add_(0, row + tap[0][k], ds * w[0][k] * w[1][b] * w[2][c])
        return image, gvol.view(self.n[2], self.n[1], self.n[0]), gtab


def exact(case, seed):
    # sort-last pieces stop on their own opacity, and the largest images would take too long
    if _nominal(case) > 1.5e9 or (case["kind"] == "pieces" and case["ert"] < 1.0):
        return None
    if case["tf"] == "random" and case["brick"] == 0 and _nominal(case) > 4e8:
        return None
    cams, table = _cameras(case, seed), _table(case, seed + 1)
    if case["kind"] == "edit":
        table = _table(case, seed + 2)
    vol = _volume(case, seed + 3 if case["kind"] == "volume" else seed)
    x = _Exact(case, vol, table)
    if case["kind"] == "train":
        images, gvol, gtab = [], 0, 0
        for k, c in enumerate(cams):
            target = _target(case, c, seed, k).double()
            im, gv, gt = x.image(c, lambda image: 2 * (image - target))
            images.append(im)
            gvol, gtab = gvol + gv, gtab + gt
        return {"images": images, "grad_volume": gvol, "grad_tf": gtab}
    if case["kind"] == "serve":
        y = _Exact(case, vol, _table(case, seed + 2))
        return [(y if k % 2 else x).image(c) for k, c in enumerate(cams)]
    images = [x.image(c) for c in cams]
    return images if case["kind"] == "host" else images[0]
