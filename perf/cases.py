"""The work this renderer is used for, as measurable cases.

A case is one call (or the short call sequence a program makes for one frame or
one VDI) through the Python binding of the C ABI.  Four kinds:

* ``render``   one new view of a resident VDI (``vdi_render``): the exact frame,
  the original view and the subsampled previews, at the three workload sizes
  (128 x 128, 720p, 1080p).
* ``batch``    a server's launch: several views of several resident VDIs in one
  ``vdi_render_batch`` with the cached graph.
* ``generate`` a VDI built from a volume (``vdi_generate``, fixed or ray-adaptive
  sensitivity) and then shown (the original view and a turned one) or
  downloaded to the host, as a program that streams VDIs to a client does.
* ``create``   a client's side: a VDI built from received supersegment buffers
  (``vdi_create``) and shown.
* ``quality``  the evaluation: direct volume rendering of a view, the VDI's
  render of the same view, and SSIM / PSNR between them.

``exact`` restates generation, rendering, previews and the quality measures in
plain torch (FP64; generation's integer decisions in IEEE FP32, the precision
they are defined in).
"""
import math

import numpy as np
import torch

import paper_2206_08660_gb300 as V

DEV = "cuda" if torch.cuda.is_available() else "cpu"
ERT = 1.0 / 4096.0  # compositing stops at this transmittance


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------


def listed():
    return [
        # the smallest frame: latency of one call (host constants, one launch)
        dict(name="tiny_render", kind="render", vol="blobs", n=64, w=128, h=128, ns=8, fmt="fp32", W=128, H=128,
             angle=10.0, zoom=1.0, d_i=1, d_r=1, out="fp32"),
        # an ordinary exact frame with FP32 colour, zoomed in on a sparse volume
        dict(name="plain_720p", kind="render", vol="noise", n=256, w=1280, h=720, ns=20, fmt="fp32", W=1280, H=720,
             angle=15.0, zoom=1.2, d_i=1, d_r=1, out="fp32"),
        # the original view: what a client shows until the user moves
        dict(name="original_1080p", kind="render", vol="mixing", n=1024, w=1920, h=1080, ns=20, fmt="fp16", W=1920,
             H=1080, angle=0.0, zoom=1.0, d_i=1, d_r=1, out="fp32"),
        # the exact frame of the large workload at a middle deviation
        dict(name="large_1080p", kind="render", vol="mixing", n=1024, w=1920, h=1080, ns=20, fmt="fp16", W=1920,
             H=1080, angle=20.0, zoom=1.0, d_i=1, d_r=1, out="fp32"),
        # the previews shown while the view moves
        dict(name="preview_2_2", kind="render", vol="mixing", n=1024, w=1920, h=1080, ns=20, fmt="fp16", W=1920,
             H=1080, angle=30.0, zoom=1.0, d_i=2, d_r=2, out="fp32"),
        dict(name="preview_4_4", kind="render", vol="mixing", n=1024, w=1920, h=1080, ns=20, fmt="fp16", W=1920,
             H=1080, angle=30.0, zoom=1.0, d_i=4, d_r=4, out="fp32"),
        # a server's launch: sixteen views of four VDIs, exact and preview mixed, FP16 images
        dict(name="batch_16", kind="batch", n=256, requests=16, scale=1.0, max_angle=45.0, previews=True),
        # a fresh VDI of the large volume, then its first two frames
        dict(name="generate_1080p", kind="generate", vol="mixing", n=1024, w=1920, h=1080, ns=20, fmt="fp16",
             adaptive=False, angle=10.0, download=False),
        # the ray-adaptive sensitivity on an ordinary volume
        dict(name="generate_adaptive", kind="generate", vol="noise", n=256, w=1280, h=720, ns=20, fmt="fp32",
             adaptive=True, angle=10.0, download=False),
        # the smallest generation, copied to the host for streaming
        dict(name="generate_tiny", kind="generate", vol="blobs", n=64, w=128, h=128, ns=8, fmt="fp32",
             adaptive=False, angle=0.0, download=True),
        # a client that receives a VDI of ragged size with an odd slot count
        dict(name="create_1366", kind="create", w=1366, h=767, ns=15, fmt="fp16", angle=20.0, mem="device"),
        # one point of the quality evaluation
        dict(name="quality_720p", kind="quality", vol="noise", n=256, w=1280, h=720, ns=20, fmt="fp32", angle=10.0,
             step=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["render", "preview", "batch", "generate", "create", "quality"], [4, 3, 1, 3, 2, 1])[0]
    aspect = rng.choice([16 / 9, 16 / 9, 4 / 3, 1.0])
    h = _log_int(rng, 96, 1080)
    w = max(16, int(round(h * aspect)) + rng.choice([0, 0, -1, 1]))
    fmt = rng.choice(["fp16", "fp32"])
    vol = rng.choice(["mixing", "noise", "blobs"])
    n = _log_int(rng, 48, {"mixing": 1024, "noise": 384, "blobs": 128}[vol])
    ns = rng.randint(4, 24)
    if kind in ("render", "preview"):
        H = max(48, min(1080, int(h * rng.uniform(0.6, 1.2))))
        W = max(64, min(1920, int(round(H * aspect))))
        angle = round(rng.uniform(1.0, 60.0), 2) * rng.choice([1, 1, -1])
        zoom = rng.choice([1.0, 1.0, 1.2, 1.5])
        if kind == "render" and rng.random() < 0.25:  # the original view at the VDI's own resolution
            W, H, angle, zoom = w, h, 0.0, 1.0
        d_i, d_r = (1, 1) if kind == "render" else rng.choice([(2, 2), (4, 4), (1, 2), (2, 1), (2, 4), (1, 4)])
        return dict(kind="render", vol=vol, n=n, w=w, h=h, ns=ns, fmt=fmt, W=W, H=H, angle=angle,
                    zoom=zoom, d_i=d_i, d_r=d_r, out=rng.choice(["fp32", "fp16"]))
    if kind == "batch":
        return dict(kind="batch", n=_log_int(rng, 96, 256), requests=rng.randint(2, 16),
                    scale=round(rng.uniform(0.3, 1.0), 3), max_angle=round(rng.uniform(10.0, 45.0), 2),
                    previews=rng.random() < 0.5)
    if kind == "generate":
        adaptive = rng.random() < 0.4
        if adaptive:
            n, h = min(n, 256), min(h, 720)
            w = int(round(h * aspect))
        small = w * h * ns < 1_000_000
        return dict(kind="generate", vol=vol, n=n, w=w, h=h, ns=ns, fmt=fmt, adaptive=adaptive,
                    angle=round(rng.uniform(0.0, 40.0), 2), download=small and rng.random() < 0.5)
    if kind == "create":
        h = min(h, 767)
        w = max(16, int(round(h * aspect)) + rng.choice([0, 1]))
        mem = "host" if w * h < 200_000 and rng.random() < 0.5 else "device"
        return dict(kind="create", w=w, h=h, ns=min(ns, 15), fmt=fmt, angle=round(rng.uniform(1.0, 45.0), 2), mem=mem)
    h = min(h, 720)
    return dict(kind="quality", vol=vol, n=min(n, 256), w=int(round(h * aspect)), h=h, ns=ns, fmt=fmt,
                angle=round(rng.uniform(0.0, 40.0), 2), step=rng.choice([1.0, 0.5]))


# ---------------------------------------------------------------------------
# inputs: cameras, volumes, transfer functions, supersegment buffers
# ---------------------------------------------------------------------------

BMIN, BMAX = np.zeros(3), np.ones(3)
ELEVATION = {"blobs": 15.0, "noise": 20.0, "mixing": 25.0, "layers": 20.0}
TAU = {"blobs": 0.02, "noise": 0.01, "mixing": 0.01}

# four-knot transfer functions (value, r, g, b, alpha per voxel length): dense for
# the blobs, sparse for the noise, an interface sheet over a haze for the mixing layer
KNOTS = {
    "blobs": [[0.00, 0.10, 0.20, 0.80, 0.00], [0.30, 0.20, 0.60, 0.90, 0.05],
              [0.60, 0.95, 0.60, 0.20, 0.35], [1.00, 0.90, 0.20, 0.10, 0.50]],
    "noise": [[0.00, 0.00, 0.00, 0.00, 0.00], [0.45, 0.30, 0.50, 0.90, 0.00],
              [0.60, 0.95, 0.70, 0.30, 0.25], [1.00, 1.00, 0.30, 0.20, 0.50]],
    "mixing": [[0.00, 0.20, 0.40, 0.90, 0.00], [0.30, 0.30, 0.70, 0.90, 0.20],
               [0.60, 1.00, 0.55, 0.15, 0.45], [1.00, 0.25, 0.35, 0.80, 0.03]],
}


def orbit(aspect, az_deg, el_deg, zoom=1.0):
    """(view, proj) of a camera facing the box centre from three bounding-sphere radii."""
    c, r = 0.5 * (BMIN + BMAX), 0.5 * np.linalg.norm(BMAX - BMIN)
    d, az, el = 3.0 * r, math.radians(az_deg), math.radians(el_deg)
    eye = c + d * np.array([math.cos(el) * math.sin(az), math.sin(el), math.cos(el) * math.cos(az)])
    f = (c - eye) / np.linalg.norm(c - eye)
    s = np.cross(f, [0.0, 1.0, 0.0])
    s /= np.linalg.norm(s)
    u = np.cross(s, f)
    view = np.eye(4)
    view[0, :3], view[1, :3], view[2, :3] = s, u, -f
    view[0, 3], view[1, 3], view[2, 3] = -s @ eye, -u @ eye, f @ eye
    near, far = d - r, d + r
    q = zoom / math.tan(math.asin(r / d))
    proj = np.zeros((4, 4))
    proj[0, 0], proj[1, 1] = q / aspect, q
    proj[2, 2], proj[2, 3] = (far + near) / (near - far), 2.0 * far * near / (near - far)
    proj[3, 2] = -1.0
    return view, proj


def _uniform(seed, *shape):
    """Seeded U[0, 1) values, the same on every machine (drawn on the CPU)."""
    g = torch.Generator().manual_seed(seed)
    return torch.rand(*shape, generator=g).to(DEV)


def blobs_volume(n, seed):
    """Sum of six Gaussian blobs, f32."""
    p = _uniform(seed, 6, 4).double()
    g = (torch.arange(n, device=DEV, dtype=torch.float64) + 0.5) / n
    v = torch.zeros(n, n, n, device=DEV, dtype=torch.float64)
    for q in p.cpu().tolist():
        c, s = [0.2 + 0.6 * t for t in q[:3]], 0.05 + 0.1 * q[3]
        e = [torch.exp(-((g - t) ** 2) / (2 * s * s)) for t in c]
        v += e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :]
    return v.clamp(0.0, 1.0).float().contiguous()


def noise_volume(n, seed, u8=False):
    """Five octaves of value noise with smoothstep interpolation, u16 (or u8)."""
    acc = torch.zeros(n, n, n, device=DEV)
    for k in range(5):
        f = 4 << k
        a = _uniform(seed + k, f + 1, f + 1, f + 1)
        pos = (torch.arange(n, device=DEV, dtype=torch.float64) + 0.5) / n * f
        i0 = pos.floor().long().clamp(max=f - 1)
        t = (pos - i0).float()
        t = t * t * (3.0 - 2.0 * t)
        for axis in (2, 1, 0):
            shape = [1, 1, 1]
            shape[axis] = n
            lo, hi = a.index_select(axis, i0), a.index_select(axis, i0 + 1)
            a = lo + (hi - lo) * t.view(shape)
        acc += 0.5 ** k * a
    acc = (acc - acc.min()) / (acc.max() - acc.min())
    if u8:
        return (acc * 255.0).round().to(torch.uint8)
    return (acc * 65535.0).round().to(torch.int32).to(torch.int16).view(torch.uint16)


def mixing_volume(n, seed):
    """A tanh interface at mid height, perturbed by 64 Fourier modes, u8."""
    p = _uniform(seed, 64, 4).double().cpu().tolist()
    g = (torch.arange(n, device=DEV, dtype=torch.float64) + 0.5) / n
    height = torch.full((n, n), 0.5, device=DEV, dtype=torch.float64)  # [z, x]
    for a, kx, kz, ph in p:
        height += 0.05 * a * torch.sin(2 * math.pi * (int(1 + 8 * kx) * g[None, :] + int(1 + 8 * kz) * g[:, None] + ph))
    out = torch.empty(n, n, n, device=DEV, dtype=torch.uint8)
    y, height = g.float(), height.float()
    for z in range(0, n, 32):
        rho = torch.tanh((y[None, :, None] - height[z:z + 32, None, :]) * 100.0)
        out[z:z + 32] = (rho.mul_(0.5).add_(0.5).mul_(255.0).round_()).to(torch.uint8)
    return out


def volume(kind, n, seed):
    return {"blobs": blobs_volume, "noise": noise_volume, "mixing": mixing_volume}[kind](n, seed)


def layers(w, h, ns, seed):
    """Supersegment buffers as a client receives them: per list a smooth stack of
    layers with gaps and touching neighbours, a quarter of the lists empty."""
    p = _uniform(seed, ns + 2, 6).cpu().tolist()
    y, x = torch.meshgrid((torch.arange(h, device=DEV) + 0.5) / h, (torch.arange(w, device=DEV) + 0.5) / w, indexing="ij")

    def wave(q):
        return 0.5 + 0.25 * (torch.sin(2 * math.pi * ((1 + 3 * q[0]) * x + q[1] + 2 * q[2] * y))
                             + torch.sin(2 * math.pi * ((1 + 5 * q[3]) * y + q[4] + 2 * q[5] * x)))

    cut = torch.stack([0.1 + 0.9 * wave(p[k]) for k in range(ns)], -1)  # thickness of each layer's cell
    edge = torch.cumsum(cut, -1) / (1.05 * ns)
    z1 = -0.7 + 1.4 * edge + 0.1 * (wave(p[ns]) - 0.5)[..., None]
    z0 = torch.cat([(-0.7 + 0.1 * (wave(p[ns]) - 0.5))[..., None], z1[..., :-1]], -1)
    solid = 0.4 + 0.6 * torch.stack([wave(p[(k + 1) % ns]) for k in range(ns)], -1)
    solid = torch.where(solid > 0.85, torch.ones_like(solid), solid)  # those touch the next layer
    depth = torch.stack([z0, torch.minimum(z0 + solid * (z1 - z0), z1)], -1).float()
    r2 = (x - 0.5) ** 2 + (y - 0.5) ** 2
    counts = (ns * (0.3 + wave(p[ns + 1]))).int().clamp(1, ns) * (r2 < 0.24).int()
    alpha = 0.02 + 0.3 * cut * (1 - 0.5 * solid)
    rgba = torch.stack([alpha * wave(p[k % ns])[..., None] for k in range(3)] + [alpha], -1).float()
    rgba[..., :3] = torch.minimum(rgba[..., :3], rgba[..., 3:])
    dead = torch.arange(ns, device=DEV)[None, None, :] >= counts[..., None]
    depth[dead] = math.inf
    rgba[dead] = 0.0
    return rgba.contiguous(), depth.contiguous(), counts.contiguous()


# ---------------------------------------------------------------------------
# prepare / run
# ---------------------------------------------------------------------------

FMT = {"fp32": V.VDI_F32, "fp16": V.VDI_F16}
DTYPE = {"fp32": torch.float32, "fp16": torch.float16}
_ctx = None


def ctx():
    """The program's one context."""
    global _ctx
    if _ctx is None:
        _ctx = V.vdi_ctx_create(0)
    return _ctx


class Vdi:
    """A resident VDI that is freed with its owner."""

    def __init__(self, handle):
        self.handle = handle

    def __del__(self):
        if self.handle is not None:
            V.vdi_destroy(self.handle)
            self.handle = None


def cam(view, proj):
    return V.camera(view, proj)


def generated(vol, kind, n, w, h, ns, fmt, view, proj, adaptive=False, tau_out=None):
    u = 1.0 / n
    return Vdi(V.vdi_generate(ctx(), vol, BMIN, BMAX, np.asarray(KNOTS[kind], np.float32), cam(view, proj), w, h, ns,
                              TAU[kind], u, u, FMT[fmt], adaptive=adaptive, tau_out=tau_out))


def image(W, H, out):
    return torch.empty(H, W, 4, dtype=DTYPE[out], device=DEV)


# the server's four resident VDIs and its image sizes
BATCH_VDIS = [(640, 360, 8), (1280, 720, 16), (1920, 1080, 20), (1920, 1080, 24)]
BATCH_SIZES = [(640, 360), (1280, 720), (1280, 720), (1920, 1080)]


def batch_plan(case, seed):
    """(VDI sizes, [(vdi, W, H, angle, d_i, d_r)]): the resolutions and previews belong to the case, the angles to the seed."""
    s = case["scale"]
    vdis = [(max(16, int(w * s)), max(16, int(h * s)), ns) for w, h, ns in BATCH_VDIS]
    shape, turn = np.random.RandomState(case["requests"]), np.random.RandomState(seed % (1 << 31))
    reqs = []
    for _ in range(case["requests"]):
        W, H = BATCH_SIZES[shape.randint(4)]
        k = shape.randint(4)
        d_i, d_r = (shape.randint(1, 3), shape.randint(1, 3)) if case["previews"] else (1, 1)
        reqs.append((int(k), max(16, int(W * s)), max(16, int(H * s)), float(turn.uniform(-1, 1)) * case["max_angle"],
                     int(d_i), int(d_r)))
    return vdis, reqs


def prepare(case, seed):
    c, s = case, {"case": case}
    kind = c["kind"]
    if kind in ("render", "quality", "generate"):
        vol = volume(c["vol"], c["n"], seed)
        el = ELEVATION[c["vol"]]
        vo = orbit(c["w"] / c["h"], 0.0, el)
    if kind == "render":
        s["vdi"] = generated(vol, c["vol"], c["n"], c["w"], c["h"], c["ns"], c["fmt"], *vo)
        s["view"] = cam(*orbit(c["W"] / c["H"], c["angle"], el, c["zoom"]))
        s["out"] = image(c["W"], c["H"], c["out"])
    elif kind == "batch":
        vdis, reqs = batch_plan(c, seed)
        s["vdis"] = []
        for k, (w, h, ns) in enumerate(vdis):
            vol = noise_volume(c["n"], seed + 10 * k, u8=True)
            s["vdis"].append(generated(vol, "noise", c["n"], w, h, ns, "fp16", *orbit(w / h, 90.0 * k, 20.0)))
        s["out"] = [image(W, H, "fp16") for _, W, H, _, _, _ in reqs]
        s["requests"] = [V.request(s["vdis"][k].handle, cam(*orbit(W / H, 90.0 * k + a, 20.0)), W, H, d_i, d_r, o, V.VDI_F16)
                         for (k, W, H, a, d_i, d_r), o in zip(reqs, s["out"])]
    elif kind == "generate":
        s["vol"], s["orig"] = vol, vo
        s["tau"] = torch.empty(c["h"], c["w"], device=DEV) if c["adaptive"] else None
        s["views"] = [cam(*vo), cam(*orbit(c["w"] / c["h"], c["angle"], el))]
        s["out"] = [image(c["w"], c["h"], "fp32") for _ in s["views"]]
        s["vdi"] = None
    elif kind == "create":
        bufs = layers(c["w"], c["h"], c["ns"], seed)
        s["bufs"] = [b.cpu().numpy() for b in bufs] if c["mem"] == "host" else bufs
        vo = orbit(c["w"] / c["h"], 0.0, ELEVATION["layers"])
        s["desc"] = V.desc(c["w"], c["h"], c["ns"], *vo, BMIN, BMAX, 1.0 / 64, FMT[c["fmt"]])
        s["view"] = cam(*orbit(c["w"] / c["h"], c["angle"], ELEVATION["layers"]))
        s["out"] = image(c["w"], c["h"], "fp32")
        s["vdi"] = None
    else:
        s["vol"] = vol
        s["vdi"] = generated(vol, c["vol"], c["n"], c["w"], c["h"], c["ns"], c["fmt"], *vo)
        s["view"] = cam(*orbit(c["w"] / c["h"], c["angle"], el))
        s["out"] = [image(c["w"], c["h"], "fp32") for _ in range(2)]
    return s


def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "render":
        V.vdi_render(s["vdi"].handle, s["view"], c["W"], c["H"], c["d_i"], c["d_r"], s["out"], FMT[c["out"]])
        return s["out"]
    if kind == "batch":
        V.vdi_render_batch(ctx(), s["requests"])
        return s["out"]
    if kind == "generate":
        s["vdi"] = None  # the program's previous VDI makes room for the new one
        s["vdi"] = generated(s["vol"], c["vol"], c["n"], c["w"], c["h"], c["ns"], c["fmt"], *s["orig"], c["adaptive"], s["tau"])
        if c["download"]:
            rgba, depth, counts, grid = V.vdi_download(s["vdi"].handle, c["w"], c["h"], c["ns"])
            r = {"rgba": rgba, "depth": depth, "counts": counts, "grid": grid.view(np.int32)}
        else:
            for view, out in zip(s["views"], s["out"]):
                V.vdi_render(s["vdi"].handle, view, c["w"], c["h"], 1, 1, out)
            r = {"images": s["out"]}
        if c["adaptive"]:
            r["tau"] = s["tau"]
        return r
    if kind == "create":
        s["vdi"] = None
        s["vdi"] = Vdi(V.vdi_create(ctx(), s["desc"], *s["bufs"]))
        V.vdi_render(s["vdi"].handle, s["view"], c["w"], c["h"], 1, 1, s["out"])
        return s["out"]
    u = 1.0 / c["n"]
    V.vdi_dvr(ctx(), s["vol"], BMIN, BMAX, np.asarray(KNOTS[c["vol"]], np.float32), s["view"], c["w"], c["h"],
              c["step"] * u, u, s["out"][0])
    V.vdi_render(s["vdi"].handle, s["view"], c["w"], c["h"], 1, 1, s["out"][1])
    ssim, psnr = V.vdi_image_quality(s["out"][1], s["out"][0])
    return {"dvr": s["out"][0], "render": s["out"][1], "ssim": ssim, "psnr": psnr}


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------


def _view_work(w, h, ns, fmt, W, H, angle, zoom, d_i, d_r, bpp):
    """One frame: the records a frame needs (the lists the box covers, about 128
    bytes each), the image, and per ray the lists crossed and pieces composited
    (per preview sample the map into the list grid and one piece)."""
    hit = min(1.0, 0.46 * h / w) * w * h
    rays = min(1.0, 0.46 * zoom * zoom * H / W) * (-(-W // d_i)) * (-(-H // d_i))
    lists = 1.0 + 0.15 * w * abs(math.sin(math.radians(angle)))
    rec = hit * min(8 + ns * (24 if fmt == "fp32" else 16), 128) / (d_i * d_i if d_r > 1 else 1)
    pieces = (0.6 * lists + 2.0) / d_r
    return rec + W * H * bpp, rays * ((12 * lists if d_r == 1 else 0) + 30 * pieces)


def work(case):
    c = case
    kind = c["kind"]
    vox = {"blobs": 4, "noise": 2, "mixing": 1}.get(c.get("vol"), 1)
    slot = 24 if c.get("fmt") == "fp32" else 16
    if kind == "render":
        b, f = _view_work(c["w"], c["h"], c["ns"], c["fmt"], c["W"], c["H"], c["angle"], c["zoom"], c["d_i"], c["d_r"],
                          16 if c["out"] == "fp32" else 8)
        return {"bytes": b, "flops": f}
    if kind == "batch":
        vdis, reqs = batch_plan(c, 0)
        parts = [_view_work(*vdis[k], "fp16", W, H, 0.5 * c["max_angle"], 1.0, d_i, d_r, 8) for k, W, H, _, d_i, d_r in reqs]
        return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}
    if kind == "create":
        b, f = _view_work(c["w"], c["h"], c["ns"], c["fmt"], c["w"], c["h"], c["angle"], 1.0, 1, 1, 16)
        lists = c["w"] * c["h"]
        return {"bytes": b + lists * (c["ns"] * (24 + slot) + 12), "flops": f + 20 * lists * c["ns"]}
    # generation and direct rendering: each sample's interpolation, classification and compositing
    samples = min(1.0, 0.46 * c["h"] / c["w"]) * c["w"] * c["h"] * 0.8 * c["n"]
    bytes_, flops = c["n"] ** 3 * vox, 60 * samples
    if kind == "generate":
        bytes_ += c["w"] * c["h"] * (c["ns"] * slot + 8)
        flops += 20 * 20 * samples if c["adaptive"] else 0
        views = [0.0, c["angle"]]
        if c["download"]:
            views, bytes_ = [], bytes_ + c["w"] * c["h"] * c["ns"] * 24
    else:
        views, bytes_, flops = [c["angle"]], bytes_ + 3 * c["w"] * c["h"] * 16, flops / c["step"]
    for a in views:
        b, f = _view_work(c["w"], c["h"], c["ns"], c["fmt"], c["w"], c["h"], a, 1.0, 1, 1, 16)
        bytes_, flops = bytes_ + b, flops + f
    return {"bytes": float(bytes_), "flops": float(flops)}


# ---------------------------------------------------------------------------
# exact: the same results in plain torch
# ---------------------------------------------------------------------------


def _t32(x):
    return torch.tensor(float(np.float32(x)), device=DEV, dtype=torch.float32)


def _rays32(view, proj, w, h, n):
    """The generation rays in IEEE FP32: (list indices, origin, direction, t0, dt, samples, |direction|) of the rays that meet the box."""
    vi = np.linalg.inv(view)
    d0 = vi[:3, :3] @ np.array([proj[0, 2] / proj[0, 0], proj[1, 2] / proj[1, 1], -1.0])
    E = [_t32(v) for v in vi[:3, 3]]
    D0, Dx, Dy = ([_t32(v) for v in col] for col in (d0, vi[:3, 0] / proj[0, 0], vi[:3, 1] / proj[1, 1]))
    near, far = proj[2, 3] / (proj[2, 2] - 1.0), proj[2, 3] / (proj[2, 2] + 1.0)
    one, two, half = _t32(1.0), _t32(2.0), _t32(0.5)
    py, px = torch.meshgrid(torch.arange(h, device=DEV), torch.arange(w, device=DEV), indexing="ij")
    px, py = px.reshape(-1).float(), py.reshape(-1).float()
    x = (two * (px + half)) / _t32(w).expand_as(px) - one
    y = one - (two * (py + half)) / _t32(h).expand_as(py)
    d = [(D0[k] + x * Dx[k]) + y * Dy[k] for k in range(3)]
    length = torch.sqrt((d[0] * d[0] + d[1] * d[1]) + d[2] * d[2])
    t0, t1 = _t32(near).expand_as(x).clone(), _t32(far).expand_as(x).clone()
    hit = torch.ones_like(x, dtype=torch.bool)
    for k in range(3):
        lo, hi = _t32(BMIN[k]), _t32(BMAX[k])
        flat = d[k] == 0
        ta, tb = (lo - E[k]).expand_as(x) / d[k], (hi - E[k]).expand_as(x) / d[k]
        ta, tb = torch.minimum(ta, tb), torch.maximum(ta, tb)
        t0 = torch.where(~flat & (ta > t0), ta, t0)
        t1 = torch.where(~flat & (tb < t1), tb, t1)
        hit &= ~(flat & ((E[k] < lo) | (E[k] > hi)))
    hit &= t0 < t1
    step = _t32(n)
    K = torch.floor(((t1 - t0) * length) / step.expand_as(x))
    dt = step.expand_as(x) / length
    at = torch.nonzero(hit & (K > 0)).reshape(-1)
    return at, E, [v[at] for v in d], t0[at], dt[at], K[at].long(), length[at]


def _sampler(vol, kind, n):
    """value(p) and classify(v) in the arithmetic type of their arguments."""
    flat = vol.view(torch.int16).reshape(-1) if vol.dtype == torch.uint16 else vol.reshape(-1)
    top = {torch.uint8: 255.0, torch.uint16: 65535.0}.get(vol.dtype)
    knots = np.asarray(KNOTS[kind], np.float32)

    def value(p):
        dt = p[0].dtype
        i0, i1, fr = [], [], []
        for k in range(3):
            q = (p[k] - float(BMIN[k])) / torch.full_like(p[k], float(BMAX[k] - BMIN[k])) * float(n) - 0.5
            fl = torch.floor(q)
            fr.append(q - fl)
            i0.append(fl.long().clamp(0, n - 1))
            i1.append((fl.long() + 1).clamp(0, n - 1))

        def voxel(i, j, k):
            v = flat[(k * n + j) * n + i]
            if vol.dtype == torch.uint16:
                v = v.int() & 0xFFFF
            v = v.to(dt)
            return v if top is None else v / torch.full_like(v, top)

        def lerp(a, b, t):
            return a + t * (b - a)

        c = [lerp(voxel(i0[0], j, k), voxel(i1[0], j, k), fr[0]) for k in (i0[2], i1[2]) for j in (i0[1], i1[1])]
        return lerp(lerp(c[0], c[1], fr[1]), lerp(c[2], c[3], fr[1]), fr[2])

    def classify(v):
        kv = torch.tensor(knots[:, 0].copy(), device=DEV).to(v.dtype)
        kc = torch.tensor(knots[:, 1:].copy(), device=DEV).to(v.dtype)
        i = (torch.searchsorted(kv, v.contiguous(), right=True) - 1).clamp(0, len(kv) - 2)
        s = (v - kv[i]) / (kv[i + 1] - kv[i])
        out = kc[i] + s[:, None] * (kc[i + 1] - kc[i])
        out = torch.where((v <= kv[0])[:, None], kc[0][None], out)
        return torch.where((v >= kv[-1])[:, None], kc[-1][None], out)

    return value, classify


def _march32(samples, K, tau, ns, t0, dt, write):
    """Eq. 1 along every ray.  samples(k) -> (alpha, premultiplied rgb) in FP32.
    Counting (write=None): min(count, ns + 1).  Writing: fills write["f" / "b" / "rgb" / "T"]."""
    R = K.shape[0]
    limit = ns if write is not None else ns + 2
    one = _t32(1.0)
    st = dict(nseg=torch.zeros(R, dtype=torch.long, device=DEV), open=torch.zeros(R, dtype=torch.bool, device=DEV),
              cnt=torch.zeros(R, device=DEV), tray=torch.ones(R, device=DEV), mean=torch.zeros(R, 3, device=DEV),
              ts=torch.zeros(R, device=DEV), te=torch.zeros(R, device=DEV), tau2=tau * tau, K=K, t0=t0, dt=dt,
              C=torch.zeros(R, 3, device=DEV, dtype=torch.float64), T=torch.ones(R, device=DEV, dtype=torch.float64),
              at=torch.arange(R, device=DEV))
    total = torch.zeros(R, dtype=torch.long, device=DEV)

    def close(m):
        if write is not None:
            i = torch.nonzero(m).reshape(-1)
            r, j = st["at"][i], st["nseg"][i]
            write["ts"][r, j], write["te"][r, j] = st["ts"][i], st["te"][i]
            write["rgb"][r, j], write["T"][r, j] = st["C"][i], st["T"][i]
        st["nseg"] = st["nseg"] + m
        st["open"] = st["open"] & ~m

    k, last = 0, int(K.max()) if R else 0
    while k < last and st["at"].numel():
        live = (k < st["K"]) & (st["tray"] > ERT)
        if write is None:
            live &= st["nseg"] <= ns
        if k % 32 == 0:  # drop the finished rays
            done = ~live
            if bool(done.any()):
                close(done & st["open"])
                total[st["at"][done]] = st["nseg"][done]
                st = {key: v[live] for key, v in st.items()}
                live = live[live]
                if not st["at"].numel():
                    return total
        a, xc = samples(k, st["at"])
        fk = _t32(float(k))
        on = live & (a > 0)
        cut = live & ~on & st["open"] & (st["nseg"] < limit - 1)
        d = st["mean"] - xc
        dist = (d[:, 0] * d[:, 0] + d[:, 1] * d[:, 1]) + d[:, 2] * d[:, 2]
        cut |= on & st["open"] & (st["nseg"] < limit - 1) & ~(st["tau2"] > dist)
        close(cut)
        new = on & ~st["open"]
        st["open"] = st["open"] | on
        st["ts"] = torch.where(new, st["t0"] + fk * st["dt"], st["ts"])
        st["cnt"] = torch.where(on, torch.where(new, torch.zeros_like(a), st["cnt"]) + one, st["cnt"])
        mean = torch.where(new[:, None], torch.zeros_like(xc), st["mean"])
        st["mean"] = torch.where(on[:, None], mean + (xc - mean) / st["cnt"].clamp(min=1.0)[:, None], mean)
        st["te"] = torch.where(on, st["t0"] + _t32(float(k + 1)) * st["dt"], st["te"])
        st["tray"] = torch.where(on, st["tray"] * (one - a), st["tray"])
        if write is not None:
            T = torch.where(new, torch.ones_like(st["T"]), st["T"])
            C = torch.where(new[:, None], torch.zeros_like(st["C"]), st["C"])
            st["C"] = torch.where(on[:, None], C + T[:, None] * xc.double(), C)
            st["T"] = torch.where(on, T * (1.0 - a.double()), T)
        k += 1
    close(st["open"])
    total[st["at"]] = st["nseg"]
    return total


def _generate(vol, kind, n, w, h, ns, view, proj, adaptive):
    """Lists as dense arrays: FP32 depths f, b [w h, ns] (+inf unused), FP64 colours chat [., ., 3] and kappa, counts, tau."""
    at, E, d, t0, dt, K, length = _rays32(view, proj, w, h, 1.0 / n)
    value, classify = _sampler(vol, kind, n)
    half = _t32(0.5)

    def sample(k, i):
        tm = t0[i] + (_t32(float(k)) + half) * dt[i]
        tf = classify(value([E[c] + tm * d[c][i] for c in range(3)]))
        return tf[:, 3], tf[:, :3] * tf[:, 3:]

    R = at.numel()
    tau = torch.full((R,), float(np.float32(TAU[kind])), device=DEV)
    if adaptive and R:
        a_all = torch.zeros(int(K.max()), R, device=DEV)
        x_all = torch.zeros(int(K.max()), R, 3, device=DEV)
        for k in range(int(K.max())):
            a_all[k], x_all[k] = sample(k, torch.arange(R, device=DEV))

        def sample(k, i):  # noqa: F811
            return a_all[k][i], x_all[k][i]

        low, high = torch.zeros(R, device=DEV), torch.full((R,), float(np.float32(math.sqrt(3.0))), device=DEV)
        gamma, found = torch.full((R,), float(np.float32(1e-5)), device=DEV), torch.zeros(R, dtype=torch.bool, device=DEV)
        first = True
        while not bool(found.all()):
            i = torch.nonzero(~found).reshape(-1)
            c = _march32(lambda k, j: sample(k, i[j]), K[i], gamma[i], ns, t0[i], dt[i], None)
            g, lo, hi = gamma[i], low[i], high[i]
            end = (hi - lo) < _t32(1e-6)
            more, fewer = ~end & (c > ns), ~end & (c < ns - (15 * ns) // 100)
            stop = end | ~(more | fewer) | (first & (c < ns))
            low[i], high[i] = torch.where(more, g, lo), torch.where(fewer, g, hi)
            g = torch.where(end, hi, g)
            gamma[i] = torch.where(stop, g, (low[i] + high[i]) / torch.full_like(g, 2.0))
            found[i] = stop
            first = False
        tau = gamma
    buf = dict(ts=torch.ones(R, ns, device=DEV), te=torch.ones(R, ns, device=DEV),
               rgb=torch.zeros(R, ns, 3, device=DEV, dtype=torch.float64), T=torch.ones(R, ns, device=DEV, dtype=torch.float64))
    cnt = _march32(sample, K, tau, ns, t0, dt, buf)
    used = torch.arange(ns, device=DEV)[None] < cnt[:, None]
    P22, P23 = _t32(proj[2, 2]), _t32(proj[2, 3])
    inf = torch.full_like(buf["ts"], math.inf)
    f = torch.full((w * h, ns), math.inf, device=DEV)
    b = f.clone()
    f[at] = torch.where(used, P23.expand_as(inf) / buf["ts"] - P22, inf)
    b[at] = torch.where(used, P23.expand_as(inf) / buf["te"] - P22, inf)
    lu = (buf["te"].double() - buf["ts"].double()) * length.double()[:, None] * n
    alpha = 1.0 - buf["T"]
    chat = torch.zeros(w * h, ns, 3, device=DEV, dtype=torch.float64)
    kappa = torch.zeros(w * h, ns, device=DEV, dtype=torch.float64)
    chat[at] = torch.where(used[..., None], (buf["rgb"] / alpha.clamp(min=1e-300)[..., None]).clamp(max=1.0), 0.0)
    kappa[at] = torch.where(used & (lu > 0), -torch.log2(buf["T"]) / lu, 0.0)
    counts = torch.zeros(w * h, dtype=torch.int32, device=DEV)
    counts[at] = cnt.int()
    g = torch.full((w * h,), float(np.float32(1e-5)) if adaptive else float(np.float32(TAU[kind])), device=DEV)
    g[at] = tau
    return dict(w=w, h=h, ns=ns, f=f, b=b, chat=chat, kappa=kappa, counts=counts, tau=g, view=view, proj=proj, u=1.0 / n)


def _edges(proj, nz=20):
    dn, df = ((proj[2, 3]) / (z + proj[2, 2]) for z in (-1.0, 1.0))
    depth = dn + (df - dn) * np.arange(nz + 1) / nz
    e = ((proj[2, 2] * -depth + proj[2, 3]) / depth).astype(np.float32)
    e[0], e[-1] = -1.0, 1.0
    return e, float(df - dn) / nz


def _grid(L, T=8, nz=20):
    """Supersegment counts [nz, gh, gw] over cells of T x T lists by equal view-depth slabs."""
    e, _ = _edges(L["proj"], nz)
    gw, gh = -(-L["w"] // T), -(-L["h"] // T)
    f, b = L["f"], L["b"]
    out = torch.zeros(nz, gh, gw, dtype=torch.long, device=DEV)
    for k in range(nz):
        hit = torch.where(f == b, (f >= float(e[k])) & (f < float(e[k + 1])), (f < float(e[k + 1])) & (b > float(e[k])))
        c = (hit & torch.isfinite(f)).sum(1).view(L["h"], L["w"])
        c = torch.nn.functional.pad(c, (0, gw * T - L["w"], 0, gh * T - L["h"]))
        out[k] = c.view(gh, T, gw, T).sum((1, 3))
    return out


def _ndc_rays(L, view, proj, W, H):
    """FP64 rays of a W x H image as segments in the VDI's clip space, clipped to the box and both frusta:
    (pixel indices, h0, h1 [R, 4], world length of the segment in length units)."""
    f64 = dict(device=DEV, dtype=torch.float64)
    q = torch.tensor(np.linalg.inv(proj @ view), **f64)
    y, x = torch.meshgrid(1 - (torch.arange(H, **f64) + 0.5) * (2.0 / H), (torch.arange(W, **f64) + 0.5) * (2.0 / W) - 1,
                          indexing="ij")
    x, y = x.reshape(-1), y.reshape(-1)
    ends = []
    for z in (-1.0, 1.0):
        p = torch.stack([x, y, torch.full_like(x, z), torch.ones_like(x)], 1) @ q.T
        ends.append(p[:, :3] / p[:, 3:])
    o, d = ends[0], ends[1] - ends[0]
    t0, t1 = torch.zeros_like(x), torch.ones_like(x)
    for k in range(3):
        inv = 1.0 / d[:, k]
        a, b = (float(BMIN[k]) - o[:, k]) * inv, (float(BMAX[k]) - o[:, k]) * inv
        flat = d[:, k] == 0
        inside = (o[:, k] >= float(BMIN[k])) & (o[:, k] <= float(BMAX[k]))
        big = torch.full_like(a, math.inf)
        a, b = torch.where(flat, torch.where(inside, -big, big), a), torch.where(flat, big, b)
        t0, t1 = torch.maximum(t0, torch.minimum(a, b)), torch.minimum(t1, torch.maximum(a, b))
    m = torch.tensor(L["proj"] @ L["view"], **f64)
    ha = torch.cat([o, torch.ones_like(o[:, :1])], 1) @ m.T
    hb = torch.cat([d, torch.zeros_like(o[:, :1])], 1) @ m.T
    for k in range(3):
        for s in (1.0, -1.0):
            c0, c1 = ha[:, 3] + s * ha[:, k], hb[:, 3] + s * hb[:, k]
            t = -c0 / c1
            t0 = torch.where(c1 > 0, torch.maximum(t0, t), t0)
            t1 = torch.where(c1 < 0, torch.minimum(t1, t), t1)
            t1 = torch.where((c1 == 0) & (c0 < 0), torch.full_like(t1, -1.0), t1)
    at = torch.nonzero(t0 < t1).reshape(-1)
    t0, t1 = t0[at, None], t1[at, None]
    ha, hb = ha[at], hb[at]
    length = (d[at].norm(dim=1) * (t1 - t0)[:, 0]) / L["u"]
    return at, ha + t0 * hb, ha + t1 * hb, length


def _to_grid(L, h):
    p = h[:, :3] / h[:, 3:]
    return (p[:, 0] + 1) * 0.5 * L["w"], (1 - p[:, 1]) * 0.5 * L["h"], p[:, 2]


def _exact_rays(L, view, proj, W, H):
    """Every list crossed, every supersegment overlapped, Eq. 2, front to back."""
    at, h0, h1, length = _ndc_rays(L, view, proj, W, H)
    gx0, gy0, z0 = _to_grid(L, h0)
    gx1, gy1, z1 = _to_grid(L, h1)
    img = torch.zeros(W * H, 4, device=DEV, dtype=torch.float64)
    w, h, big = L["w"], L["h"], torch.full_like(z0, math.inf)
    dx, dy, dz = gx1 - gx0, gy1 - gy0, z1 - z0
    r = dict(ix=gx0.floor().long().clamp(0, w - 1), iy=gy0.floor().long().clamp(0, h - 1), s=torch.zeros_like(z0), gx0=gx0,
             gy0=gy0, dx=dx, dy=dy, z0=z0, dz=dz, w0=h0[:, 3].clone(), w1=h1[:, 3].clone(), ln=length, at=at,
             acc=torch.zeros(at.numel(), 3, device=DEV, dtype=torch.float64), T=torch.ones_like(z0))
    for _ in range(w + h + 2):
        if not r["at"].numel():
            break
        big = torch.full_like(r["s"], math.inf)
        bx, by = r["ix"] + (r["dx"] > 0), r["iy"] + (r["dy"] > 0)
        sx = torch.where(r["dx"] != 0, (bx - r["gx0"]) / r["dx"], big)
        sy = torch.where(r["dy"] != 0, (by - r["gy0"]) / r["dy"], big)
        so = torch.minimum(torch.minimum(sx, sy), torch.ones_like(sx))
        li = r["iy"] * w + r["ix"]
        f, b = L["f"][li].double(), L["b"][li].double()
        din, dout = r["z0"] + r["s"] * r["dz"], r["z0"] + so * r["dz"]
        lo, hi = torch.minimum(din, dout)[:, None], torch.maximum(din, dout)[:, None]
        idz = (1.0 / r["dz"])[:, None]
        inside = (b >= lo) & (f <= hi)
        za, zb = torch.maximum(f, lo), torch.minimum(b, hi)
        za, zb = torch.where(inside, za, lo), torch.where(inside, zb, lo)
        sa, sb = (za - r["z0"][:, None]) * idz, (zb - r["z0"][:, None]) * idz
        down = (r["dz"] < 0)[:, None]
        sa, sb = torch.where(down, sb, sa), torch.where(down, sa, sb)
        full_a, full_b = torch.where(down, b >= hi, f <= lo), torch.where(down, f <= lo, b >= hi)
        s0, s1 = r["s"][:, None], torch.maximum(so, r["s"])[:, None]
        sa, sb = torch.where(full_a, s0, sa).clamp(s0, s1), torch.where(full_b, s1, sb).clamp(s0, s1)
        D = r["w1"][:, None] + torch.stack([sa, sb]) * (r["w0"] - r["w1"])[:, None]
        ln = (r["ln"] * r["w0"] * r["w1"])[:, None] * (sb - sa).clamp(min=0) / (D[0] * D[1])
        ln = torch.where(inside, ln, torch.zeros_like(ln))
        dep = torch.where(ln > 0, L["kappa"][li] * ln, torch.zeros_like(ln))
        chat = L["chat"][li]
        if bool(down.any()):
            dep = torch.where(down, dep.flip(1), dep)
            chat = torch.where(down[..., None], chat.flip(1), chat)
        after = torch.cumsum(dep, 1)
        before = r["T"][:, None] * torch.exp2(-(after - dep).clamp(min=0))
        alive = before > ERT
        e = torch.exp2(-dep)
        wgt = torch.where(alive, before * (1 - e), torch.zeros_like(e))
        r["acc"] = r["acc"] + (wgt[..., None] * chat).sum(1)
        r["T"] = r["T"] * torch.exp2(-torch.where(alive, dep, torch.zeros_like(dep)).sum(1))
        xs = sx <= sy
        r["ix"] = torch.where(xs, r["ix"] + torch.where(r["dx"] > 0, 1, -1), r["ix"])
        r["iy"] = torch.where(xs, r["iy"], r["iy"] + torch.where(r["dy"] > 0, 1, -1))
        r["s"] = torch.maximum(r["s"], so)
        on = (so < 1) & (r["T"] > ERT) & (r["ix"] >= 0) & (r["ix"] < w) & (r["iy"] >= 0) & (r["iy"] < h)
        if not bool(on.all()):
            end = ~on
            img[r["at"][end]] = torch.cat([r["acc"][end], (1 - r["T"][end])[:, None]], 1)
            r = {k: v[on] for k, v in r.items()}
    return img.view(H, W, 4)


def _preview_rays(L, view, proj, W, H, d_r, T=8, nz=20):
    """Per grid cell crossed: ceil((count / lists) (length / slab extent) / D_R) samples at equal world spacing."""
    at, h0, h1, length = _ndc_rays(L, view, proj, W, H)
    edges, dz_cell = _edges(L["proj"], nz)
    scale = L["u"] / (dz_cell * d_r)
    e = torch.tensor(edges, device=DEV).double()
    grid = _grid(L, T, nz)
    gx0, gy0, z0 = _to_grid(L, h0)
    gx1, gy1, z1 = _to_grid(L, h1)
    w, h, gw, gh = L["w"], L["h"], grid.shape[2], grid.shape[1]
    img = torch.zeros(W * H, 4, device=DEV, dtype=torch.float64)
    cz = (torch.searchsorted(e[1:-1].contiguous(), z0.contiguous(), right=True)).clamp(0, nz - 1)
    r = dict(cx=(gx0.clamp(min=0) / T).floor().long().clamp(0, gw - 1), cy=(gy0.clamp(min=0) / T).floor().long().clamp(0, gh - 1),
             cz=cz, s=torch.zeros_like(z0), gx0=gx0, gy0=gy0, dx=gx1 - gx0, dy=gy1 - gy0, z0=z0, dz=z1 - z0, ln=length, at=at,
             h0=h0, h1=h1, acc=torch.zeros(at.numel(), 3, device=DEV, dtype=torch.float64), T=torch.ones_like(z0))
    for step in range(gw + gh + nz + 3):
        if not r["at"].numel():
            break
        big = torch.full_like(r["s"], math.inf)
        bx, by = (r["cx"] + (r["dx"] > 0)) * T, (r["cy"] + (r["dy"] > 0)) * T
        sx = torch.where(r["dx"] != 0, (bx - r["gx0"]) / r["dx"], big)
        sy = torch.where(r["dy"] != 0, (by - r["gy0"]) / r["dy"], big)
        sz = torch.where(r["dz"] != 0, (e[r["cz"] + (r["dz"] >= 0)] - r["z0"]) / r["dz"], big)
        so = torch.minimum(torch.minimum(sx, sy), torch.minimum(sz, torch.ones_like(sz)))
        cnt = grid[r["cz"], r["cy"], r["cx"]].double()
        lists = ((w - r["cx"] * T).clamp(max=T) * (h - r["cy"] * T).clamp(max=T)).double()
        w0, w1 = r["h0"][:, 3], r["h1"][:, 3]
        ua = r["s"] * w0 / (w1 + r["s"] * (w0 - w1))
        ub = so * w0 / (w1 + so * (w0 - w1))
        lc = r["ln"] * (ub - ua)
        n = torch.where((cnt > 0) & (so > r["s"]), (cnt / lists * lc * scale).ceil().clamp(min=1), torch.zeros_like(cnt)).long()
        for k in range(int(n.max()) if n.numel() else 0):
            i = torch.nonzero(k < n).reshape(-1)
            u = ua[i] + (k + 0.5) * (ub - ua)[i] / n[i]
            gx, gy, z = _to_grid(L, r["h0"][i] + u[:, None] * (r["h1"] - r["h0"])[i])
            li = gy.floor().long().clamp(0, h - 1) * w + gx.floor().long().clamp(0, w - 1)
            f, b = L["f"][li].double(), L["b"][li].double()
            j = (b < z[:, None]).sum(1).clamp(max=L["ns"] - 1)[:, None]
            hit = (f.gather(1, j)[:, 0] <= z) & (b.gather(1, j)[:, 0] >= z)
            ex = torch.exp2(-torch.where(hit, L["kappa"][li].gather(1, j)[:, 0] * (lc / n)[i], torch.zeros_like(z)))
            chat = L["chat"][li, j[:, 0]]
            r["acc"][i] += (r["T"][i] * (1 - ex))[:, None] * chat
            r["T"][i] *= ex
        xs, ys = (sx <= sy) & (sx <= sz), sy <= sz
        r["cx"] = torch.where(xs, r["cx"] + torch.where(r["dx"] > 0, 1, -1), r["cx"])
        r["cy"] = torch.where(~xs & ys, r["cy"] + torch.where(r["dy"] > 0, 1, -1), r["cy"])
        r["cz"] = torch.where(~xs & ~ys, r["cz"] + torch.where(r["dz"] >= 0, 1, -1), r["cz"])
        r["s"] = torch.maximum(r["s"], so)
        on = (so < 1) & (r["cx"] >= 0) & (r["cx"] < gw) & (r["cy"] >= 0) & (r["cy"] < gh) & (r["cz"] >= 0) & (r["cz"] < nz)
        if step % 8 == 7:  # early termination is checked once per eight cells
            on &= r["T"] > ERT
        if not bool(on.all()):
            end = ~on
            img[r["at"][end]] = torch.cat([r["acc"][end], (1 - r["T"][end])[:, None]], 1)
            r = {k: v[on] for k, v in r.items()}
    return img.view(H, W, 4)


def _upsample(lo, W, H):
    h0, w0 = lo.shape[:2]
    u = (torch.arange(W, device=DEV, dtype=torch.float64) + 0.5) * (w0 / W) - 0.5
    v = (torch.arange(H, device=DEV, dtype=torch.float64) + 0.5) * (h0 / H) - 0.5
    i, j = u.floor().long(), v.floor().long()
    fu, fv = (u - i)[None, :, None], (v - j)[:, None, None]
    ia, ib, ja, jb = i.clamp(0, w0 - 1), (i + 1).clamp(0, w0 - 1), j.clamp(0, h0 - 1), (j + 1).clamp(0, h0 - 1)
    top = lo[ja][:, ia] * (1 - fu) + lo[ja][:, ib] * fu
    bot = lo[jb][:, ia] * (1 - fu) + lo[jb][:, ib] * fu
    return top * (1 - fv) + bot * fv


def _view(L, view, proj, W, H, d_i=1, d_r=1):
    Wr, Hr = -(-W // d_i), -(-H // d_i)
    img = _exact_rays(L, view, proj, Wr, Hr) if d_r == 1 else _preview_rays(L, view, proj, Wr, Hr, d_r)
    return img if d_i == 1 else _upsample(img, W, H)


def _dvr(vol, kind, n, view, proj, w, h, step):
    at, E, d, t0, dt, K, _ = _rays32(view, proj, w, h, step / n)
    E, d, t0, dt = [v.double() for v in E], [v.double() for v in d], t0.double(), dt.double()
    value, classify = _sampler(vol, kind, n)
    img = torch.zeros(w * h, 4, device=DEV, dtype=torch.float64)
    acc = torch.zeros(at.numel(), 3, device=DEV, dtype=torch.float64)
    T = torch.ones(at.numel(), device=DEV, dtype=torch.float64)
    live = torch.arange(at.numel(), device=DEV)
    for k in range(int(K.max())):
        if k % 16 == 0:
            live = live[(K[live] > k) & (T[live] > ERT)]
        tm = t0[live] + (k + 0.5) * dt[live]
        tf = classify(value([E[c] + tm * d[c][live] for c in range(3)]))
        a = tf[:, 3] if step == 1.0 else 1 - (1 - tf[:, 3]) ** step
        a = torch.where((K[live] > k) & (T[live] > ERT), a, torch.zeros_like(a))
        acc[live] += (T[live] * a)[:, None] * tf[:, :3]
        T[live] *= 1 - a
    img[at] = torch.cat([acc, (1 - T)[:, None]], 1)
    return img.view(h, w, 4)


def _ssim_psnr(a, b):
    a, b = a[..., :3].permute(2, 0, 1)[:, None], b[..., :3].permute(2, 0, 1)[:, None]

    def box(x):
        return torch.nn.functional.avg_pool2d(x, 7, 1)

    ma, mb = box(a), box(b)
    k = 49.0 / 48.0
    vaa, vbb, vab = (k * (box(a * a) - ma * ma), k * (box(b * b) - mb * mb), k * (box(a * b) - ma * mb))
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    s = ((2 * ma * mb + c1) * (2 * vab + c2)) / ((ma * ma + mb * mb + c1) * (vaa + vbb + c2))
    return float(s.mean()), float(10 * torch.log10(1.0 / ((a - b) ** 2).mean()))


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind == "create":
        rgba, depth, counts = layers(c["w"], c["h"], c["ns"], seed)
        alpha = rgba[..., 3].double().reshape(-1, c["ns"])
        chat = rgba[..., :3].double().reshape(-1, c["ns"], 3) / alpha.clamp(min=1e-300)[..., None]
        view, proj = orbit(c["w"] / c["h"], 0.0, ELEVATION["layers"])
        L = dict(w=c["w"], h=c["h"], ns=c["ns"], f=depth[..., 0].reshape(-1, c["ns"]), b=depth[..., 1].reshape(-1, c["ns"]),
                 chat=chat.clamp(max=1.0), kappa=-torch.log2(1 - alpha), view=view, proj=proj, u=1.0 / 64)
        return _view(L, *orbit(c["w"] / c["h"], c["angle"], ELEVATION["layers"]), c["w"], c["h"])
    if kind == "batch":
        vdis, reqs = batch_plan(c, seed)
        Ls = []
        for k, (w, h, ns) in enumerate(vdis):
            vol = noise_volume(c["n"], seed + 10 * k, u8=True)
            Ls.append(_generate(vol, "noise", c["n"], w, h, ns, *orbit(w / h, 90.0 * k, 20.0), False))
        return [_view(Ls[k], *orbit(W / H, 90.0 * k + a, 20.0), W, H, d_i, d_r) for k, W, H, a, d_i, d_r in reqs]
    vol, el = volume(c["vol"], c["n"], seed), ELEVATION[c["vol"]]
    vo = orbit(c["w"] / c["h"], 0.0, el)
    L = _generate(vol, c["vol"], c["n"], c["w"], c["h"], c["ns"], *vo, bool(c.get("adaptive")))
    if kind == "render":
        return _view(L, *orbit(c["W"] / c["H"], c["angle"], el, c["zoom"]), c["W"], c["H"], c["d_i"], c["d_r"])
    turned = orbit(c["w"] / c["h"], c["angle"], el)
    if kind == "generate":
        if c["download"]:
            shape = (c["h"], c["w"], c["ns"])
            alpha = 1 - torch.exp2(-L["kappa"])
            r = {"rgba": torch.cat([L["chat"] * alpha[..., None], alpha[..., None]], -1).view(*shape, 4),
                 "depth": torch.stack([L["f"], L["b"]], -1).double().view(*shape, 2), "counts": L["counts"].view(c["h"], c["w"]),
                 "grid": _grid(L)}
        else:
            r = {"images": [_view(L, *v, c["w"], c["h"]) for v in (vo, turned)]}
        if c["adaptive"]:
            r["tau"] = L["tau"].double().view(c["h"], c["w"])
        return r
    dvr = _dvr(vol, c["vol"], c["n"], *turned, c["w"], c["h"], c["step"])
    ren = _view(L, *turned, c["w"], c["h"])
    ssim, psnr = _ssim_psnr(ren, dvr)
    return {"dvr": dvr, "render": ren, "ssim": ssim, "psnr": psnr}
