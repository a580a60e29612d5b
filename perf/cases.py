"""The work this library is asked to do, as cases to be timed: single frames
from thumbnails to 3M Gaussians at 1256x832, the 8-resolution sweep of one
pose, training steps (forward and backward), a served batch of requests and
the insertion of a coarse level.

Every case goes through the package's public calls on seeded synthetic
scenes of the recipes in paper_2311_17089_gb300/inputs.py (four-level
clustered scenes, single-level RGB scenes, dense foreground with a far
shell), drawn on the GPU, with coverage ranges as a trained model has them.

listed() names the cases, draw() gives others of the same ranges, prepare()
makes what a program holds before the call, run() is one pass, work() says
what a pass cannot do without, and exact() is the same result in FP64 with
plain torch.
"""
import math
import weakref

import numpy as np
import torch

import paper_2311_17089_gb300 as msgs
from paper_2311_17089_gb300 import autograd, inputs

SPLIT = (0.70, 0.20, 0.07, 0.03)  # Gaussians on levels 1 .. 4
SWEEP = (1, 2, 4, 8, 16, 32, 64, 128)


def listed():
    return [
        # the smallest call: a thumbnail of a small scene (launches and latency)
        {"name": "frame 96x80 4k", "kind": "frame", "scene": "clusters", "n": 4000, "sh": 3,
         "width": 96, "height": 80, "scale": 1, "mode": "selective", "radius": 4.0},
        # a single-scale model with plain RGB colours in a small viewport
        {"name": "frame 256x256 10k rgb", "kind": "frame", "scene": "single", "n": 10000,
         "sh": -1, "width": 256, "height": 256, "scale": 1, "mode": "all_levels", "radius": 3.0},
        # a mid-size scene at an odd size, degree-2 colours, the small-splat
        # filter alone (the "Filter Small" rendering mode)
        {"name": "frame 333x217 50k filter", "kind": "frame", "scene": "clusters", "n": 50001,
         "sh": 2, "width": 333, "height": 217, "scale": 1, "mode": "filter_small",
         "radius": 25.0},
        # the ordinary frame: a trained scene at full resolution
        {"name": "frame 1256x832 1M", "kind": "frame", "scene": "clusters", "n": 1000000,
         "sh": 3, "width": 1256, "height": 832, "scale": 1, "mode": "selective",
         "radius": 25.0},
        # the same scene seen small (8x downscale: few tiles, long lists)
        {"name": "frame 157x104 1M", "kind": "frame", "scene": "clusters", "n": 1000000,
         "sh": 3, "width": 1256, "height": 832, "scale": 8, "mode": "selective",
         "radius": 25.0},
        # every level rendered together (no selection): long tile lists
        {"name": "frame 628x416 1M all", "kind": "frame", "scene": "clusters", "n": 1000000,
         "sh": 3, "width": 1256, "height": 832, "scale": 2, "mode": "all_levels",
         "radius": 25.0},
        # a large unbounded scene: dense foreground, far background shell
        {"name": "frame 1256x832 3M near/far", "kind": "frame", "scene": "nearfar", "n": 3000000,
         "sh": 3, "width": 1256, "height": 832, "scale": 1, "mode": "selective",
         "radius": 12.0},
        # one pose at 1x .. 128x, the frames side by side, replayed from a
        # captured graph as a viewer with fixed buffers does
        {"name": "sweep 1x-128x 1M", "kind": "sweep", "scene": "clusters", "n": 1000000, "sh": 3,
         "width": 1256, "height": 832, "mode": "selective", "radius": 25.0},
        # a training step's render and gradients on a small scene
        {"name": "train 2 views 20k", "kind": "train", "scene": "clusters", "n": 20011, "sh": 1,
         "width": 240, "height": 160, "scales": "1,4", "radius": 25.0},
        # a multi-scale training step on a full scene, each view at the
        # creation scale of one level
        {"name": "train 4 views 1M", "kind": "train", "scene": "clusters", "n": 1000000, "sh": 3,
         "width": 1256, "height": 832, "scales": "1,4,16,64", "radius": 25.0},
        # a render server under load: requests for two resident scenes at
        # mixed resolutions and poses, queued at once
        {"name": "serve 32 requests 2x2M", "kind": "serve", "scene": "clusters", "n": 2000000,
         "sh": 3, "width": 1256, "height": 832, "requests": 32, "mode": "selective",
         "radius": 25.0},
        # the insertion of a coarse level from the Gaussians below it
        {"name": "aggregate 1M 8 cameras", "kind": "aggregate", "scene": "clusters", "n": 1000000,
         "sh": 3, "width": 1256, "height": 832, "level_m": 2, "cameras": 8, "radius": 25.0},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(["frame", "sweep", "train", "serve", "aggregate"], [12, 2, 3, 1, 1])[0]
    scene = rng.choice(["clusters", "clusters", "clusters", "single", "nearfar"])
    if kind != "frame":
        scene = "clusters"
    if scene == "single":
        n, radius, sh = _log_uniform(rng, 2000, 60000), rng.uniform(2.5, 4.0), -1
    else:
        n, radius, sh = _log_uniform(rng, 4000, 1500000), rng.uniform(18.0, 30.0), rng.randint(0, 3)
        if scene == "nearfar":
            radius = rng.uniform(6.0, 40.0)
        elif n < 10000:  # the small scenes sit in a unit box
            radius = rng.uniform(3.0, 6.0)
    width = _log_uniform(rng, 64, 1256)
    height = max(16, int(width * rng.uniform(0.5, 1.0)))
    c = {"kind": kind, "scene": scene, "n": n, "sh": sh, "width": width, "height": height,
         "radius": round(radius, 3)}
    if kind == "frame":
        c["scale"] = rng.choice(SWEEP if width >= 256 else (1, 1, 2, 4))
        c["mode"] = rng.choice(["selective", "selective", "all_levels", "filter_small"])
        if scene == "single":
            c["mode"] = "all_levels"
        elif c["mode"] == "all_levels":
            c["n"] = min(n, 900000)
            c["scale"] = max(2, c["scale"])
    elif kind == "sweep":
        c["n"], c["mode"] = min(n, 1000000), "selective"
    elif kind == "train":
        c["n"] = min(n, 900000)
        c["scales"] = rng.choice(["1", "2", "1,4", "4,16", "1,2,4"])
    elif kind == "serve":
        c["n"], c["mode"] = min(n, 1000000), rng.choice(["selective", "all_levels"])
        c["requests"] = rng.randint(1, 24)
        c["width"], c["height"] = min(width, 628), min(height, 416)
    else:
        c["n"], c["level_m"], c["cameras"] = min(n, 900000), rng.randint(2, 4), rng.randint(2, 8)
    return c


# ------------------------------------------------------------ scenes, cameras

def _camera(radius, az, el, width, height):
    """A pinhole on an orbit around the origin, horizontal field of view 60
    degrees, image up = -y: plain numbers."""
    eye = np.array([radius * math.cos(el) * math.sin(az), radius * math.sin(el),
                    -radius * math.cos(el) * math.cos(az)])
    fwd = -eye / np.linalg.norm(eye)
    right = np.cross(np.array([0.0, 1.0, 0.0]), fwd)
    right /= np.linalg.norm(right)
    R = np.stack([right, np.cross(fwd, right), fwd])
    f = 0.5 * width / math.tan(math.radians(30.0))
    return {"R": R.astype(np.float32), "t": (-R @ eye).astype(np.float32),
            "campos": eye.astype(np.float32), "f": f, "width": width, "height": height}


def _at_scale(cam, s):
    return dict(cam, f=cam["f"] / s, width=max(1, cam["width"] // s),
                height=max(1, cam["height"] // s))


def _as_camera(cam):
    f = float(np.float32(cam["f"]))
    return inputs.Camera(cam["R"].copy(), cam["t"].copy(), cam["campos"].copy(), f, f,
                         0.5 * cam["width"], 0.5 * cam["height"], cam["width"], cam["height"])


def _cameras(case, seed):
    """The poses of a case, all from the seed; a train or sweep case has one
    pose, or one per view, at the scales it names."""
    rng = np.random.default_rng(seed + 7919)

    def pose():
        return _camera(case["radius"], rng.uniform(0.0, 2.0 * math.pi),
                       math.radians(rng.uniform(-15.0, 15.0)), case["width"], case["height"])

    kind = case["kind"]
    if kind == "frame":
        return [_at_scale(pose(), case["scale"])]
    if kind == "sweep":
        p = pose()
        return [_at_scale(p, s) for s in SWEEP]
    if kind == "train":
        return [_at_scale(pose(), int(s)) for s in case["scales"].split(",")]
    if kind == "serve":
        return [_at_scale(pose(), SWEEP[k % len(SWEEP)]) for k in range(case["requests"])]
    return [_at_scale(pose(), 4 ** (case["level_m"] - 1)) for _ in range(case["cameras"])]


def _arrays(case, seed):
    """A scene's arrays on the GPU, of the recipe the case names."""
    g = torch.Generator("cuda").manual_seed(seed)
    n, sh = case["n"], case["sh"]

    def rnd(*shape):
        return torch.rand(shape, generator=g, device="cuda")

    def nrm(*shape):
        return torch.randn(shape, generator=g, device="cuda")

    if case["scene"] == "single":
        mean, level = rnd(n, 3) * 2.0 - 1.0, torch.ones(n, dtype=torch.uint8, device="cuda")
        base = torch.full((n,), -3.5, device="cuda")
    else:
        counts = [int(round(n * f)) for f in SPLIT]
        counts[0] += n - sum(counts)
        level = torch.cat([torch.full((c,), l + 1, dtype=torch.uint8, device="cuda")
                           for l, c in enumerate(counts)])
        level = level[torch.randperm(n, generator=g, device="cuda")]
        if case["scene"] == "clusters":
            small = n < 10000  # the small scenes: 8 tight clusters in a unit box
            box, sigma, k = (1.0, 0.3, 8) if small else (10.0, 1.0, 64)
            centres = (rnd(k, 3) * 2.0 - 1.0) * box
            which = torch.randint(0, k, (n,), generator=g, device="cuda")
            mean = (centres[which] + sigma * nrm(n, 3)).clamp(-box, box)
            base = torch.full((n,), -3.5, device="cuda")
        else:
            nf = (2 * n) // 3
            d = torch.nn.functional.normalize(nrm(n, 3), dim=1)
            r = torch.cat([rnd(nf) ** (1.0 / 3.0), 48.0 + 4.0 * rnd(n - nf)])
            mean = d * r[:, None]
            base = torch.where(torch.arange(n, device="cuda") < nf, -3.5, -1.5)
    log_scale = 0.5 * nrm(n, 3) + (base + 1.4 * (level.float() - 1.0))[:, None]
    quat = torch.nn.functional.normalize(nrm(n, 4), dim=1)
    opacity = torch.sigmoid(nrm(n))
    if sh < 0:
        color = rnd(n, 3)
    else:
        color = torch.cat([rnd(n, 1, 3), 0.05 * nrm(n, (sh + 1) ** 2 - 1, 3)], dim=1)
    a = {"mean": mean.contiguous(), "log_scale": log_scale, "quat": quat, "opacity": opacity,
         "color": color.contiguous(), "level": level}
    a["n_levels"] = 1 if case["scene"] == "single" else len(SPLIT)
    a["s_max"], a["s_min"] = _ranges(case, a, seed)
    return a


def _ranges(case, a, seed):
    """Coverage ranges as training leaves them (Eq. 5, each level at its
    creation scale 4^(l-1)) over six orbit cameras; none for one level."""
    n = case["n"]
    smax = torch.zeros(n, device="cuda")
    smin = torch.full((n,), math.inf, device="cuda")
    if a["n_levels"] == 1:
        return smax, smin
    rng = np.random.default_rng(seed + 104729)
    down = 4.0 ** (a["level"].float() - 1.0)
    for k in range(6):
        cam = _camera(case["radius"], rng.uniform(0.0, 2.0 * math.pi),
                      math.radians(rng.uniform(-15.0, 15.0)), case["width"], case["height"])
        with torch.no_grad():
            p = _splat(a, cam, torch.float32)
        S = p["S"] / down
        hit = p["valid"] & (p["ntiles"] > 0)
        smax = torch.where(hit, torch.maximum(0.95 * smax, S), smax)
        smin = torch.where(hit, torch.minimum(1.05 * smin, S), smin)
    return smax, smin


def _device_scene(case, a):
    host = {k: a[k].cpu().numpy() for k in
            ("mean", "log_scale", "quat", "opacity", "color", "level", "s_max", "s_min")}
    return msgs.DeviceScene(inputs.Scene(n_levels=a["n_levels"], sh_degree=case["sh"], **host))


def _capacity(ds, cam, mode):
    """The duplicate capacity a program learns from one binning of the frame."""
    r = msgs.Renderer(ds.n, cam.tiles_x * cam.tiles_y, max(4096, 2 * ds.n), with_cover=False,
                      with_mask=False)
    msgs.ms_project(ds.struct, msgs.camera_struct(cam), msgs.MODES[mode], r.proj)
    r.bin(ds, cam)
    _, d, listed_n = msgs.ms_bin_counts(r.bins)
    return int(1.05 * d) + 1024, listed_n


# ------------------------------------------------------------------- prepare

class State:
    """What a program holds between calls."""


def prepare(case, seed):
    s = State()
    s.kind, s.mode = case["kind"], case.get("mode", "selective")
    a = _arrays(case, seed)
    views = [_as_camera(c) for c in _cameras(case, seed)]
    s.cams = views
    if s.kind == "frame":
        s.ds = _device_scene(case, a)
        cam = views[0]
        s.r = msgs.Renderer(s.ds.n, cam.tiles_x * cam.tiles_y, _capacity(s.ds, cam, s.mode)[0],
                            with_cover=False, with_mask=False)
    elif s.kind == "sweep":
        s.ds = _device_scene(case, a)
        caps, counts = zip(*[_capacity(s.ds, c, s.mode) for c in views])
        s.rs = [msgs.Renderer(s.ds.n, c.tiles_x * c.tiles_y, cap, with_cover=False,
                              with_mask=False) for c, cap in zip(views, caps)]
        s.outs = [r.images(c) for r, c in zip(s.rs, views)]
        s.streams = [torch.cuda.Stream(priority=-1 if k < 3 else 0) for k in range(len(views))]
        s.order = msgs.DepthOrder(s.ds.n, split_views=len(views)
                                  if msgs.depth_order_plan(counts)[1] else 0)

        def sweep():
            msgs.render_views(s.ds, s.rs, views, s.mode, s.outs, s.streams, order=s.order,
                              share_sms=True)
        sweep()
        torch.cuda.synchronize()
        s.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s.graph):
            sweep()
    elif s.kind == "train":
        ds = _device_scene(case, a)
        s.frames = [autograd.Frame(ds.n, c, _capacity(ds, c, s.mode)[0]) for c in views]
        s.params = {k: a[k].requires_grad_() for k in
                    ("mean", "log_scale", "quat", "opacity", "color")}
        s.rest = (a["level"], a["s_max"], a["s_min"], a["n_levels"], case["sh"])
        s.targets = _targets(views, seed)
    elif s.kind == "serve":
        s.scenes = [_device_scene(case, a), _device_scene(case, _arrays(case, seed + 1))]
        server = msgs.Server(case["n"], case["width"], case["height"], 16 << 30)
        weakref.finalize(s, server.close)
        s.server = server
        s.ids = [server.add_scene(d) for d in s.scenes]
        s.images = [torch.empty((3, c.height, c.width), device="cuda") for c in views]
    else:
        # buffers for the new Gaussians, sized for the worst case (one each)
        s.ds = _device_scene(case, a)
        n, dev = s.ds.n, s.ds.mean.device
        s.new = {"mean": torch.zeros((n, 3), device=dev), "log_scale": torch.zeros((n, 3), device=dev),
                 "quat": torch.zeros((n, 4), device=dev), "opacity": torch.zeros(n, device=dev),
                 "color": torch.zeros_like(s.ds.color),
                 "level": torch.zeros(n, dtype=torch.uint8, device=dev),
                 "s_max": torch.zeros(n, device=dev), "s_min": torch.zeros(n, device=dev),
                 "count": torch.zeros(2, dtype=torch.int64, device=dev)}
        s.out = msgs.ms_scene_t(n, s.ds.n_levels, s.ds.sh_degree,
                                *(s.new[k].data_ptr() for k in
                                  ("mean", "log_scale", "quat", "opacity", "color", "level",
                                   "s_max", "s_min")), 0, 0)
        s.ws = torch.empty(msgs.ms_aggregate_workspace_bytes(n), dtype=torch.uint8, device=dev)
        s.structs = [msgs.camera_struct(c) for c in views]
        s.level_m = case["level_m"]
        s.extent = float(max(np.abs(c.campos).max() for c in views))
    return s


def _targets(views, seed):
    g = torch.Generator("cuda").manual_seed(seed + 1)
    return [torch.rand((3, c.height, c.width), generator=g, device="cuda") for c in views]


# ----------------------------------------------------------------------- run

def run(s):
    if s.kind == "frame":
        image, final_t, n_contrib = s.r.render(s.ds, s.cams[0], s.mode)
        return {"image": image, "final_t": final_t, "n_contrib": n_contrib}
    if s.kind == "sweep":
        s.graph.replay()
        return [{"image": i, "final_t": t, "n_contrib": c} for i, t, c in s.outs]
    if s.kind == "train":
        level, smax, smin, n_levels, sh = s.rest
        images = autograd.render_views(s.params, level, smax, smin, n_levels, sh, s.frames, s.mode)
        loss = sum((i - t).abs().mean() for i, t in zip(images, s.targets))
        grads = torch.autograd.grad(loss, list(s.params.values()))
        return {"loss": loss, "images": list(images), "grads": dict(zip(s.params, grads))}
    if s.kind == "serve":
        tickets = [s.server.submit(s.ids[k % 2], c, s.mode, image_dev=s.images[k])
                   for k, c in enumerate(s.cams)]
        for t in tickets:
            r = s.server.wait(t)
            if r.status != msgs.MS_OK:
                raise RuntimeError(f"request status {r.status}")
        return s.images
    msgs.ms_aggregate(s.ds.struct, s.structs, s.level_m, s.extent, s.out, s.ds.n,
                      s.new["count"].data_ptr(), s.ws.data_ptr(), s.ws.numel())
    return s.new


# ---------------------------------------------------------------------- work

def _blends(case, w, h, scale):
    """Pixel-Gaussian evaluations of one frame, about: what the pixels of
    these scenes walk before they end (measured 300 a pixel on the 1M scene
    at full resolution, 600 at 2x, 770 at 4x; all levels end sooner)."""
    per = 3e-4 * case["n"] * min(scale, 4) ** 0.7
    if case["scene"] == "single":
        per = 6e-3 * case["n"]
    if case.get("mode") == "all_levels":
        per *= 0.25
    return w * h * max(1.0, per)


def work(case):
    """Bytes: each Gaussian's geometry (61 B) once a pass, the colours of the
    Gaussians that are drawn (about 0.6 in selective frames), the images; for
    a step also the gradients.  Operations: a footprint is about 300 a view,
    an evaluation about 27 (16 FP32 and an exponential), 60 more backward."""
    n, kind = case["n"], case["kind"]
    sh_b = 12 * (1 if case["sh"] < 0 else (case["sh"] + 1) ** 2)
    cams = _cameras(case, 0)
    pix = sum(c["width"] * c["height"] for c in cams)
    drawn = 1.0 if case.get("mode") == "all_levels" or case["scene"] == "single" else 0.6
    if kind in ("sweep", "train"):
        drawn = min(1.0, 0.6 + 0.1 * len(cams))
    scenes = 2 if kind == "serve" else 1
    if kind == "aggregate":
        # geometry once, the pooled parameters of the lower levels, 5% as many new ones
        return {"bytes": n * 61 + 0.75 * n * (sh_b + 44) + 0.05 * n * (sh_b + 53),
                "flops": 300.0 * n * len(cams)}
    ev = sum(_blends(case, c["width"], c["height"], case["width"] / max(1, c["width"]))
             for c in cams)
    work_b = scenes * n * (61 + drawn * sh_b) + 20 * pix
    flops = 300.0 * n * len(cams) + 27.0 * ev
    if kind == "train":
        work_b += n * (44 + sh_b) + n * (44 + drawn * sh_b) + 24 * pix
        flops += 60.0 * ev + 600.0 * n * len(cams)
    return {"bytes": float(work_b), "flops": float(flops)}


# --------------------------------------------- the same results in 64 bits

def _sh_color(color, d):
    """max(0, sum_k f_k Y_k(d) + 0.5), the real orthonormal basis to degree 3."""
    if color.dim() == 2:
        return color
    x, y, z = d.unbind(1)
    xx, yy, zz = x * x, y * y, z * z
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if color.shape[1] > 1:
        c1 = math.sqrt(3 / (4 * pi))
        Y += [c1 * y, c1 * z, c1 * x]
    if color.shape[1] > 4:
        c2 = 0.5 * math.sqrt(15 / pi)
        Y += [c2 * x * y, c2 * y * z, 0.25 * math.sqrt(5 / pi) * (2 * zz - xx - yy), c2 * x * z,
              0.5 * c2 * (xx - yy)]
    if color.shape[1] > 9:
        a, b = 0.25 * math.sqrt(35 / (2 * pi)), 0.5 * math.sqrt(105 / pi)
        c, e = 0.25 * math.sqrt(21 / (2 * pi)), 0.25 * math.sqrt(7 / pi)
        Y += [a * y * (3 * xx - yy), b * x * y * z, c * y * (4 * zz - xx - yy),
              e * z * (2 * zz - 3 * xx - 3 * yy), c * x * (4 * zz - xx - yy),
              0.5 * b * z * (xx - yy), a * x * (xx - 3 * yy)]
    return (torch.einsum("nkc,nk->nc", color, torch.stack(Y, 1)) + 0.5).clamp_min(0.0)


def _splat(a, cam, dtype, color=False):
    """Every Gaussian's splat in one camera (Sec. 3.1, 4.1) with plain torch."""
    R = torch.from_numpy(cam["R"]).to("cuda", dtype)
    t = torch.from_numpy(cam["t"]).to("cuda", dtype)
    f = float(np.float32(cam["f"]))
    W, H = cam["width"], cam["height"]
    mean, q, ls, op = (a[k].to(dtype) for k in ("mean", "quat", "log_scale", "opacity"))
    p = mean @ R.T + t
    tz = p[:, 2]
    xr, yr = p[:, 0] / tz, p[:, 1] / tz
    lx, ly = 1.3 * 0.5 * W / f, 1.3 * 0.5 * H / f
    xc, yc = xr.clamp(-lx, lx), yr.clamp(-ly, ly)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                       2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                       2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)],
                      1).reshape(-1, 3, 3)
    m = rot * ls.exp()[:, None, :]
    zero = torch.zeros_like(tz)
    J = torch.stack([f / tz, zero, -f * xc / tz, zero, f / tz, -f * yc / tz], 1).reshape(-1, 2, 3)
    jm = torch.matmul(torch.matmul(J, R), m)
    V = torch.matmul(jm, jm.transpose(1, 2))
    v00, v01, v11 = V[:, 0, 0], V[:, 0, 1], V[:, 1, 1]
    ca, cc = v00 + 0.3, v11 + 0.3
    detd = ca * cc - v01 * v01
    L = (255.0 * op).log()
    ux, uy = f * xr + 0.5 * W, f * yr + 0.5 * H
    out = {"feat": [ux, uy, cc / detd, -v01 / detd, ca / detd, op]}
    with torch.no_grad():
        Lp = L.clamp_min(0.0)
        out["valid"] = (tz > 0.2) & (L > 0) & (detd > 0)
        det = (v00 * v11 - v01 * v01).clamp_min(0.0)
        out["S"] = (8.0 * Lp * det / torch.maximum(v00, v11)).sqrt()
        ex, ey = (2.0 * Lp * ca).sqrt(), (2.0 * Lp * cc).sqrt()
        x0, x1 = ((ux - ex) / 16).floor(), ((ux + ex) / 16).floor()
        y0, y1 = ((uy - ey) / 16).floor(), ((uy + ey) / 16).floor()
        x0, y0 = x0.clamp_min(0), y0.clamp_min(0)
        x1, y1 = x1.clamp_max((W + 15) // 16 - 1), y1.clamp_max((H + 15) // 16 - 1)
        out["rect"] = [x0, y0, x1, y1]
        out["ntiles"] = (x1 - x0 + 1).clamp_min(0) * (y1 - y0 + 1).clamp_min(0)
        out["depth"] = tz.float()
    if color:
        d = mean - torch.from_numpy(cam["campos"]).to("cuda", dtype)
        out["feat"] += list(_sh_color(a["color"].to(dtype),
                                      d / d.norm(dim=1, keepdim=True)).unbind(1))
    return out


def _selected(S, a, mode):
    if mode == "all_levels":
        return torch.ones_like(S, dtype=torch.bool)
    small = (S / a["s_min"].double() >= 0.5) | (S >= 2.0)
    if mode == "filter_small":
        return small
    large = (a["level"] == 1) | (S / a["s_max"].double() <= 1.5)
    return large & ((a["level"] == a["n_levels"]) | small)


def _alphas(f, px, py):
    dx, dy = px[:, None] - f[:, 0], py[:, None] - f[:, 1]
    power = -0.5 * (f[:, 2] * dx * dx + f[:, 4] * dy * dy) - f[:, 3] * dx * dy
    al = (f[:, 5] * power.exp()).clamp_max(0.99)
    return torch.where((power <= 0) & (al >= 1.0 / 255.0), al, 0.0)


def _blend(f, px, py, T0):
    """Front-to-back blend of entries f (in list order) from transmittance T0
    at pixels (px, py): colour added and transmittance after it; a pixel that
    ended (T0 = 0) adds nothing."""
    al = _alphas(f, px, py)
    T = T0[:, None] * torch.cumprod(1.0 - al, 1)
    before = torch.cat([T0[:, None], T[:, :-1]], 1)
    on = T >= 1e-4
    return (torch.where(on, al * before, 0.0) @ f[:, 6:9]), T, on


def _exact_frame(a, cam, mode, target=None):
    """One frame in FP64: (image, final_t), and with a target also the mean
    L1 loss, accumulating its gradient into the leaves of `a`."""
    p = _splat(a, cam, torch.float64, color=True)
    keep = p["valid"] & _selected(p["S"], a, mode) & (p["ntiles"] > 0)
    idx = keep.nonzero()[:, 0]
    idx = idx[torch.sort(p["depth"][idx], stable=True)[1]]
    feat = torch.stack(p["feat"], 1)[idx]
    grad = None
    if target is not None:
        grad = torch.zeros_like(feat)
    ff = feat.detach()
    x0, y0, x1, y1 = (r[idx] for r in p["rect"])
    W, H = cam["width"], cam["height"]
    image = torch.zeros((3, H, W), dtype=torch.float64, device="cuda")
    final = torch.ones((H, W), dtype=torch.float64, device="cuda")
    loss = 0.0
    for ty in range((H + 15) // 16):
        row = ((y0 <= ty) & (y1 >= ty)).nonzero()[:, 0]
        rx0, rx1 = x0[row], x1[row]
        for tx in range((W + 15) // 16):
            e = row[(rx0 <= tx) & (rx1 >= tx)]
            ys, xs = range(ty * 16, min(H, ty * 16 + 16)), range(tx * 16, min(W, tx * 16 + 16))
            py, px = (v.reshape(-1) for v in torch.meshgrid(
                torch.tensor(ys, device="cuda") + 0.5, torch.tensor(xs, device="cuda") + 0.5,
                indexing="ij"))
            px, py = px.double(), py.double()
            live = torch.ones_like(px)      # transmittance, 0 once ended
            T_out = torch.ones_like(px)
            C = torch.zeros((px.numel(), 3), dtype=torch.float64, device="cuda")
            done = 0
            while done < e.numel():
                part = ff[e[done:done + 1024]]
                add, T, on = _blend(part, px, py, live)
                done += part.shape[0]
                C += add
                T_out = torch.where(on, T, math.inf).amin(1).minimum(T_out)
                live = torch.where(on[:, -1], T[:, -1], 0.0)
                if not bool((live > 0).any()):
                    break
            sl = (slice(ys[0], ys[-1] + 1), slice(xs[0], xs[-1] + 1))
            image[:, sl[0], sl[1]] = C.T.reshape(3, len(ys), len(xs))
            final[sl] = T_out.reshape(len(ys), len(xs))
            if target is not None and done > 0:
                leaf = ff[e[:done]].requires_grad_()
                col, _, _ = _blend(leaf, px, py, torch.ones_like(px))
                dl = torch.sign(C - target[:, sl[0], sl[1]].reshape(3, -1).T.double())
                grad.index_add_(0, e[:done],
                                torch.autograd.grad(col, leaf, dl / target.numel())[0])
    if target is not None:
        loss = (image - target.double()).abs().mean()
        feat.backward(grad)
    return image, final, loss


def exact(case, seed):
    kind, mode = case["kind"], case.get("mode", "selective")
    if kind == "aggregate":
        return None  # which Gaussians share a voxel is decided in FP32
    cams = _cameras(case, seed)
    a = _arrays(case, seed)
    if kind in ("frame", "sweep"):
        with torch.no_grad():
            r = [_exact_frame(a, c, mode)[:2] for c in cams]
        r = [{"image": i, "final_t": t, "n_contrib": None} for i, t in r]
        return r[0] if kind == "frame" else r
    if kind == "serve":
        b = _arrays(case, seed + 1)
        with torch.no_grad():
            # one frame of each resolution: all of them would take half a minute
            return [_exact_frame(b if k % 2 else a, c, mode)[0] if k < len(SWEEP) else None
                    for k, c in enumerate(cams)]
    keys = ("mean", "log_scale", "quat", "opacity", "color")
    targets = _targets([_as_camera(c) for c in cams], seed)
    for k in keys:
        a[k] = a[k].double().requires_grad_()
    images, loss = [], 0.0
    for c, t in zip(cams, targets):
        i, _, l = _exact_frame(a, c, mode, t)
        images.append(i)
        loss = loss + l
    return {"loss": loss, "images": images, "grads": {k: a[k].grad for k in keys}}
