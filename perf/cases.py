"""What a user of this framework has it do, as cases that can be timed and compared.

A case is a training iteration, a render or a fusion of one RGB-D frame, through the calls that a
program makes: ``Trainer`` and ``BatchedTrainer`` (eager, and replayed from the CUDA graph that
they capture), ``StreamingOptimizer.iterate``, the autograd ``render``, ``gs_render_fwd`` and
``TSDFGrid``.  The inputs are seeded: a procedural room with boxes and a noise texture seen by one
or several cameras (ray-cast on the GPU), and a Gaussian map seeded from those frames with the
contrast quadtree, then disturbed the way a few iterations leave it.

Fields of a case:
  kind     graph: a training iteration replayed from a captured graph; step: the same, eager;
           split: eager, forward, loss, backward and Adam as calls of their own; stream: an
           iteration of the streaming loop on a map with free slots; autograd: differentiable
           render and its backward pass with the pose; render: forward only; tsdf: fuse a depth
           image and look its surface points up
  views    "WxH@f" per view, separated by blanks (f: focal length in pixels)
  n, sh    Gaussians and SH degree (tsdf: earlier frames in the grid, unused)
  slots    stream: slots of the map (n of them live)
  large    share of the Gaussians replaced by large, nearly opaque ones
  cloud    random Gaussians in the first view's frustum instead of the quadtree's
  tile     "16x16", "8x32" or "32x8"
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2408_12677_gb300 import abi
from paper_2408_12677_gb300.streaming import Keyframe, StreamingOptimizer
from paper_2408_12677_gb300.torch_api import BatchedTrainer, Context, GaussianModel, Trainer, render
from paper_2408_12677_gb300.tsdf import TSDFGrid

W_COLOR, W_DEPTH = 0.8, 0.2
FIRST_STEP = 100  # the iterations of a case are not the first of their map
# Learning rates of a late iteration: a hundredth of the defaults, so that the map, and with it the
# work of a pass, stays what it is over the thousands of passes that a timing makes.
LR = dict(lr_means=1.6e-6, lr_log_scales=5e-5, lr_quats=1e-5, lr_opacity=5e-4, lr_sh_dc=2.5e-5, lr_sh_rest=1.25e-6)
NAMES = ("means", "log_scales", "quats", "opacity_logits", "sh")
Y00 = 0.28209479177387814
UNEVEN_8 = "640x480@320 640x480@320 " + "1200x680@600 " * 4 + "1752x1168@1200 1752x1168@1200"


def case(kind, views, n=0, sh=0, slots=0, large=0.0, cloud=False, tile="16x16", name=None):
    c = dict(kind=kind, views=views.strip(), n=n, sh=sh, slots=slots, large=large, cloud=cloud, tile=tile)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest iteration: a toy map fitted from a notebook or a test, where launches are all there is
        case("graph", "64x48@60", 500, 0, cloud=True, name="tiny_graph"),
        # the online optimisation on one frame, as a mapping loop replays it
        case("graph", "1200x680@600", 300_000, 3, name="online_graph"),
        # the same, eager, at a size whose borders no tile divides, on a middling map of SH degree 2
        case("step", "843x567@421", 100_003, 2, name="online_eager"),
        # eight keyframes of uneven size against one map, one Adam step
        case("graph", UNEVEN_8, 500_000, 3, name="keyframes_graph"),
        # the streaming loop: the frame and four past keyframes on a map that has grown to 600k of 2^20 slots
        case("stream", "1200x680@600 " * 5, 600_000, 3, slots=1 << 20, name="streaming"),
        # a user's own loss and tracker: gradients of the images w.r.t. the map and the pose
        case("autograd", "640x480@320", 60_001, 1, name="autograd_pose"),
        # showing the map: a novel view of a large map
        case("render", "1752x1168@1200", 1_000_000, 3, name="render_large"),
        # forward, loss, backward and Adam called one by one, colours without view dependence, tall tiles
        case("split", "641x479@320", 50_000, 0, tile="8x32", name="split_calls"),
        # the scale stress: a fifth of a million Gaussians large and overlapping, lists of many thousands
        case("step", "1752x1168@1200", 1_000_000, 3, large=0.2, name="scale_stress"),
        # the per-frame TSDF fusion and the look-up of the frame's surface points
        case("tsdf", "1200x680@600", name="tsdf_frame"),
    ]


def draw(rng):
    kind = rng.choices(("graph", "step", "split", "stream", "autograd", "render", "tsdf"), (5, 4, 2, 2, 3, 3, 1))[0]

    def size(most=1752):
        w = int(round(48 * (most / 48) ** rng.random()))
        return w, max(16, int(w * rng.uniform(0.5, 0.8)))

    many = kind in ("stream", "graph", "step", "render") and (kind == "stream" or rng.random() < 0.4)
    sizes = [size(1200) for _ in range(rng.randint(2, 8))] if many else [size()]
    if kind == "stream":  # one camera model
        sizes = [sizes[0]] * min(5, len(sizes))
    views = " ".join("%dx%d@%d" % (w, h, max(20, int(w * rng.uniform(0.45, 0.7)))) for w, h in sizes)
    if kind == "stream":
        views = " ".join([views.split()[0]] * len(sizes))
    if kind == "tsdf":
        return case(kind, views)
    pixels = max(w * h for w, h in sizes)
    n = int(min(1_000_000, max(300, pixels * 0.02 * 25 ** rng.random())))
    tile = rng.choice(("16x16", "16x16", "16x16", "8x32", "32x8"))
    large = round(0.2 * 0.01 ** rng.random(), 4) if kind in ("step", "render") and not many and rng.random() < 0.25 else 0.0
    slots = int(n * rng.uniform(1.0, 2.0)) if kind == "stream" else 0
    cloud = n <= 20_000 and rng.random() < 0.5  # larger clouds of such splats are fog
    return case(kind, views, n, rng.randint(0, 3), slots, 0.0 if cloud else large, cloud, tile)


# ----------------------------------------------------------------------------------------------
# the scene: a room [0, 8] x [0, 6] x [0, 3] m with boxes, ray-cast on the GPU
# ----------------------------------------------------------------------------------------------
class Cam:
    def __init__(self, w, h, f):
        self.width, self.height, self.fx, self.fy, self.cx, self.cy = w, h, float(f), float(f), w / 2.0, h / 2.0


def cameras(c):
    out = []
    for v in c["views"].split():
        size, f = v.split("@")
        w, h = size.split("x")
        out.append(Cam(int(w), int(h), int(f)))
    return out


def look(eye, yaw, pitch):
    """World-to-camera (R, t), float32, of a camera at `eye` (x right, y down, z forward)."""
    f = np.array([math.cos(pitch) * math.cos(yaw), math.cos(pitch) * math.sin(yaw), math.sin(pitch)])
    r = np.cross(f, [0.0, 0.0, 1.0])
    r /= np.linalg.norm(r)
    R = np.stack([r, np.cross(f, r), f]).astype(np.float32)
    return R, (-R.astype(np.float64) @ np.asarray(eye)).astype(np.float32)


def poses(rng, n, smooth):
    """`n` cameras near the room's centre: scattered keyframes, or consecutive frames of one sweep."""
    eye, yaw, pitch = rng.uniform([3.0, 2.4, 1.2], [4.6, 3.6, 1.7]), rng.uniform(-0.5, 0.5), rng.uniform(-0.25, 0.0)
    out = []
    for k in range(n):
        if smooth:
            e, y, p = eye + 0.12 * k * np.array([0.3, 1.0, 0.05]), yaw + 0.09 * k, pitch
        else:
            e = np.clip(eye + rng.uniform(-1.5, 1.5, 3), [2.2, 1.7, 0.5], [5.3, 4.3, 2.5])
            y, p = rng.uniform(-0.5, 0.5), rng.uniform(-0.4, 0.3)
        out.append(look(e, y, p))
    return out


def hash01(ix, iy, iz, salt):
    """Integer lattice points -> [0, 1): a multiplicative hash in int64."""
    h = ix * 73856093 ^ iy * 19349663 ^ iz * 83492791 ^ salt
    h = (h ^ (h >> 15)) * 0x2C1B3C6D & 0xFFFFFFFF
    h = (h ^ (h >> 12)) * 0x297A2D39 & 0xFFFFFFFF
    return ((h ^ (h >> 15)) & 0xFFFFFF).to(torch.float32) / float(1 << 24)


def noise(p, salt):
    """Trilinear value noise of points [M, 3] in [0, 1)."""
    fl = torch.floor(p)
    f = p - fl
    w = f * f * (3.0 - 2.0 * f)
    i = fl.to(torch.int64)
    out = torch.zeros(p.shape[0], device=p.device)
    for k in range(8):
        d = (k & 1, (k >> 1) & 1, k >> 2)
        wk = 1.0
        for a in range(3):
            wk = wk * (w[:, a] if d[a] else 1.0 - w[:, a])
        out += wk * hash01(i[:, 0] + d[0], i[:, 1] + d[1], i[:, 2] + d[2], salt)
    return out


def frame(room, cam, R, t):
    """rgb [3, H, W] in [0, 1] and camera depth [H, W] (0 outside 0.5 .. 6 m)."""
    dev = torch.device("cuda")
    H, W = cam.height, cam.width
    j, i = torch.meshgrid(torch.arange(H, device=dev), torch.arange(W, device=dev), indexing="ij")
    d = torch.stack([(i.reshape(-1) + 0.5 - cam.cx) / cam.fx, (j.reshape(-1) + 0.5 - cam.cy) / cam.fy,
                     torch.ones(H * W, device=dev)], 1).float()
    Rd = torch.tensor(R, device=dev)
    d = (d[:, None, :] * Rd.T[None]).sum(2)
    o = torch.tensor(-(R.astype(np.float64).T @ t.astype(np.float64)), dtype=torch.float32, device=dev)
    far = torch.tensor([8.0, 6.0, 3.0], device=dev)
    tw = torch.where(d > 0, (far - o) / d, torch.where(d < 0, -o / d, torch.full_like(d, 1e9)))
    best, ax = tw.min(1)
    obj = 2 * ax + (d.gather(1, ax[:, None])[:, 0] > 0)
    for b, (lo, hi) in enumerate(zip(room["lo"], room["hi"])):
        inv = 1.0 / d
        t1, t2 = (lo - o) * inv, (hi - o) * inv
        near, end = torch.minimum(t1, t2).amax(1), torch.maximum(t1, t2).amin(1)
        hit = (end >= near) & (near > 0.05) & (near < best)
        best, obj = torch.where(hit, near, best), torch.where(hit, 6 + b, obj)
    p = o + best[:, None] * d
    rgb = room["colors"][obj]
    for k in range(3):
        q = p * (45.0 * 2.0 ** k)
        rgb = rgb + 0.5 * 0.5 ** k * 2.0 * (torch.stack([noise(q, room["salt"] + 101 * k + 7 * ch) for ch in range(3)], 1) - 0.5)
    depth = torch.where((best >= 0.5) & (best <= 6.0), best, torch.zeros_like(best))
    return rgb.clamp(0.0, 1.0).T.reshape(3, H, W).contiguous(), depth.reshape(H, W).contiguous()


def make_room(rng):
    dev = torch.device("cuda")
    lo, hi = [], []
    while len(lo) < 16:  # axis-aligned boxes, none around the cameras
        half = rng.uniform(0.1, 0.6, 3)
        c = rng.uniform([0.6, 0.6, half[2]], [7.4, 5.4, 2.4])
        if not (1.4 < c[0] < 6.1 and 0.9 < c[1] < 5.1):
            lo.append(torch.tensor(c - half, dtype=torch.float32, device=dev))
            hi.append(torch.tensor(c + half, dtype=torch.float32, device=dev))
    return {"lo": lo, "hi": hi, "colors": torch.tensor(rng.uniform(0, 1, (22, 3)), dtype=torch.float32, device=dev),
            "salt": int(rng.integers(1, 1 << 30))}


def leaves(rgb):
    """Leaves (x0, y0, w, h) of the contrast quadtree (64 px cells, variance over 0.01 splits), in a fixed order."""
    H, W = rgb.shape[1:]
    Hp, Wp = -(-H // 64) * 64, -(-W // 64) * 64
    pad = torch.zeros((7, Hp, Wp), dtype=torch.float64, device=rgb.device)
    pad[:3, :H, :W], pad[3:6, :H, :W], pad[6, :H, :W] = rgb.double(), rgb.double() ** 2, 1.0
    alive = torch.ones((Hp // 64, Wp // 64), dtype=torch.bool, device=rgb.device)
    found = []
    for size in (64, 32, 16, 8, 4, 2, 1):
        s = pad.reshape(7, Hp // size, size, Wp // size, size).sum((2, 4))
        area = s[6].clamp(min=1.0)
        var = (s[3:6] / area - (s[:3] / area) ** 2).clamp(min=0.0).mean(0)
        alive = alive & (s[6] > 0)
        split = alive & (var > 0.01) & (s[6] > 1) if size > 1 else torch.zeros_like(alive)
        yx = torch.nonzero(alive & ~split) * size
        x0, y0 = yx[:, 1], yx[:, 0]
        found.append(torch.stack([x0, y0, (W - x0).clamp(max=size), (H - y0).clamp(max=size)], 1))
        alive = split.repeat_interleave(2, 0).repeat_interleave(2, 1)
    return torch.cat(found).double()


def seeded(views, n, gen):
    """(means, scales, colours) of exactly n Gaussians at the frames' quadtree leaves, spread evenly over the frames."""
    parts = []
    for cam, R, t, rgb, depth in views:
        q = leaves(rgb)
        u, v = q[:, 0] + q[:, 2] / 2, q[:, 1] + q[:, 3] / 2
        pi, pj = u.long().clamp(max=cam.width - 1), v.long().clamp(max=cam.height - 1)
        z = depth[pj, pi].double()
        ok = z > 0
        u, v, z, pi, pj, q = u[ok], v[ok], z[ok], pi[ok], pj[ok], q[ok]
        parts.append(torch.cat([torch.stack([(u - cam.cx) * z / cam.fx, (v - cam.cy) * z / cam.fy, z], 1),
                                (0.5 * torch.hypot(q[:, 2], q[:, 3]) * z / cam.fx)[:, None], rgb[:, pj, pi].T.double()], 1))
        Rd, td = torch.tensor(R, device=z.device).double(), torch.tensor(t, device=z.device).double()
        d = parts[-1][:, :3] - td
        parts[-1][:, :3] = d[:, :1] * Rd[0] + d[:, 1:2] * Rd[1] + d[:, 2:] * Rd[2]
    a = torch.cat(parts)
    if a.shape[0] == 0:
        a = torch.tensor([[6.0, 3.0, 1.5, 0.01, 0.5, 0.5, 0.5]], dtype=torch.float64, device="cuda")
    reps = -(-n // a.shape[0])
    pick = torch.cat([torch.randperm(a.shape[0], generator=gen, device="cuda") for _ in range(reps)])[:n].sort().values
    b = a[pick]
    if reps > 1:  # a Gaussian that is there more than once moves by up to half its size
        b[:, :3] += b[:, 3:4] * (torch.rand((n, 3), generator=gen, device="cuda").double() - 0.5)
    elif a.shape[0] > 1.2 * n:  # fewer Gaussians than leaves cover the frame: larger ones
        b[:, 3] *= math.sqrt(a.shape[0] / n)
    return b[:, :3], b[:, 3], b[:, 4:7]


def make_params(c, views, gen):
    """The map: five float32 arrays on the GPU."""
    n, K, dev = c["n"], (c["sh"] + 1) ** 2, "cuda"

    def normal(*s):
        return torch.randn(s, generator=gen, device=dev)

    if c["cloud"]:
        cam, R, t = views[0][:3]
        u = torch.rand((n, 6), generator=gen, device=dev).double()
        z = (0.5 ** 3 + u[:, 0] * (4.0 ** 3 - 0.5 ** 3)) ** (1 / 3)
        pc = torch.stack([(u[:, 1] * cam.width - cam.cx) * z / cam.fx, (u[:, 2] * cam.height - cam.cy) * z / cam.fy, z], 1)
        d = pc - torch.tensor(t, device=dev).double()
        Rd = torch.tensor(R, device=dev).double()
        means, rgb = d[:, :1] * Rd[0] + d[:, 1:2] * Rd[1] + d[:, 2:] * Rd[2], u[:, 3:]
        ls = -4.0 + 3.0 * torch.rand((n, 3), generator=gen, device=dev)
        quats, logits = normal(n, 4), normal(n)
    else:
        means, size, rgb = seeded(views, n, gen)
        ls = size.log().float()[:, None] + 0.2 * normal(n, 3)
        quats = torch.tensor([1.0, 0, 0, 0], device=dev) + 0.2 * normal(n, 4)
        logits = 0.3 + 0.8 * normal(n)
    m = int(round(c["large"] * n))
    if m:
        big = torch.randperm(n, generator=gen, device=dev)[:m]
        ls[big] = -torch.rand((m, 3), generator=gen, device=dev)
        quats[big] = normal(m, 4)
        logits[big] = 2.0
    sh = 0.03 * normal(n, K, 3)
    sh[:, 0] = ((rgb - 0.5) / Y00).float()
    return {"means": means.float(), "log_scales": ls, "quats": quats, "opacity_logits": logits, "sh": sh}


def moments(c, slots, pixels, gen):
    """Adam moments of a map in mid-optimisation, in the flat layout (of the size that gradients have here)."""
    K = (c["sh"] + 1) ** 2
    scale = torch.cat([torch.full((k * slots,), s / pixels, device="cuda")
                       for k, s in ((3, 300.0), (3, 1.0), (4, 1.0), (1, 1.0), (3 * K, 0.3))])
    m = 0.3 * scale * torch.randn(scale.shape[0], generator=gen, device="cuda")
    return m, scale * scale * (0.2 + torch.rand(scale.shape[0], generator=gen, device="cuda"))


def inputs(c, seed):
    """Views (camera, R, t, rgb, depth), the map and its moments, from the seed alone."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(int(rng.integers(1 << 40)))
    room = make_room(rng)
    cams = cameras(c)
    extra = 2 if c["kind"] == "tsdf" else 0  # the frames before
    at = poses(rng, len(cams) + extra, c["kind"] in ("stream", "tsdf"))
    cams = cams[:1] * extra + cams
    views = [(cam, R, t, *frame(room, cam, R, t)) for cam, (R, t) in zip(cams, at)]
    if c["kind"] == "tsdf":
        return views, None, None
    params = make_params(c, views, gen)
    if c["kind"] in ("render", "autograd"):
        return views, params, gen
    slots = max(c["slots"], c["n"])
    return views, params, moments(c, slots, sum(v[0].width * v[0].height for v in views), gen)


def host(params, sh):
    return {**{k: params[k].cpu().numpy() for k in NAMES}, "sh_degree": sh}


def raster(c):
    w, h = c["tile"].split("x")
    return abi.raster_cfg(tile_w=int(w), tile_h=int(h))


# ----------------------------------------------------------------------------------------------
# what a program has in hand before the call, and the call
# ----------------------------------------------------------------------------------------------
def prepare(c, seed):
    views, params, more = inputs(c, seed)
    kind, s = c["kind"], {"kind": c["kind"]}
    if kind == "tsdf":
        s["ctx"] = Context(0)
        s["grid"] = TSDFGrid(s["ctx"], capacity=1 << 16)
        for cam, R, t, _, depth in views[:-1]:
            s["grid"].integrate(depth, abi.make_camera(cam.fx, cam.fy, cam.cx, cam.cy, cam.width, cam.height),
                                abi.make_viewmat(R, t))
        cam, R, t, _, depth = views[-1]
        s["cam"] = abi.make_camera(cam.fx, cam.fy, cam.cx, cam.cy, cam.width, cam.height)
        s["view"], s["depth"] = abi.make_viewmat(R, t), depth
        j, i = torch.nonzero(depth > 0, as_tuple=True)
        z = depth[j, i]
        d = torch.stack([(i + 0.5 - cam.cx) * z / cam.fx, (j + 0.5 - cam.cy) * z / cam.fy, z], 1) - torch.tensor(t, device="cuda")
        Rd = torch.tensor(R, device="cuda")
        s["points"] = (d[:, :1] * Rd[0] + d[:, 1:2] * Rd[1] + d[:, 2:] * Rd[2]).float().contiguous()
        return s
    if kind == "render":
        s["ctx"], s["params"], s["rcfg"] = Context(0), params, raster(c)
        s["g"] = abi.make_gaussians(*[params[k] for k in NAMES], c["sh"])
        s["cams"] = [abi.make_camera(v[0].fx, v[0].fy, v[0].cx, v[0].cy, v[0].width, v[0].height) for v in views]
        s["views"] = [abi.make_viewmat(v[1], v[2]) for v in views]
        for k, ch in (("color", (3,)), ("depth", ()), ("alpha", ())):
            s[k] = [torch.empty(ch + (v[0].height, v[0].width), device="cuda") for v in views]
        return s
    if kind == "autograd":
        cam, R, t = views[0][:3]
        s.update(ctx=Context(0), params={k: params[k].requires_grad_() for k in NAMES}, sh=c["sh"], cam=cam, R=R, t=t,
                 rcfg=raster(c), xi=torch.zeros(6, device="cuda", requires_grad=True), up=upstream(cam, more))
        return s
    m, v = more
    acfg = abi.adam_cfg(zero_grads=1, **LR)
    if kind == "stream":
        opt = StreamingOptimizer(views[0][0], c["sh"], n_past=4, capacity=c["slots"], raster_cfg=raster(c), adam_cfg=acfg)
        opt.map.append(host(params, c["sh"]))
        opt.map.model.m.copy_(m)
        opt.map.model.v.copy_(v)
        opt.step = FIRST_STEP
        s["opt"], s["views"] = opt, [Keyframe(cam, abi.make_viewmat(R, t), rgb, depth) for cam, R, t, rgb, depth in views]
        return s
    model = GaussianModel(host(params, c["sh"]))
    model.m.copy_(m)
    model.v.copy_(v)
    if len(views) == 1:
        cam, R, t, rgb, depth = views[0]
        tr = Trainer(model, cam, R, t, raster_cfg=raster(c), adam_cfg=acfg, fused=kind != "split")
    else:
        tr = BatchedTrainer(model, [v[:3] for v in views], raster_cfg=raster(c), adam_cfg=acfg)
        rgb, depth = [v[3] for v in views], [v[4] for v in views]
    tr.step_count = FIRST_STEP
    if kind == "graph":
        tr.capture(rgb, depth)  # runs one iteration
    s["tr"], s["rgb"], s["depth"] = tr, rgb, depth
    return s


def upstream(cam, gen):
    """Image gradients of a user's loss on a colour, depth and alpha image."""
    g = [torch.randn(sh, generator=gen, device="cuda") / (cam.width * cam.height)
         for sh in ((3, cam.height, cam.width), (cam.height, cam.width), (cam.height, cam.width))]
    return g


def run(s):
    kind = s["kind"]
    if kind == "tsdf":
        counts = s["grid"].integrate(s["depth"], s["cam"], s["view"])
        tsdf, weight = s["grid"].query(s["points"])
        return {"tsdf": tsdf, "weight": weight, **{k: counts[k] for k in ("blocks", "touched", "updated")}}
    if kind == "render":
        h = s["ctx"].handle
        if len(s["cams"]) == 1:
            abi.gs_render_fwd(h, s["g"], s["cams"][0], s["views"][0], s["rcfg"], s["color"][0], s["depth"][0], s["alpha"][0])
        else:
            abi.gs_render_fwd_batched(h, s["g"], s["cams"], s["views"], s["rcfg"], s["color"], s["depth"], s["alpha"])
        return {k: s[k] for k in ("color", "depth", "alpha")}
    if kind == "autograd":
        out = render(s["ctx"], s["params"], s["sh"], s["cam"], s["R"], s["t"], raster_cfg=s["rcfg"], pose_xi=s["xi"])
        wrt = [s["params"][k] for k in NAMES] + [s["xi"]]
        grads = torch.autograd.grad(out, wrt, s["up"])
        return {"images": list(out), "grads": list(grads)}
    if kind == "stream":
        s["opt"].iterate(s["views"])
        model, loss = s["opt"].map.model, s["opt"].loss
    else:
        tr = s["tr"]
        loss = tr.replay() if kind == "graph" else tr.step(s["rgb"], s["depth"])
        model = tr.model
    return {"loss": loss, "params": model.flat, "m": model.m, "v": model.v}


def work(c):
    """Inputs read once, outputs written once; a pixel of these maps blends about 20 Gaussians before it is
    opaque, at 27 operations forward and 68 backward, and a Gaussian's projection takes about 300 each way."""
    px = sum(cam.width * cam.height for cam in cameras(c))
    if c["kind"] == "tsdf":  # about 6.5 voxels in the band per pixel, (tsdf, weight) read and written
        return {"bytes": px * (4 + 6.5 * 16 + 20), "flops": px * 6.5 * 40}
    V, n = len(c["views"].split()), max(c["n"], c["slots"])
    floats = n * (11 + 3 * (c["sh"] + 1) ** 2)
    if c["kind"] == "render":
        return {"bytes": 4 * floats + 20 * px, "flops": 27 * 20 * px + 300 * V * n}
    if c["kind"] == "autograd":
        return {"bytes": 2 * 4 * floats + 40 * px, "flops": 95 * 20 * px + 600 * V * n}
    return {"bytes": 6 * 4 * floats + 16 * px, "flops": 95 * 20 * px + 600 * V * n + 15 * floats}


# ----------------------------------------------------------------------------------------------
# the same in 64 bits
# ----------------------------------------------------------------------------------------------
def sh_values(d, deg):
    """Real spherical harmonics (Condon-Shortley phase) up to degree `deg` at unit vectors d [N, 3]."""
    x, y, z = d.unbind(1)
    s = math.sqrt
    out = [torch.full_like(x, s(1 / (4 * math.pi)))]
    if deg > 0:
        a = s(3 / (4 * math.pi))
        out += [-a * y, a * z, -a * x]
    if deg > 1:
        a = s(15 / (4 * math.pi))
        out += [a * x * y, -a * y * z, s(5 / (16 * math.pi)) * (3 * z * z - 1), -a * x * z, a / 2 * (x * x - y * y)]
    if deg > 2:
        a, b, e = s(35 / (32 * math.pi)), s(105 / (4 * math.pi)), s(21 / (32 * math.pi))
        out += [-a * y * (3 * x * x - y * y), b * x * y * z, -e * y * (5 * z * z - 1), s(7 / (16 * math.pi)) * z * (5 * z * z - 3),
                -e * x * (5 * z * z - 1), b / 2 * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(out, 1)


def project64(P, deg, cam, R, t):
    """Per Gaussian, columns (mu 2, inverse covariance 3, opacity, colour 3, z), the 2D variances and which to draw."""
    q = P["quats"] / P["quats"].norm(dim=1, keepdim=True)
    w, x, y, z = q.unbind(1)
    Q = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y), 2 * (x * y + w * z),
                     1 - 2 * (x * x + z * z), 2 * (y * z - w * x), 2 * (x * z - w * y), 2 * (y * z + w * x),
                     1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)
    pc = P["means"] @ R.T + t
    X, Y, Z = pc.unbind(1)
    seen = Z > 0.2
    Z = torch.where(seen, Z, torch.ones_like(Z))
    lx, ly = 1.3 * cam.width / (2 * cam.fx), 1.3 * cam.height / (2 * cam.fy)
    xt, yt, o = Z * (X / Z).clamp(-lx, lx), Z * (Y / Z).clamp(-ly, ly), torch.zeros_like(Z)
    J = torch.stack([cam.fx / Z, o, -cam.fx * xt / Z ** 2, o, cam.fy / Z, -cam.fy * yt / Z ** 2], 1).reshape(-1, 2, 3)
    M = J @ (R @ (Q * P["log_scales"].exp()[:, None, :]))
    cov = M @ M.transpose(1, 2)
    a, b, d = cov[:, 0, 0] + 0.3, cov[:, 0, 1], cov[:, 1, 1] + 0.3
    det = a * d - b * b
    dirs = P["means"] + R.T @ t
    rgb = (0.5 + (sh_values(dirs / dirs.norm(dim=1, keepdim=True), deg)[:, :, None] * P["sh"]).sum(1)).clamp(min=0.0)
    cols = torch.cat([torch.stack([cam.fx * X / Z + cam.cx, cam.fy * Y / Z + cam.cy, d / det, -b / det, a / det,
                                   P["opacity_logits"].sigmoid()], 1), rgb, Z[:, None]], 1)
    return cols, a.detach(), d.detach(), seen & (det > 0)


def composite64(P, deg, cam, R, t, score):
    """Renders 16 x 16 tiles in chunks; score(pixels, colour, depth, alpha) gives a chunk's scalar loss, whose
    gradient goes back to the leaves of P.  Returns the summed loss and the images, or None for very long lists."""
    with torch.enable_grad():
        cols, va, vd, ok = project64(P, deg, cam, R, t)
    leaf = cols.detach()
    TX, TY, dev = -(-cam.width // 16), -(-cam.height // 16), leaf.device
    rx, ry = 3 * va.sqrt() + 1e-6, 3 * vd.sqrt() + 1e-6

    def span(mid, r, most):
        return [(e / 16).floor().clamp(-1, most).long() for e in (mid - r, mid + r)]

    (x0, x1), (y0, y1) = span(leaf[:, 0], rx, TX), span(leaf[:, 1], ry, TY)
    x0, y0 = x0.clamp(min=0), y0.clamp(min=0)
    nx, ny = (x1.clamp(max=TX - 1) - x0 + 1).clamp(min=0), (y1.clamp(max=TY - 1) - y0 + 1).clamp(min=0)
    count = torch.where(ok, nx * ny, torch.zeros_like(nx))
    if int(count.sum()) > 40_000_000:
        return None
    by_depth = torch.sort(leaf[:, 9].float(), stable=True).indices
    ids = by_depth.repeat_interleave(count[by_depth])
    first = count[by_depth].cumsum(0) - count[by_depth]
    k = torch.arange(ids.numel(), device=dev) - first.repeat_interleave(count[by_depth])
    tiles = (y0[ids] + k // nx[ids].clamp(min=1)) * TX + x0[ids] + k % nx[ids].clamp(min=1)
    order = torch.sort(tiles, stable=True).indices
    ids, length = ids[order], torch.bincount(tiles, minlength=TX * TY)
    start = length.cumsum(0) - length
    tile_order = torch.sort(length, descending=True, stable=True).indices
    lens, todo, at = length[tile_order].tolist(), tile_order, 0
    images = torch.zeros((cam.height * cam.width, 5), dtype=torch.float64, device=dev)
    total, grad = torch.zeros((), dtype=torch.float64, device=dev), torch.zeros_like(leaf)
    gp = torch.arange(256, device=dev)
    while at < len(lens):
        L = max(lens[at], 1)
        G = max(1, min(len(lens) - at, (1 << 23) // (256 * L)))
        tl = todo[at:at + G]
        at += G
        j = torch.arange(L, device=dev)
        have = j[None] < length[tl][:, None]
        g = ids[(start[tl][:, None] + j[None]).clamp(max=max(ids.numel() - 1, 0))] if ids.numel() else j[None].expand(G, L) * 0
        px, py = (tl % TX * 16)[:, None] + gp % 16, (tl // TX * 16)[:, None] + gp // 16
        inside = (px < cam.width) & (py < cam.height)
        with torch.enable_grad():
            e = leaf[g].requires_grad_()
            dx = px[:, :, None] + 0.5 - e[:, None, :, 0]
            dy = py[:, :, None] + 0.5 - e[:, None, :, 1]
            qq = e[:, None, :, 2] * dx * dx + 2 * e[:, None, :, 3] * dx * dy + e[:, None, :, 4] * dy * dy
            alpha = (e[:, None, :, 5] * torch.exp(-0.5 * qq)).clamp(max=0.99)
            act = have[:, None] & (qq <= 9.0) & (alpha >= 1.0 / 255.0)
            alpha = torch.where(act, alpha, torch.zeros_like(alpha))
            T = torch.cumprod(1 - alpha, 2)
            add = act & (T >= 1e-4)
            wgt = torch.where(add, alpha * torch.cat([torch.ones_like(T[:, :, :1]), T[:, :, :-1]], 2), torch.zeros_like(T))
            cd = torch.cat([wgt @ e[:, :, 6:10], wgt.sum(2, keepdim=True)], 2)
            at_px = (py * cam.width + px)[inside]
            cd = cd[inside]
            loss = score(at_px, cd[:, :3], cd[:, 3], cd[:, 4]) if score else None
        images[at_px] = cd.detach()
        if score:
            total += loss.detach()
            ge, = torch.autograd.grad(loss, e)
            grad.index_add_(0, g[have], ge[have])
    if score:
        cols.backward(grad)
    return total, images.T.reshape(5, cam.height, cam.width)


def exact(c, seed):
    """What run() returns, in float64 without tiles of this framework's kind, its lists or its kernels.  None for the
    fusion, whose block, pixel and update decisions are float32 by definition, and for lists too long for it."""
    if c["kind"] == "tsdf" or c["large"] > 0.002:
        return None
    views, params, more = inputs(c, seed)
    P = {k: params[k].double().requires_grad_() for k in NAMES}

    def pose(v):
        return torch.tensor(v[1], device="cuda").double(), torch.tensor(v[2], device="cuda").double()

    if c["kind"] == "render":
        got = [composite64(P, c["sh"], v[0], *pose(v), None) for v in views]
        if any(g is None for g in got):
            return None
        return {"color": [g[1][:3] for g in got], "depth": [g[1][3] for g in got], "alpha": [g[1][4] for g in got]}
    if c["kind"] == "autograd":
        cam = views[0][0]
        up = [u.double() for u in upstream(cam, more)]
        xi = torch.zeros(6, dtype=torch.float64, device="cuda", requires_grad=True)
        R, t = pose(views[0])
        with torch.enable_grad():
            o = torch.zeros((), dtype=torch.float64, device="cuda")
            a, b, d = xi[3], xi[4], xi[5]
            S = torch.stack([o, -d, b, d, o, -a, -b, a, o]).reshape(3, 3)  # exp to first order: xi is 0
            Rx, tx = R + S @ R, t + S @ t + xi[:3]
        uc, ud, ua = up[0].reshape(3, -1).T, up[1].reshape(-1), up[2].reshape(-1)
        got = composite64(P, c["sh"], cam, Rx, tx, lambda p, C, D, A: (C * uc[p]).sum() + (D * ud[p]).sum() + (A * ua[p]).sum())
        if got is None:
            return None
        im = got[1]
        return {"images": [im[:3], im[3], im[4]], "grads": [P[k].grad for k in NAMES] + [xi.grad]}
    m, v = (x.double() for x in more)
    slots, n, K = max(c["slots"], c["n"]), c["n"], (c["sh"] + 1) ** 2
    per = (3, 3, 4, 1, 3 * K)
    flat = torch.zeros(slots * sum(per), dtype=torch.float64, device="cuda")
    g = torch.zeros_like(flat)
    lr = torch.zeros_like(flat)
    at, off = [], 0
    for k, (name, p) in enumerate(zip(NAMES, per)):
        at.append((name, off, off + n * p))
        block = flat[off:off + slots * p].view(slots, p)
        block[:] = {"log_scales": -30.0, "opacity_logits": -30.0}.get(name, 0.0)  # the free slots of a growing map
        if name == "quats":
            block[:, 0] = 1.0
        block[:n] = params[name].reshape(n, p).double()
        lr[off:off + slots * p].view(slots, p)[:] = LR[("lr_means", "lr_log_scales", "lr_quats", "lr_opacity", "lr_sh_rest")[k]]
        if name == "sh":
            lr[off:off + slots * p].view(slots, p)[:, :3] = LR["lr_sh_dc"]
        off += slots * p
    for it in range(2 if c["kind"] == "graph" else 1):
        for name, a, b in at:
            P[name] = flat[a:b].view(params[name].shape).clone().requires_grad_()
        loss = 0.0
        for view in views:
            cam, rgb, dep = view[0], view[3].double().reshape(3, -1).T, view[4].double().reshape(-1)
            npx, nv = cam.width * cam.height, max(int((dep > 0).sum()), 1)
            got = composite64(P, c["sh"], cam, *pose(view), lambda p, C, D, A: W_COLOR * (C - rgb[p]).abs().sum() / (3 * npx)
                              + W_DEPTH * ((D - dep[p]).abs() * (dep[p] > 0)).sum() / nv)
            if got is None:
                return None
            loss = loss + got[0]
        for name, a, b in at:
            g[a:b] = P[name].grad.reshape(-1)
        step = FIRST_STEP + it + 1
        b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
        m, v = b1 * m + (1 - b1) * g, b2 * v + (1 - b2) * g * g
        flat = flat - lr * (m / (1 - b1 ** step)) / ((v / (1 - b2 ** step)).sqrt() + 1e-15)
    return {"loss": loss.reshape(1), "params": flat, "m": m, "v": v}
