"""Workloads of the rasterizer and of the SLAM steps around it, through the public entry points.

Each case stands for one thing that a mapping or tracking program does with this library:

  preview   a view rendered without gradients (`render.render` under no_grad)
  train     a window rendered and differentiated by autograd (`render.render`)
  map       a mapping step on kept buffers: forward, backward with the regulariser and a depth
            term, anchor update, prune mask (`Renderer.forward_raw` / `backward_raw`,
            `mapping.MapRegularizer`)
  window    forward + backward of a keyframe window on kept buffers, every gradient
  track     one captured tracking iteration from a frame's initial poses (`track.Tracker`)
  seed      triangulation and seed initialisation of matched pixels (`seeding`)
  upkeep    maintenance between steps: anchor update, prune mask, co-visibility of frame pairs

Scenes stand in for indoor sequences: Gaussians on the walls of a 6 x 5 x 3 m room and on spheres
in it, cameras inside. Every input is drawn on the GPU from the seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2601_00705_gb300 import binding, seeding
from paper_2601_00705_gb300.mapping import MapRegularizer
from paper_2601_00705_gb300.render import Renderer, render
from paper_2601_00705_gb300.track import Tracker

ROOM = (6.0, 5.0, 3.0)
RESOLUTIONS = ((320, 240), (640, 480), (1200, 680), (1920, 1080))
# Focal length over image width: a TUM RGB-D camera and the wide Replica / 1080p ones.
FOCAL = {320: 0.808, 640: 0.808}
PARAMS = ("means", "log_scales", "quats", "opacity_logits", "sh")


def listed():
    return [
        # The smallest call: a thumbnail of a few thousand Gaussians, latency and launches only.
        dict(name="preview_small", kind="preview", scene="slab", views=1, width=160, height=120,
             n=2000, degree=0, bwd_ppt=0),
        # One Replica-sized frame of a finished map, rendered for display or evaluation.
        dict(name="preview_frame", kind="preview", scene="room", views=1, width=1200, height=680,
             n=300000, degree=0, bwd_ppt=0),
        # A first, small differentiable fit (tests and notebooks): autograd on one little view.
        dict(name="train_small", kind="train", scene="slab", views=1, width=160, height=120,
             n=2000, degree=0, bwd_ppt=0),
        # A mapping window of ten TUM-sized keyframes trained through autograd.
        dict(name="train_window", kind="train", scene="room", views=10, width=640, height=480,
             n=150000, degree=3, bwd_ppt=0),
        # A mapping step on three cropped views of odd size, regulariser and depth term included.
        dict(name="map_ragged", kind="map", scene="room", views=3, width=601, height=347,
             n=50021, degree=2, bwd_ppt=0),
        # A mapping window of ten TUM-sized keyframes on kept buffers, blend settings as tuned.
        dict(name="window_tum", kind="window", scene="room", views=10, width=640, height=480,
             n=150000, degree=3, bwd_ppt=8),
        # Keyframes of mixed resolution over a cluttered room of a million Gaussians.
        dict(name="window_mixed", kind="window", scene="clutter", views=24, width=0, height=0,
             n=1000000, degree=3, bwd_ppt=8),
        # The largest window: sixteen 1080p views of three million Gaussians of widely spread size.
        dict(name="window_large", kind="window", scene="spread", views=16, width=1920, height=1080,
             n=3000000, degree=3, bwd_ppt=8),
        # Tracking a Replica-sized frame against a map with plain colours.
        dict(name="track_frame", kind="track", scene="room", views=1, width=1200, height=680,
             n=300000, degree=0, bwd_ppt=8),
        # Refining the poses of ten TUM-sized keyframes together.
        dict(name="track_window", kind="track", scene="room", views=10, width=640, height=480,
             n=150000, degree=3, bwd_ppt=8),
        # Dense initialisation from the matches of a keyframe window.
        dict(name="seed_window", kind="seed", views=10, width=640, height=480, m=131072, k=4,
             degree=3, voxel=0.0),
        # Maintenance of a million Gaussians and the keyframe test on nine frame pairs.
        dict(name="upkeep", kind="upkeep", n=1000000, pairs=9, width=640, height=480),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("preview", "train", "map", "window", "track", "seed", "upkeep"))
    if kind == "seed":
        return dict(kind=kind, views=rng.randint(3, 10), width=640, height=480,
                    m=_log_int(rng, 777, 131072), k=rng.randint(1, 5), degree=rng.randint(0, 3),
                    voxel=rng.choice((0.0, 0.0, 0.04)))
    if kind == "upkeep":
        width = _log_int(rng, 160, 1200)
        return dict(kind=kind, n=_log_int(rng, 10007, 3000000), pairs=rng.randint(1, 12),
                    width=width, height=int(width * 0.6))
    n = _log_int(rng, 2000, 1000000)
    width = _log_int(rng, 160, 1920 if n < 500000 else 900)
    height = int(width * rng.uniform(0.5, 0.8))
    views = 1 if kind == "preview" else rng.randint(1, 12 if width < 1000 else 4)
    scene = "slab" if n < 20000 else rng.choice(("room", "room", "clutter"))
    return dict(kind=kind, scene=scene, views=views, width=width, height=height, n=n,
                degree=rng.randint(0, 3), bwd_ppt=rng.choice((0, 8)))


# ------------------------------------------------------------------------------------------
# Inputs
# ------------------------------------------------------------------------------------------
def _generator(seed, salt):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + salt)


def _uniform(g, *shape):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _normal(g, *shape):
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)


def _camera(width, height, R, t, fx=None, fy=None):
    fx = FOCAL.get(width, 0.5) * width if fx is None else fx
    fy = fx * 0.998 if fy is None else fy
    return dict(width=width, height=height, fx=fx, fy=fy, cx=(width - 1) / 2, cy=(height - 1) / 2,
                R=np.asarray(R, np.float32), t=np.asarray(t, np.float32))


def _look(p, yaw, pitch):
    fwd = np.array([math.cos(pitch) * math.cos(yaw), math.cos(pitch) * math.sin(yaw),
                    math.sin(pitch)])
    right = np.cross(fwd, [0.0, 0.0, 1.0])
    right /= np.linalg.norm(right)
    R = np.stack([right, np.cross(fwd, right), fwd])
    return R, -R @ p


def _cameras(case, rng):
    """(cameras, their positions): a walk through the room, a ring looking outward, or poses all
    over the room with mixed resolutions."""
    size = np.array(ROOM)
    V, W, H = case["views"], case["width"], case["height"]
    scene = case.get("scene", "room")
    if scene == "slab":
        ang = 0.05 * rng.standard_normal((V, 2))
        cams = []
        for a, b in ang:
            ry = np.array([[math.cos(a), 0, math.sin(a)], [0, 1, 0], [-math.sin(a), 0, math.cos(a)]])
            rx = np.array([[1, 0, 0], [0, math.cos(b), -math.sin(b)], [0, math.sin(b), math.cos(b)]])
            cams.append(_camera(W, H, rx @ ry, 0.05 * rng.standard_normal(3), 0.94 * W, 0.94 * W))
        return cams, np.zeros((1, 3)) - 5.0
    cams, where = [], []
    if scene == "spread":
        for k in range(V):
            th = 2.0 * math.pi * k / V
            p = size / 2 + 1.5 * np.array([math.cos(th), math.sin(th), 0.0])
            where.append(p)
            cams.append(_camera(W, H, *_look(p, th, 0.0)))
        return cams, np.array(where)
    p, yaw = rng.uniform(1.0, size - 1.0), rng.uniform(0, 2 * math.pi)
    pitch = math.radians(rng.normal(0.0, 10.0))
    for k in range(V):
        if scene == "clutter":
            p, yaw = rng.uniform(1.0, size - 1.0), rng.uniform(0, 2 * math.pi)
            pitch = math.radians(rng.normal(0.0, 10.0))
        w, h = (W, H) if W else RESOLUTIONS[(k + k // 4) % 4]
        where.append(p)
        cams.append(_camera(w, h, *_look(p, yaw, pitch)))
        yaw += math.radians(rng.normal(0.0, 3.0))
        pitch = float(np.clip(pitch + math.radians(rng.normal(0.0, 3.0)), -0.5, 0.5))
        q = p + 0.1 * np.array([math.cos(yaw), math.sin(yaw), 0.0])
        if np.all(q > 0.5) and np.all(q < size - 0.5):
            p = q
        else:
            yaw += math.pi
    return cams, np.array(where)


def _spheres(rng, count, rmin, rmax, clear):
    out = []
    while len(out) < count:
        r = rng.uniform(rmin, rmax)
        c = rng.uniform(r + 0.3, np.array(ROOM) - r - 0.3)
        if np.linalg.norm(clear - c, axis=1).min() > r + 0.35:
            out.append((*c, r))
    return np.array(out)


def _surface(g, n, spheres, jitter):
    """n points on the walls and spheres, uniform by area, and that area."""
    size = torch.tensor(ROOM, device="cuda", dtype=torch.float64)
    sph = torch.as_tensor(spheres, device="cuda")
    X, Y, Z = ROOM
    walls = torch.tensor([Y * Z, X * Z, X * Y], device="cuda", dtype=torch.float64)
    areas = torch.cat([walls, walls, 4 * math.pi * sph[:, 3] ** 2])
    # The cumulated areas pick each point's surface (multinomial is limited in categories).
    pick = torch.searchsorted(areas.cumsum(0) / areas.sum(), _uniform(g, n)).clamp(max=len(areas) - 1)
    pts = _uniform(g, n, 3) * size
    axis = pick % 3
    wall = pick < 6
    rows = torch.arange(n, device="cuda")
    side = torch.where(pick < 3, torch.zeros_like(size[axis]), size[axis])
    pts[rows[wall], axis[wall]] = side[wall] + jitter * _normal(g, n)[wall]
    d = _normal(g, n, 3)
    d /= d.norm(dim=1, keepdim=True)
    s = sph[(pick - 6).clamp(min=0)]
    on = s[:, :3] + (s[:, 3:] + jitter * _normal(g, n, 1)) * d
    return torch.where(wall[:, None], pts, on), float(areas.sum())


def _scene(case, seed):
    """(parameters, cameras): float32 tensors on the GPU and camera dicts."""
    rng = np.random.default_rng(seed)
    g = _generator(seed, 1)
    n, K = case["n"], (case["degree"] + 1) ** 2
    cams, where = _cameras(case, rng)
    if case["scene"] == "slab":
        means = _uniform(g, n, 3) * torch.tensor([2.0, 2.0, 3.0], device="cuda") + torch.tensor(
            [-1.0, -1.0, 2.0], device="cuda")
        scales = -3.5 + 0.5 * _normal(g, n, 3) - math.log(max(n, 2000) / 2000) / 3
        logits = _normal(g, n)
    else:
        many = case["scene"] != "room"
        spheres = _spheres(rng, 200 if many else 20, *((0.05, 0.3) if many else (0.2, 0.6)), where)
        means, area = _surface(g, n, spheres, 0.01)
        if case["scene"] == "spread":
            scales = -4.0 + 0.7 * _normal(g, n, 3)
        else:
            scales = math.log(math.sqrt(area / n)) + 0.1 * _normal(g, n, 3)
        # Freshly seeded maps hold one opacity; optimised ones spread, some beyond the clamp.
        logits = (torch.full((n,), math.log(9.0), device="cuda") if many else
                  1.5 + 1.3 * _normal(g, n))
    quats = _normal(g, n, 4)
    sh = 0.1 * torch.randn((n, K, 3), generator=g, device="cuda")
    sh[:, 0] = (torch.rand((n, 3), generator=g, device="cuda") - 0.5) * math.sqrt(4 * math.pi)
    params = (means, scales, quats, logits, sh)
    return {k: v.float().contiguous() for k, v in zip(PARAMS, params)}, cams


def _pixels(cams):
    return sum(c["width"] * c["height"] for c in cams)


def _upstream(seed, P, depth):
    """The gradient of a mean L1 loss on colour (and a tenth of it on depth)."""
    g = _generator(seed, 2)
    sign = lambda *s: torch.randint(0, 2, s, generator=g, device="cuda").float() * 2 - 1  # noqa: E731
    return sign(P, 3) / P, (sign(P) * (0.1 / P) if depth else None)


def _frames(seed, cams):
    """Smooth colour frames, one pattern per view."""
    g = _generator(seed, 3)
    out = []
    for c in cams:
        y = torch.arange(c["height"], device="cuda")[:, None, None]
        x = torch.arange(c["width"], device="cuda")[None, :, None]
        f = 0.01 + 0.04 * torch.rand((2, 3), generator=g, device="cuda")
        ph = 6.28 * torch.rand(3, generator=g, device="cuda")
        out.append((0.5 + 0.4 * torch.sin(f[0] * x + f[1] * y + ph)).reshape(-1, 3))
    return torch.cat(out)


def _matches(case, seed):
    """Matched pixels of surface points: a reference view each and up to k other views, with
    0.3 px noise, 5 % outliers and confidences; frames and exposures."""
    rng = np.random.default_rng(seed)
    g = _generator(seed, 4)
    cams, where = _cameras(case, rng)
    spheres = _spheres(rng, 20, 0.2, 0.6, where)
    V, k, m, W, H = case["views"], case["k"], case["m"], case["width"], case["height"]
    R = torch.tensor(np.stack([c["R"] for c in cams]), device="cuda").double()
    t = torch.tensor(np.stack([c["t"] for c in cams]), device="cuda").double()
    f = torch.tensor([[c["fx"], c["fy"]] for c in cams], device="cuda", dtype=torch.float64)
    cc = torch.tensor([[c["cx"], c["cy"]] for c in cams], device="cuda", dtype=torch.float64)
    edge = torch.tensor([W - 2.0, H - 2.0], device="cuda")
    # The other views of each view, nearest in time first.
    near = torch.tensor([sorted((u for u in range(V) if u != v), key=lambda u: (abs(u - v), u))
                         for v in range(V)], device="cuda")[:, :k]
    found, have = [], 0
    while have < m:
        N = 6 * (m - have) + 4096
        X = _surface(g, N, spheres, 0.0)[0]
        cam = torch.einsum("vij,nj->nvi", R, X) + t
        uv = f * cam[..., :2] / cam[..., 2:].clamp(min=0.05) + cc
        ok = (cam[..., 2] > 0.05) & (uv >= 1).all(-1) & (uv <= edge).all(-1)
        ref = torch.randint(0, V, (N,), generator=g, device="cuda")
        row = torch.arange(N, device="cuda")
        nb = near[ref]
        seen = ok[row[:, None], nb]
        keep = (ok[row, ref] & seen.any(1)).nonzero()[:m - have, 0]
        xy = uv[row[:, None], nb] + 0.3 * _normal(g, N, nb.shape[1], 2)
        bad = _uniform(g, N, nb.shape[1]) < 0.05
        xy = torch.where(bad[..., None], 1 + _uniform(g, N, nb.shape[1], 2) * (edge - 1), xy)
        conf = torch.where(bad, 0.4 * _uniform(g, N, nb.shape[1]),
                           0.6 + 0.4 * _uniform(g, N, nb.shape[1]))
        nb = torch.where(seen, nb, -1)
        fill = k - nb.shape[1]  # fewer other views than slots
        nb = torch.nn.functional.pad(nb, (0, fill), value=-1)
        xy = torch.nn.functional.pad(xy, (0, 0, 0, fill))
        conf = torch.nn.functional.pad(conf, (0, fill))
        xr = uv[row, ref] + 0.3 * _normal(g, N, 2)
        found.append([a[keep] for a in (ref.int(), xr, nb.int(), xy, conf.float())])
        have += len(keep)
    ref, xr, nb, xy, conf = (torch.cat(a).contiguous() for a in zip(*found))
    gain_bias = torch.tensor(np.stack([rng.uniform(0.8, 1.2, V), rng.uniform(-0.05, 0.05, V)], 1),
                             dtype=torch.float32, device="cuda")
    return dict(cams=cams, ref=ref, ref_xy=xr, nb=nb, nb_xy=xy, conf=conf,
                frames=_frames(seed, cams), gain_bias=gain_bias)


def _seed_shapes(case):
    m = case["m"]
    return dict(means=(m, 3), log_scales=(m, 3), quats=(m, 4), opacity_logits=(m,),
                sh=(m, (case["degree"] + 1) ** 2, 3), normals=(m, 3))


def _upkeep(case, seed):
    g = _generator(seed, 5)
    n, P = case["n"], case["width"] * case["height"]
    f32 = lambda t: t.float().contiguous()  # noqa: E731
    return dict(means=f32(_normal(g, n, 3)), ema=f32(_normal(g, n, 3)),
                log_scales=f32(-1.5 + _normal(g, n, 3)), logits=f32(-2 + 3 * _normal(g, n)),
                obs=torch.randint(0, 10, (n,), generator=g, device="cuda", dtype=torch.int32),
                vis=f32(3 * _uniform(g, n)),
                a=f32(_uniform(g, case["pairs"], P)), b=f32(_uniform(g, case["pairs"], P)))


# ------------------------------------------------------------------------------------------
# One pass of each kind
# ------------------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind, case=case)
    if kind == "seed":
        s.update(_matches(case, seed))
        s["r"] = Renderer(0)
        # The map's arrays, with room for every match.
        s["map"] = {k: torch.zeros(v, device="cuda") for k, v in _seed_shapes(case).items()}
        return s
    if kind == "upkeep":
        s.update(_upkeep(case, seed))
        s["r"] = Renderer(0)
        s["map"] = MapRegularizer(s["r"].ctx, s["ema"])
        s["map"].obs_count.copy_(s["obs"])
        s["map"].vis_score.copy_(s["vis"])
        s["counts"] = torch.empty((case["pairs"], 2), dtype=torch.int64, device="cuda")
        s["iou"] = torch.empty(case["pairs"], device="cuda")
        return s
    params, cams = _scene(case, seed)
    n, K, V, P = case["n"], (case["degree"] + 1) ** 2, case["views"], _pixels(cams)
    r = Renderer(0, backward_pixels_per_thread=case["bwd_ppt"])
    s.update(r=r, cams=cams, n=n, K=K, V=V, p=[params[k] for k in PARAMS])
    if kind == "train":
        s["twist"] = torch.zeros((V, 6), device="cuda", requires_grad=True)
        for p in s["p"]:
            p.requires_grad_(True)
        s["up"] = _upstream(seed, P, False)[0]
    elif kind in ("map", "window"):
        s["cams_c"] = binding.make_cameras(cams)
        s["up"], s["up_depth"] = _upstream(seed, P, kind == "map")
        s["images"] = (torch.empty((P, 3), device="cuda"), torch.empty(P, device="cuda"),
                       torch.empty(P, device="cuda"))
        shapes = dict(means=(n, 3), log_scales=(n, 3), quats=(n, 4), opacity_logits=(n,),
                      sh=(n, K, 3), pose=(V, 6))
        s["grads"] = {k: torch.empty(v, device="cuda") for k, v in shapes.items()}
        s["state"] = 0
        if kind == "map":
            g = _generator(seed, 6)
            s["ema"] = s["p"][0] + 0.02 * torch.randn((n, 3), generator=g, device="cuda")
            s["map"] = MapRegularizer(r.ctx, s["ema"])
    elif kind == "track":
        s["tracker"] = Tracker(r, cams, _frames(seed, cams), lr=2e-3, iterations=30)
        s["pose0"] = s["tracker"].world_to_cam.clone()
        s["tracker"].step(*s["p"])
        s["graph"] = s["tracker"].capture(*s["p"])
    return s


def run(s):
    kind = s["kind"]
    if kind == "preview":
        with torch.no_grad():
            return list(render(s["r"], s["cams"], *s["p"]))
    if kind == "train":
        color, depth, alpha = render(s["r"], s["cams"], *s["p"], s["twist"])
        grads = torch.autograd.grad(color, s["p"] + [s["twist"]], s["up"])
        return [color.detach(), depth.detach(), alpha.detach(), *grads]
    if kind == "window":
        r = s["r"]
        *_, s["state"] = r.forward_raw(*s["p"], s["cams_c"], state=s["state"], out=s["images"])
        r.backward_raw(s["state"], s["n"], s["K"], s["V"], s["up"], out=s["grads"])
        return dict(images=s["images"], grads=s["grads"])
    if kind == "map":
        r, m = s["r"], s["map"]
        m.ema_means.copy_(s["ema"])
        m.obs_count.zero_()
        m.vis_score.zero_()
        stream = r.stream_handle()
        *_, s["state"] = r.forward_raw(*s["p"], s["cams_c"], state=s["state"], out=s["images"])
        r.backward_raw(s["state"], s["n"], s["K"], s["V"], s["up"], s["up_depth"], out=s["grads"],
                       reg=m.reg())
        m.update_anchor(s["p"][0], stream)
        keep, n_keep = m.prune_mask(s["p"][1], s["p"][3], stream)
        return dict(images=s["images"], grads=s["grads"], value=m.value, ema=m.ema_means,
                    obs=m.obs_count, vis=m.vis_score, keep=keep, n_keep=n_keep)
    if kind == "track":
        t = s["tracker"]
        t.world_to_cam.copy_(s["pose0"])
        t.adam_state.zero_()
        t.step_count.zero_()
        s["graph"].replay()
        return dict(images=t.images, loss=t.loss, gain_bias=t.gain_bias, d_pose=t.d_pose,
                    pose=t.world_to_cam)
    if kind == "seed":
        r, stream = s["r"], s["r"].stream_handle()
        tri = seeding.triangulate(r.ctx, s["cams"], s["ref"], s["ref_xy"], s["nb"], s["nb_xy"],
                                  s["conf"], r.device, stream)
        seeds = seeding.init_seeds(r.ctx, s["cams"], tri, s["frames"], s["gain_bias"], r.device,
                                   s["case"]["degree"], stream, voxel=s["case"]["voxel"])
        for k, v in s["map"].items():
            v[:len(seeds[k])].copy_(seeds[k])
        return dict(tri={k: v for k, v in tri.items() if k != "inputs"}, map=s["map"],
                    count=len(seeds["index"]))
    r, m, c = s["r"], s["map"], s["case"]
    stream = r.stream_handle()
    m.ema_means.copy_(s["ema"])
    m.update_anchor(s["means"], stream)
    keep, n_keep = m.prune_mask(s["log_scales"], s["logits"], stream)
    r.ctx.covisibility(s["a"].data_ptr(), s["b"].data_ptr(), c["width"] * c["height"], c["pairs"],
                       0.5, s["counts"].data_ptr(), s["iou"].data_ptr(), stream)
    return dict(ema=m.ema_means, keep=keep, n_keep=n_keep, counts=s["counts"], iou=s["iou"])


# ------------------------------------------------------------------------------------------
# What a pass cannot do without
# ------------------------------------------------------------------------------------------
# List positions a pixel visits before it is opaque, by scene, and FP32 operations per position
# of the forward and backward compositing.
POSITIONS = dict(slab=20, room=50, clutter=60, spread=119)
FORWARD_FLOPS, BACKWARD_FLOPS = 15, 40
TRIANGULATION_FLOPS = 4000  # FP64, per two-view hypothesis


def _case_pixels(case):
    if case["width"]:
        return case["views"] * case["width"] * case["height"]
    return case["views"] * sum(w * h for w, h in RESOLUTIONS) // len(RESOLUTIONS)


def work(case):
    kind = case["kind"]
    if kind == "seed":
        m, k, K = case["m"], case["k"], (case["degree"] + 1) ** 2
        frames = case["views"] * case["width"] * case["height"] * 12
        out = 56 + 4 * (15 + 3 * K)
        return dict(bytes=m * (20 + 24 * k + out) + frames, flops=m * k * TRIANGULATION_FLOPS)
    if kind == "upkeep":
        P = case["pairs"] * case["width"] * case["height"]
        return dict(bytes=case["n"] * (60 + 25) + 8 * P, flops=case["n"] * 30 + 2 * P)
    P, n, K = _case_pixels(case), case["n"], (case["degree"] + 1) ** 2
    params = 4 * n * (11 + 3 * K)
    at = P * POSITIONS[case["scene"]]
    if kind == "preview":
        return dict(bytes=params + 20 * P, flops=at * FORWARD_FLOPS)
    flops = at * (FORWARD_FLOPS + BACKWARD_FLOPS)
    if kind == "track":  # images written, colour and opacity read with the frame and its weights
        return dict(bytes=params + 20 * P + 44 * P, flops=flops)
    grads = params + (12 * n * 3 + 40 * n if kind == "map" else 0)
    return dict(bytes=params + grads + 20 * P + (16 if kind == "map" else 12) * P, flops=flops)


# ------------------------------------------------------------------------------------------
# The same results in 64 bits, in plain torch
# ------------------------------------------------------------------------------------------
ALPHA_MIN, ALPHA_MAX, T_MIN, ZNEAR, EPS2D, JAC_CLAMP = (
    float(np.float32(x)) for x in (1 / 255, 0.99, 1e-4, 0.2, 0.3, 1.3))
TILE = 16
CHUNK = 1 << 24  # (pixel, Gaussian) positions evaluated at a time


def _sh_basis(d, degree):
    x, y, z = d.unbind(-1)
    pi = math.pi
    Y = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if degree >= 1:
        c = math.sqrt(3 / (4 * pi))
        Y += [-c * y, c * z, -c * x]
    if degree >= 2:
        a, b = math.sqrt(15 / pi) / 2, math.sqrt(5 / pi) / 4
        Y += [a * x * y, -a * y * z, b * (2 * z * z - x * x - y * y), -a * x * z,
              a / 2 * (x * x - y * y)]
    if degree >= 3:
        a, b = math.sqrt(35 / (2 * pi)) / 4, math.sqrt(105 / pi) / 2
        c, e = math.sqrt(21 / (2 * pi)) / 4, math.sqrt(7 / pi) / 4
        Y += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (4 * z * z - x * x - y * y),
              e * z * (2 * z * z - 3 * x * x - 3 * y * y), -c * x * (4 * z * z - x * x - y * y),
              b / 2 * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(Y, -1)


def _rotation(q):
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)],
                       1).reshape(-1, 3, 3)


def _project(p, cam, twist, degree, pick):
    """Projected quantities of the Gaussians `pick` in one view: pixel mean, inverse 2-D
    covariance, colour, depth, opacity. The twist moves the pose to first order."""
    dev = dict(device="cuda", dtype=torch.float64)
    R, t = torch.tensor(cam["R"], **dev), torch.tensor(cam["t"], **dev)
    w0, w1, w2 = twist[3:].unbind()
    zero = torch.zeros_like(w0)
    left = torch.eye(3, **dev) + torch.stack([zero, -w2, w1, w2, zero, -w0, -w1, w0,
                                              zero]).reshape(3, 3)
    R, t = left @ R, left @ t + twist[:3]
    m, ls, q, lg, sh = (x[pick] for x in p)
    xc = m @ R.T + t
    z = xc[:, 2]
    u = xc[:, :2] / z[:, None]
    f = torch.tensor([float(np.float32(cam["fx"])), float(np.float32(cam["fy"]))], **dev)
    c = torch.tensor([float(np.float32(cam["cx"])), float(np.float32(cam["cy"]))], **dev)
    lim = JAC_CLAMP * 0.5 * torch.tensor([cam["width"], cam["height"]], **dev) / f
    uc = torch.maximum(torch.minimum(u, lim), -lim)
    J = torch.zeros((len(m), 2, 3), **dev)
    J[:, 0, 0], J[:, 1, 1] = f[0] / z, f[1] / z
    J[:, :, 2] = -f * uc / z[:, None]
    A = J @ R @ (_rotation(q) * torch.exp(ls)[:, None, :])
    cov = A @ A.transpose(1, 2) + EPS2D * torch.eye(2, **dev)
    det = cov[:, 0, 0] * cov[:, 1, 1] - cov[:, 0, 1] ** 2
    conic = torch.stack([cov[:, 1, 1], -cov[:, 0, 1], cov[:, 0, 0]], 1) / det[:, None]
    d = m + t @ R  # mean minus camera centre
    Y = _sh_basis(d / d.norm(dim=1, keepdim=True), degree)
    rgb = ((sh * Y[..., None]).sum(1) + 0.5).clamp(min=0)
    o = torch.sigmoid(lg)
    reach = 2 * torch.log(o / ALPHA_MIN)
    extent = torch.sqrt(reach.clamp(min=0)[:, None] * torch.stack([cov[:, 0, 0], cov[:, 1, 1]], 1))
    return torch.cat([f * u + c, conic, rgb, z[:, None], o[:, None]], 1), extent, reach


def _tile_lists(proj, extent, z32, cam):
    """(tile, entry) pairs whose boxes overlap, tiles in order and near to far inside each."""
    tx, ty = -(-cam["width"] // TILE), -(-cam["height"] // TILE)
    lo = torch.floor((proj[:, :2] - extent - 0.01) / TILE).long()
    hi = torch.floor((proj[:, :2] + extent + 0.01) / TILE).long()
    most = torch.tensor([tx - 1, ty - 1], device="cuda")
    lo, hi = lo.clamp(min=0), torch.minimum(hi, most)
    size = (hi - lo + 1).clamp(min=0)
    order = torch.argsort(z32, stable=True)
    count = (size[:, 0] * size[:, 1])[order]
    e = torch.repeat_interleave(order, count)
    at = torch.arange(len(e), device="cuda") - torch.repeat_interleave(count.cumsum(0) - count, count)
    tile = (lo[e, 1] + at // size[e, 0]) * tx + lo[e, 0] + at % size[e, 0]
    tile, by = torch.sort(tile, stable=True)
    return e[by], torch.bincount(tile, minlength=tx * ty)


def _blend(proj, entries, counts, cam, grads):
    """Images of one view from its tile lists and, given upstream gradients, the gradient with
    respect to the projected quantities."""
    W, H = cam["width"], cam["height"]
    tx = -(-W // TILE)
    dev = dict(device="cuda", dtype=torch.float64)
    out = torch.zeros((H, W, 5), **dev)
    g_proj = torch.zeros_like(proj)
    first = counts.cumsum(0) - counts
    order = torch.argsort(counts)
    lengths = counts[order].cpu()
    i, T = 0, len(counts)
    px = torch.arange(TILE * TILE, device="cuda")
    while i < T:
        if lengths[i] == 0:
            i = int((lengths == 0).sum())
            continue
        j = i + 1  # tiles of similar length together
        while j < T and int(lengths[j]) * (j + 1 - i) * TILE * TILE <= CHUNK:
            j += 1
        tiles, L = order[i:j], int(lengths[j - 1])
        slot = torch.arange(L, device="cuda")
        live = slot < counts[tiles][:, None]
        idx = entries[torch.where(live, first[tiles][:, None] + slot, 0)]
        x = (tiles % tx * TILE)[:, None] + px % TILE
        y = (tiles // tx * TILE)[:, None] + px // TILE
        inside = (x < W) & (y < H)
        where = (y.clamp(max=H - 1), x.clamp(max=W - 1))
        with torch.set_grad_enabled(grads is not None):
            g = proj[idx].detach().requires_grad_(grads is not None)  # [B, L, 10]
            dx = x[:, None] - g[..., 0:1]
            dy = y[:, None] - g[..., 1:2]
            power = -0.5 * (g[..., 2:3] * dx * dx + g[..., 4:5] * dy * dy) - g[..., 3:4] * dx * dy
            a = (g[..., 9:10] * torch.exp(power)).clamp(max=ALPHA_MAX)
            a = torch.where((a >= ALPHA_MIN) & live[..., None], a, 0.0)
            after = torch.cumprod(1 - a, 1)
            # Transmittance only falls: everything from the stop on is below the bound.
            a = torch.where(after >= T_MIN, a, 0.0)
            after = torch.cumprod(1 - a, 1)
            w = a * torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
            rgbz = torch.einsum("blp,blc->bpc", w, g[..., 5:9])
            img = torch.cat([rgbz, (1 - after[:, -1])[..., None]], 2)
            if grads is not None:
                up = grads[where] * inside[..., None]
                (gg,) = torch.autograd.grad(img, g, up)
                g_proj.index_put_((idx[live],), gg[live], accumulate=True)
        out[where[0][inside], where[1][inside]] = img.detach()[inside]
        i = j
    return out.reshape(-1, 5), g_proj


def _reference(params, cams, degree, upstream):
    """(images [P,5], gradients of the parameters, twist gradients [V,6]); `upstream` maps the
    images to their gradient [P,5], or is None."""
    p = [params[k].double() for k in PARAMS]
    views, images = [], []
    no_twist = torch.zeros(6, device="cuda", dtype=torch.float64)
    for cam in cams:
        R = torch.tensor(cam["R"], device="cuda").double()
        z = p[0] @ R[2] + float(cam["t"][2])
        pick = (z > ZNEAR).nonzero()[:, 0]
        with torch.no_grad():
            proj, extent, reach = _project(p, cam, no_twist, degree, pick)
            near = torch.tensor([cam["width"], cam["height"]], device="cuda")
            on = (reach >= 0) & (proj[:, :2] + extent > -1).all(1) & (
                proj[:, :2] - extent < near).all(1)
            pick, proj, extent = pick[on], proj[on], extent[on]
        lists = _tile_lists(proj, extent, proj[:, 8].float(), cam)
        views.append((cam, pick, proj, lists))
        images.append(_blend(proj, *lists, cam, None)[0])
    images = torch.cat(images)
    if upstream is None:
        return images, None, None
    up = upstream(images)
    for x in p:
        x.requires_grad_(True)
    total, twists, at = [torch.zeros_like(x) for x in p], [], 0
    for cam, pick, proj, lists in views:
        size = cam["width"] * cam["height"]
        g = up[at:at + size].reshape(cam["height"], cam["width"], 5)
        at += size
        _, g_proj = _blend(proj, *lists, cam, g)
        twist = no_twist.clone().requires_grad_(True)
        again, *_ = _project(p, cam, twist, degree, pick)
        *gp, gt = torch.autograd.grad(again, [*p, twist], g_proj)
        total = [a + b for a, b in zip(total, gp)]
        twists.append(gt)
    return images, total, torch.stack(twists)


def _exact_render(case, seed):
    params, cams = _scene(case, seed)
    kind, P = case["kind"], _pixels(cams)
    if P * POSITIONS[case["scene"]] > 1.5e9:
        return None  # minutes in 64 bits
    split = lambda im: [im[:, :3], im[:, 3], im[:, 4]]  # noqa: E731
    if kind == "preview":
        return split(_reference(params, cams, case["degree"], None)[0])
    if kind == "track":
        return _exact_track(case, seed, params, cams, split)
    uc, ud = _upstream(seed, P, kind == "map")
    up = torch.zeros((P, 5), device="cuda", dtype=torch.float64)
    up[:, :3] = uc
    if ud is not None:
        up[:, 3] = ud
    images, g, twists = _reference(params, cams, case["degree"], lambda _: up)
    if kind == "train":
        return [*split(images), *g, twists]
    grads = dict(zip(PARAMS, g), pose=twists)
    if kind == "window":
        return dict(images=split(images), grads=grads)
    gen = _generator(seed, 6)
    n = case["n"]
    m0 = params["means"]
    ema = (m0 + 0.02 * torch.randn((n, 3), generator=gen, device="cuda")).double()
    li, la, lm, eta = (float(np.float32(x)) for x in (0.01, 1e-3, 0.1, 0.1))
    p = [params[k].double().requires_grad_(True) for k in PARAMS[:4]]
    s2 = torch.exp(2 * p[1])
    reg = (li * (s2 - s2.mean(1, keepdim=True)).norm(dim=1).sum() + lm * (p[0] - ema).square().sum()
           + la * (p[3].abs() + 2 * torch.log1p(torch.exp(-p[3].abs()))).sum())
    for k, x in zip(PARAMS[:4], torch.autograd.grad(reg, p, allow_unused=True)):
        if x is not None:
            grads[k] = grads[k] + x
    return dict(images=split(images), grads=grads, value=reg.detach().reshape(1),
                ema=(ema + eta * (m0.double() - ema)), obs=None, vis=None, keep=None, n_keep=None)


def _exact_track(case, seed, params, cams, split):
    frames = _frames(seed, cams).double()
    sizes = [c["width"] * c["height"] for c in cams]
    tau_a, tau_g = 0.5, float(np.float32(0.05))
    weights = []
    for o, c in zip(frames.split(sizes), cams):
        o = o.reshape(c["height"], c["width"], 3)
        gy, gx = torch.gradient(o, dim=(0, 1))
        weights.append(((gx.square() + gy.square()).sum(2).sqrt() / tau_g).clamp(max=1).reshape(-1))
    loss, fit = [], []

    def upstream(images):
        ups = []
        for im, o, wg in zip(images.split(sizes), frames.split(sizes), weights):
            c = im[:, :3]
            g = ((c - c.mean()) * (o - o.mean())).sum() / (c - c.mean()).square().sum()
            b = o.mean() - g * c.mean()
            w = (im[:, 4] / tau_a).clamp(0, 1) * wg
            res = o - (g * c + b)
            loss.append((w * res.abs().sum(1)).sum())
            fit.append(torch.stack([g, b]))
            up = torch.zeros_like(im)
            up[:, :3] = -(w * g)[:, None] * torch.sign(res)
            ups.append(up)
        return torch.cat(ups)

    images, _, twists = _reference(params, cams, case["degree"], upstream)
    poses = []
    lr, eps = float(np.float32(2e-3)), float(np.float32(1e-8))
    for c, g in zip(cams, twists):
        xi = -lr * g / (g.abs() + eps)  # Adam's first step
        w0, w1, w2 = xi[3:].tolist()
        M = torch.zeros((4, 4), device="cuda", dtype=torch.float64)
        M[:3, :3] = torch.tensor([[0, -w2, w1], [w2, 0, -w0], [-w1, w0, 0]])
        M[:3, 3] = xi[:3]
        T = torch.eye(4, device="cuda", dtype=torch.float64)
        T[:3, :3], T[:3, 3] = torch.tensor(c["R"]), torch.tensor(c["t"])
        poses.append((torch.linalg.matrix_exp(M) @ T)[:3].reshape(12))
    return dict(images=split(images), loss=torch.stack(loss), gain_bias=torch.stack(fit),
                d_pose=twists, pose=torch.stack(poses))


def _exact_triangulation(s, R, t, f, c):
    """The best accepted two-view hypothesis of every reference pixel."""
    K = torch.zeros((len(f), 3, 3), device="cuda", dtype=torch.float64)
    K[:, 0, 0], K[:, 1, 1], K[:, 2, 2] = f[:, 0], f[:, 1], 1
    K[:, :2, 2] = c
    Pm = K @ torch.cat([R, t[..., None]], 2)
    centre = -(R.transpose(1, 2) @ t[..., None])[..., 0]
    r, nb = s["ref"].long(), s["nb"].long()
    has = nb >= 0
    nv = nb.clamp(min=0)

    def rows(v, xy):
        return xy[..., :, None] * Pm[v][..., 2:3, :] - Pm[v][..., :2, :]

    k = nb.shape[1]
    ref_xy = s["ref_xy"][:, None].expand(-1, k, 2)
    rr = r[:, None].expand(-1, k)
    A = torch.cat([rows(rr, ref_xy), rows(nv, s["nb_xy"])], 2)
    Xh = torch.linalg.svd(A.reshape(-1, 4, 4))[2][:, 3].reshape(*nb.shape, 4)
    X = Xh[..., :3] / Xh[..., 3:]

    def at(v):
        cam = (R[v] @ X[..., None])[..., 0] + t[v]
        return f[v] * cam[..., :2] / cam[..., 2:] + c[v], cam[..., 2]

    (ur, zr), (un, zn) = at(rr), at(nv)
    err = (0.5 * ((ur - ref_xy).square().sum(-1) + (un - s["nb_xy"]).square().sum(-1))).sqrt()
    d1, d2 = X - centre[rr], X - centre[nv]
    cosine = (d1 * d2).sum(-1) / (d1.norm(dim=-1) * d2.norm(dim=-1))
    angle = torch.arccos(cosine.clamp(-1, 1))
    least = float(np.float32(math.pi / 180))
    ok = has & (zr > 0) & (zn > 0) & ~(angle < least) & ~(err > 2.0)
    low = torch.where(ok, err, torch.inf).amin(1, keepdim=True)
    tie = ok & (err <= low + float(np.float32(1e-3)))
    best = torch.where(tie, angle, -1.0).argmax(1)
    valid = ok.any(1)
    one = lambda x: torch.where(valid, x[torch.arange(len(r), device="cuda"), best], 0.0)  # noqa: E731
    count = has.sum(1)
    kappa = (s["conf"].double() * has).sum(1) / count.clamp(min=1)
    X = torch.stack([one(X[..., a]) for a in range(3)], 1)
    return valid, X, one(err), one(angle), kappa


def _exact_seed(case, seed):
    s = _matches(case, seed)
    if case["m"] * case["k"] > 600000:
        return None
    cams = s["cams"]
    R = torch.tensor(np.stack([c["R"] for c in cams]), device="cuda").double()
    t = torch.tensor(np.stack([c["t"] for c in cams]), device="cuda").double()
    single = lambda *k: torch.tensor([[float(np.float32(c[x])) for x in k] for c in cams],  # noqa: E731
                                     device="cuda", dtype=torch.float64)
    f, c = single("fx", "fy"), single("cx", "cy")
    valid, X, err, angle, kappa = _exact_triangulation(s, R, t, f, c)
    tri = dict(valid=None, X=X, best=None, err=err, angle=angle, kappa=kappa)
    if case["voxel"] > 0:
        return dict(tri=tri, map=dict.fromkeys(_seed_shapes(case)), count=None)
    v = valid.nonzero()[:, 0]
    X, err, angle, kappa, r = X[v], err[v], angle[v], kappa[v], s["ref"].long()[v]
    one = torch.ones_like(X[:, :1])
    pairs = [(0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)]
    origin = X.mean(0)
    Xo = X - origin
    feats = torch.cat([one, Xo, torch.stack([Xo[:, a] * Xo[:, b] for a, b in pairs], 1)], 1)
    h = float(np.float32(0.05))
    mom = torch.cat([((q[:, None] - X[None]).square().sum(-1) <= h * h).double() @ feats
                     for q in X.split(512)])
    cnt = mom[:, :1]
    mu = mom[:, 1:4] / cnt
    S = torch.zeros((len(X), 3, 3), device="cuda", dtype=torch.float64)
    for j, (a, b) in enumerate(pairs):
        S[:, a, b] = S[:, b, a] = mom[:, 4 + j] / cnt[:, 0] - mu[:, a] * mu[:, b]
    normal = torch.cat([torch.linalg.eigh(x)[1][:, :, 0] for x in S.split(16384)])
    centre = -(R.transpose(1, 2) @ t[..., None])[..., 0]
    to = centre[r] - X
    normal = normal * torch.where((normal * to).sum(1, keepdim=True) < 0, -1.0, 1.0)
    normal = torch.where(cnt >= 3, normal, to / to.norm(dim=1, keepdim=True))
    cam = (R[r] @ X[..., None])[..., 0] + t[r]
    J = torch.zeros((len(X), 2, 3), device="cuda", dtype=torch.float64)
    J[:, 0, 0], J[:, 1, 1] = f[r, 0] / cam[:, 2], f[r, 1] / cam[:, 2]
    J[:, :, 2] = -f[r] * cam[:, :2] / cam[:, 2:].square()
    JR = J @ R[r]
    perp = torch.linalg.det(JR @ JR.transpose(1, 2)) ** -0.25
    par = torch.minimum(perp * (1 + err) / torch.sin(angle), 10 * perp)
    ls = torch.stack([perp, perp, par], 1).log()
    lo, hi = float(np.float32(0.1)), float(np.float32(0.9))
    alpha = lo + (hi - lo) * kappa.float().double()
    padded = lambda x: torch.cat([x, x.new_zeros(case["m"] - len(x), *x.shape[1:])])  # noqa: E731
    found = dict(means=X, log_scales=ls, opacity_logits=torch.log(alpha / (1 - alpha)),
                 normals=normal)
    return dict(tri=tri, count=None, map={k: padded(found[k]) if k in found else None
                                          for k in _seed_shapes(case)})


def exact(case, seed):
    if case["kind"] == "seed":
        return _exact_seed(case, seed)
    if case["kind"] == "upkeep":
        s = _upkeep(case, seed)
        eta = float(np.float32(0.1))
        a, b = s["a"] > 0.5, s["b"] > 0.5
        iou = (a & b).sum(1).double() / (a | b).sum(1).clamp(min=1)
        return dict(ema=s["ema"].double() + eta * (s["means"].double() - s["ema"].double()),
                    keep=None, n_keep=None, counts=None, iou=iou)
    return _exact_render(case, seed)
