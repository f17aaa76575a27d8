"""Performance cases of the cloud renderer, through its Python entry points.

What the cases stand for: a renderer that marches cloud images (from a thumbnail
of 128x128 to 1920x1080, 8 jittered view steps for real time, 128 for reference
quality), resolves them against the reprojected history of the previous frame
(fused, or as the separate motion and TAA calls), lays a low-resolution cloud
buffer over a background, and renders many uneven views in one launch.

Inputs are seeded: volume descriptors, cameras and lighting constants from
``paper_1609_05344_gb300.inputs``, frames, histories and motion fields from a
seeded generator on the device.  ``exact`` evaluates the same definitions in
FP64 with torch and shares no code with the library.
"""
from __future__ import annotations

import functools
import math
import random

import torch

from paper_1609_05344_gb300 import api
from paper_1609_05344_gb300 import inputs as I

RENDER = dict(kind="render", volume="full", precision="fp32", light_steps=6, jitter="pixel",
              integration="analytic", height=500.0)


def listed() -> list:
    return [
        # a thumbnail or probe image: latency and launches are all of it
        dict(RENDER, name="render-128", volume="tiny", width=128, rows=128, steps=16, jitter="none"),
        # reference quality: 128 fixed steps at 720p
        dict(RENDER, name="render-reference", width=1280, rows=720, steps=128, jitter="none"),
        # the real-time path: 8 jittered steps at 1080p, FP32 and FP16 volumes
        dict(RENDER, name="render-1080p", width=1920, rows=1080, steps=8),
        dict(RENDER, name="render-1080p-fp16", width=1920, rows=1080, steps=8, precision="fp16"),
        # a half-resolution cloud buffer of an odd size, one offset for all rays of the frame
        dict(RENDER, name="render-half-odd", width=957, rows=541, steps=8, jitter="frame"),
        # one whole real-time frame: render, then reprojection and TAA resolve
        dict(RENDER, name="frame-1080p", kind="frame", width=1920, rows=1080, steps=8, history="fp32"),
        # the resolve alone: full size with FP32 history, ragged size with FP16 history
        dict(kind="resolve", name="resolve-1080p", width=1920, rows=1080, history="fp32", height=500.0),
        dict(kind="resolve", name="resolve-odd-fp16", width=1277, rows=717, history="fp16", height=500.0),
        # motion and TAA as separate calls (an application with its own motion vectors)
        dict(kind="motion-taa", name="motion-taa-1080p", width=1920, rows=1080, history="fp32",
             height=500.0),
        # a half-resolution FP16 cloud buffer laid over a 1080p scene
        dict(kind="composite", name="composite-1080p", width=1920, rows=1080, cloud_width=960,
             cloud_rows=540, history="fp16"),
        # a serving tick: new cameras for 8 small views, the launch replayed from its graph
        dict(kind="views", name="views-8", views=8, precision="fp16", min_width=640, min_rows=360,
             max_width=1280, max_rows=720, steps="8,16", layout=4),
        # many uneven views, up to reference quality, in one persistent launch
        dict(kind="batch", name="batch-64", views=64, precision="bf16", min_width=256, min_rows=256,
             max_width=1920, max_rows=1080, steps="8,16,32,128", layout=4),
    ]


def _log_int(rng: random.Random, lo: int, hi: int) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random) -> dict:
    """Another case of the same ranges: image sizes between a thumbnail and 1080p, 8 to 128
    view steps, every storage precision, jitter mode and integration rule, cameras below,
    inside and above the layer."""
    kind = rng.choice(["render", "render", "render", "frame", "resolve", "motion-taa", "composite",
                       "views", "batch"])
    size = dict(width=_log_int(rng, 97, 1920), rows=_log_int(rng, 65, 1080))
    height = rng.choice([round(rng.uniform(0.0, 1400.0), 1)] * 3 + [2500.0, 5200.0])
    history = rng.choice(["fp32", "fp16"])
    if kind in ("render", "frame"):
        case = dict(RENDER, kind=kind, steps=_log_int(rng, 8, 128), height=height,
                    volume=rng.choice(["full", "full", "full", "tiny"]),
                    precision=rng.choice(["fp32", "fp16", "bf16", "unorm16"]),
                    light_steps=rng.choice([6, 6, 6, 4, 9]),
                    jitter=rng.choice(["pixel", "pixel", "frame", "none"]),
                    integration=rng.choice(["analytic", "analytic", "basic"]), **size)
        return dict(case, history=history) if kind == "frame" else case
    if kind in ("resolve", "motion-taa"):
        return dict(kind=kind, history=history, height=height, **size)
    if kind == "composite":
        part = rng.choice([1, 2, 3, 4])
        return dict(kind=kind, history=history, cloud_width=max(1, size["width"] // part),
                    cloud_rows=max(1, size["rows"] // part), **size)
    if kind == "views":
        return dict(kind=kind, views=rng.randint(1, 16), precision=rng.choice(["fp32", "fp16"]),
                    min_width=320, min_rows=180, max_width=rng.randint(640, 1280),
                    max_rows=rng.randint(360, 720), steps="8,16", layout=rng.randint(0, 999))
    return dict(kind=kind, views=rng.randint(2, 40), precision=rng.choice(["fp32", "fp16", "bf16"]),
                min_width=rng.randint(64, 256), min_rows=rng.randint(64, 256),
                max_width=rng.randint(300, 1920), max_rows=rng.randint(300, 1080),
                steps=rng.choice(["8,16", "8,16,32", "8,16,32,128"]), layout=rng.randint(0, 999))


# --------------------------------------------------------------------------- inputs

def _descriptor(case: dict, seed: int) -> dict:
    return I.volume_desc(case.get("volume", "full"), 1 + seed % 100003, case.get("precision", "fp32"))


def _params(case: dict) -> dict:
    return I.params(jitter_mode="frame" if case.get("jitter") == "frame" else "pixel")


def _cameras(case: dict, seed: int) -> tuple:
    """The previous and the current camera: a slow seeded orbit as in a moving view."""
    rng = random.Random(seed * 7919 + 11)
    x, y = rng.uniform(-3000.0, 3000.0), rng.uniform(-3000.0, 3000.0)
    yaw, pitch = rng.uniform(0.0, 360.0), rng.uniform(11.0, 21.0)
    if case["height"] > I.SLAB_HI_M:
        pitch = -pitch
    return tuple(I.camera((x + 13.0 * f, y - 4.0 * f, case["height"]), yaw + 0.25 * f, pitch, 60.0)
                 for f in range(2))


def _jitter_frame(case: dict, seed: int) -> int:
    return -1 if case["jitter"] == "none" else seed % 997


def _generator(seed: int) -> torch.Generator:
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _image(g: torch.Generator, rows: int, width: int, noise: float) -> torch.Tensor:
    """A cloud-buffer-like premultiplied RGBA image: smooth blobs and per-pixel noise."""
    y = torch.arange(rows, device="cuda", dtype=torch.float32)[:, None]
    x = torch.arange(width, device="cuda", dtype=torch.float32)[None, :]
    p = torch.rand((6, 3), generator=g, device="cuda")
    alpha = torch.zeros((rows, width), device="cuda")
    for k in range(6):
        r = (0.1 + 0.3 * p[k, 2]) * max(width, rows)
        alpha += torch.exp(-((x - p[k, 0] * width) ** 2 + (y - p[k, 1] * rows) ** 2) / (r * r))
    n = torch.randn((2, rows, width), generator=g, device="cuda")
    alpha = (0.7 * alpha + noise * n[0]).clamp(0.0, 1.0)
    tint = 0.4 + 1.6 * torch.rand(3, generator=g, device="cuda")
    rgb = ((alpha * (1.0 + noise * n[1]))[..., None] * tint).clamp(0.0, 2.0)
    return torch.cat([rgb, alpha[..., None]], dim=2).contiguous()


def _motion_field(g: torch.Generator, rows: int, width: int) -> torch.Tensor:
    """Smooth motion of a few pixels with a little noise, some of it pointing off the screen."""
    y = torch.arange(rows, device="cuda", dtype=torch.float32)[:, None]
    x = torch.arange(width, device="cuda", dtype=torch.float32)[None, :]
    c = 2.0 * torch.rand((2, 4), generator=g, device="cuda") - 1.0
    m = torch.stack([6.0 * (c[k, 0] + c[k, 1] * x / width + c[k, 2] * y / rows
                            + 0.3 * torch.sin(6.0 * c[k, 3] + x / 37.0 + y / 23.0))
                     for k in range(2)], dim=2)
    m += 0.05 * torch.randn(m.shape, generator=g, device="cuda")
    off = torch.rand((rows, width), generator=g, device="cuda") < 0.005
    return torch.where(off[..., None], torch.full_like(m, 2.0 * (width + rows)), m).contiguous()


def _frame_buffers(case: dict, seed: int) -> tuple:
    """(history in its own format, current frame)"""
    g = _generator(seed)
    hist = _image(g, case["rows"], case["width"], 0.03)
    cur = _image(g, case["rows"], case["width"], 0.15)
    return (hist.half() if case["history"] == "fp16" else hist), cur


def _composite_inputs(case: dict, seed: int) -> tuple:
    g = _generator(seed)
    cloud = _image(g, case["cloud_rows"], case["cloud_width"], 0.05)
    background = torch.rand((case["rows"], case["width"], 4), generator=g, device="cuda")
    return (cloud.half() if case["history"] == "fp16" else cloud), background


def _views(case: dict, seed: int, moved: bool) -> list:
    """Sizes and step counts follow the case's layout, cameras and jitter frames the seed."""
    views = I.random_views(case["views"], case["layout"], (case["max_width"], case["max_rows"]),
                           (case["min_width"], case["min_rows"]),
                           tuple(int(s) for s in case["steps"].split(",")))
    for v, w in zip(views, I.random_views(case["views"], seed)):
        v["camera"], v["jitter_frame"] = w["camera"], w["jitter_frame"]
        if moved:  # the next tick: the camera a little further on, the next jitter frame
            x, y, z = v["camera"]["pos"]
            v["camera"] = dict(v["camera"], pos=(x + 13.0, y - 4.0, z))
            v["jitter_frame"] += 1
    return views


def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    state = dict(case=case)
    if kind == "composite":
        state["cloud"], state["background"] = _composite_inputs(case, seed)
        state["out"] = torch.empty_like(state["background"])
        return state
    state["volume"], state["params"] = api.Volume(_descriptor(case, seed)), _params(case)
    if kind in ("views", "batch"):
        state["batch"] = api.Batch(state["volume"], state["params"], _views(case, seed, False))
        state["views"] = _views(case, seed, kind == "views")
        return state
    state["prev"], state["cam"] = _cameras(case, seed)
    shape = (case["rows"], case["width"])
    if kind in ("render", "frame"):
        state["jitter_frame"] = _jitter_frame(case, seed)
        state["image"] = torch.empty((*shape, 4), device="cuda")
    if kind != "render":
        state["history"], state["current"] = _frame_buffers(case, seed)
        state["out"] = torch.empty_like(state["history"])
    if kind == "motion-taa":
        state["given"] = _motion_field(_generator(seed + 1), *shape)
        state["motion"] = torch.empty((*shape, 2), device="cuda")
    return state


def run(state: dict):
    case, s = state["case"], state
    kind = case["kind"]
    if kind in ("render", "frame"):
        image = api.render(s["volume"], s["cam"], s["params"], case["width"], case["rows"],
                           case["steps"], case["light_steps"], s["jitter_frame"],
                           case["integration"], out=s["image"])
        if kind == "render":
            return image
        resolved = api.taa_reproject(s["volume"], s["params"], s["prev"], s["cam"], s["history"],
                                     image, out=s["out"], history_fmt=case["history"])
        return dict(image=image, resolved=resolved)
    if kind == "resolve":
        return api.taa_reproject(s["volume"], s["params"], s["prev"], s["cam"], s["history"],
                                 s["current"], out=s["out"], history_fmt=case["history"])
    if kind == "motion-taa":
        motion = api.motion(s["volume"], s["params"], s["prev"], s["cam"], case["width"],
                            case["rows"], out=s["motion"])
        resolved = api.taa(s["history"], s["current"], s["given"], out=s["out"],
                           history_fmt=case["history"])
        return dict(motion=motion, resolved=resolved)
    if kind == "composite":
        return api.composite(s["cloud"], s["background"], out=s["out"])
    if kind == "views":
        s["batch"].set_views(s["views"])
        return s["batch"].render(graph=True)
    return s["batch"].render()


# --------------------------------------------------------------------------- work

# Shares of the view steps of a frame that the method cannot skip: rays that reach the layer
# before the early out, and steps with density (each then needs its light samples); counted on
# the 8-step 1080p frame.  One density evaluation: two trilinear and one bilinear
# interpolation, the remap and the height profile.
_REACHED, _DENSE, _LOOKUP_FLOPS, _RAY_FLOPS, _LIT_FLOPS = 0.6, 0.07, 50, 150, 40


def _render_work(pixels: int, steps: int, light_steps: int) -> tuple:
    reached, lit = _REACHED * pixels * steps, _DENSE * pixels * steps
    flops = _RAY_FLOPS * pixels + (reached + lit * light_steps) * _LOOKUP_FLOPS + lit * _LIT_FLOPS
    return 16 * pixels, flops


def _tile_bytes(volume: str, precision: str) -> int:
    value = 4 if precision == "fp32" else 2
    return value * (64 ** 3 if volume == "tiny" else 128 ** 3 + 32 ** 3 + 512 ** 2)


def work(case: dict) -> dict:
    kind = case["kind"]
    if kind in ("views", "batch"):
        nbytes, flops = _tile_bytes("full", case["precision"]), 0.0
        for v in _views(case, 0, False):
            b, f = _render_work(v["width"] * v["height"], v["steps"], 6)
            nbytes, flops = nbytes + b, flops + f
        return dict(bytes=nbytes, flops=flops)
    pixels = case["width"] * case["rows"]
    hist = 16 if case.get("history") == "fp32" else 8
    if kind == "composite":
        return dict(bytes=32 * pixels + hist * case["cloud_width"] * case["cloud_rows"],
                    flops=(12 * 2 + 2 * 4 + 6) * pixels)
    nbytes, flops = 0, 0.0
    if kind in ("render", "frame"):
        nbytes, flops = _render_work(pixels, case["steps"], case["light_steps"])
        nbytes += _tile_bytes(case["volume"], case["precision"])
    if kind == "frame":
        nbytes -= 16 * pixels  # the image is written once; the resolve finds it there
    if kind in ("frame", "resolve"):  # motion about 60, history 24, range 64, clamp and blend 16
        nbytes, flops = nbytes + (16 + 2 * hist) * pixels, flops + 164 * pixels
    if kind == "motion-taa":
        nbytes, flops = nbytes + (8 + 16 + 8 + 2 * hist) * pixels, flops + 164 * pixels
    return dict(bytes=nbytes, flops=flops)


# --------------------------------------------------------------------------- exact (FP64)

_M32 = 0xFFFFFFFF
_D = dict(dtype=torch.float64, device="cuda")


def _pcg(v: torch.Tensor) -> torch.Tensor:
    s = (v * 747796405 + 2891336453) & _M32
    w = (((s >> ((s >> 28) + 4)) ^ s) * 277803737) & _M32
    return (w >> 22) ^ w


def _hash4(a, b, c, d) -> torch.Tensor:
    return _pcg(a ^ _pcg(b ^ _pcg(c ^ _pcg(d))))


def _fbm(n: int, dims: int, seed: int, salt: int) -> torch.Tensor:
    """Periodic 4-octave value noise on n^dims texels, indexed [z, y, x] or [y, x]."""
    k = torch.arange(n, device="cuda", dtype=torch.int64)
    total, amps = 0.0, 0.0
    for o in range(4):
        m = (n >> 4) << o
        lattice = torch.arange(m, device="cuda", dtype=torch.int64)
        key = torch.tensor((seed ^ (o * 0x9E37) ^ salt) & _M32, device="cuda", dtype=torch.int64)
        zero = torch.zeros((), device="cuda", dtype=torch.int64)
        x, y = lattice, lattice[:, None]
        z = lattice[:, None, None] if dims == 3 else zero
        v = (_hash4(x, y, z, key) >> 8).double() / 16777216.0
        lo, f = (k * m) // n, ((k * m) % n).double() / n
        for axis in range(dims):  # plain linear interpolation, one axis at a time
            shape = [1] * dims
            shape[axis] = n
            w = f.reshape(shape)
            v = v.index_select(axis, lo) * (1.0 - w) + v.index_select(axis, (lo + 1) % m) * w
        total, amps = total + 0.5 ** o * v, amps + 0.5 ** o
    return total / amps


def _corners(t: torch.Tensor) -> torch.Tensor:
    """Rows of the 2^d corner texels of every cell, x fastest."""
    rows = [t]
    for axis in range(t.dim() - 1, -1, -1):
        rows = rows + [torch.roll(r, -1, dims=axis) for r in rows]
    return torch.stack([r.reshape(-1) for r in rows], dim=1).contiguous()


@functools.lru_cache(maxsize=2)
def _tiles(seed: int, base_n: int, detail_n: int, weather_n: int) -> tuple:
    return (_corners(_fbm(base_n, 3, seed, 0xB45E)),
            _corners(_fbm(detail_n, 3, seed, 0xDE7A)) if detail_n else None,
            _corners(_fbm(weather_n, 2, seed, 0x3EA7)) if weather_n else None)


def _sample(rows: torch.Tensor, n: int, period: float, coords: list) -> torch.Tensor:
    index, fracs = 0, []
    for c in reversed(coords):
        u = c * (n / period) - 0.5
        fl = torch.floor(u)
        fracs.insert(0, u - fl)
        index = index * n + fl.long() % n
    v = rows[index]
    for f in fracs:  # x halves the row first, then y, then z
        v = v.reshape(v.shape[0], -1, 2)
        v = v[..., 0] + f[:, None] * (v[..., 1] - v[..., 0])
    return v[:, 0]


def _density(desc: dict, tiles: tuple, x, y, z) -> torch.Tensor:
    h = (z - desc["slab_lo"]) / (desc["slab_hi"] - desc["slab_lo"])
    g = (h / 0.1).clamp(0.0, 1.0) * ((1.0 - h) / 0.4).clamp(0.0, 1.0)
    r = _sample(tiles[0], desc["base_n"], desc["base_period"], [x, y, z]) - desc["coverage"]
    if tiles[1] is not None:
        r = r - desc["detail_weight"] * _sample(tiles[1], desc["detail_n"], desc["detail_period"], [x, y, z])
    r = (r / (1.0 - desc["coverage"])).clamp(min=0.0)
    if tiles[2] is not None:
        r = r * _sample(tiles[2], desc["weather_n"], desc["weather_period"], [x, y])
    return g * r


def _rays(cam: dict, width: int, rows: int, first: int, count: int) -> tuple:
    """Unit directions (n, 3) of the pixels of some image rows, and the pixel indices."""
    py, px = torch.meshgrid(torch.arange(first, first + count, device="cuda"),
                            torch.arange(width, device="cuda"), indexing="ij")
    px, py = px.reshape(-1), py.reshape(-1)
    t = cam["tan_half_fovy"]
    a = (2.0 * (px.double() + 0.5) / width - 1.0) * (width / rows) * t
    b = (1.0 - 2.0 * (py.double() + 0.5) / rows) * t
    f, r, u = (torch.tensor(cam[k], **_D) for k in ("forward", "right", "up"))
    v = f + a[:, None] * r + b[:, None] * u
    return v / v.norm(dim=1, keepdim=True), px, py


def _clip(desc: dict, prm: dict, z0: float, dz: torch.Tensor) -> tuple:
    """[t0, t1] of rays inside the layer and the far clip, and whether they enter it."""
    lo, hi = desc["slab_lo"] - z0, desc["slab_hi"] - z0
    flat = dz.abs() < 1e-8
    safe = torch.where(flat, torch.ones_like(dz), dz)
    a, b = lo / safe, hi / safe
    t0 = torch.minimum(a, b).clamp(min=0.0)
    t1 = torch.maximum(a, b).clamp(max=prm["t_max"])
    t0 = torch.where(flat, torch.zeros_like(t0), t0)
    t1 = torch.where(flat, torch.full_like(t1, prm["t_max"] if lo <= 0.0 <= hi else 0.0), t1)
    return t0, t1, t1 > t0


def _march(desc: dict, prm: dict, cam: dict, width: int, rows: int, steps: int, light_steps: int,
           jitter_frame: int, integration: str, rays_at_once: int = 1 << 21) -> torch.Tensor:
    tiles = _tiles(desc["seed"], desc["base_n"], desc["detail_n"], desc["weather_n"])
    sun = torch.tensor(prm["sun_dir"], **_D)
    sun = sun / sun.norm()
    radiance, ambient = torch.tensor(prm["sun_radiance"], **_D), torch.tensor(prm["ambient"], **_D)
    origin, alpha, g = torch.tensor(cam["pos"], **_D), prm["absorption"], prm["hg_g"]
    tau_max = prm["tau_max"] if prm["tau_max"] > 0.0 else math.inf
    key = torch.tensor((desc["seed"] ^ 0x4A17) & _M32, device="cuda", dtype=torch.int64)
    away = (torch.arange(light_steps, **_D) + 0.5) * prm["light_step"]
    out = torch.zeros((rows, width, 4), **_D)
    at_once = max(1, rays_at_once // width)
    for first in range(0, rows, at_once):
        count = min(at_once, rows - first)
        d, px, py = _rays(cam, width, rows, first, count)
        t0, t1, hit = _clip(desc, prm, cam["pos"][2], d[:, 2])
        hit = hit.nonzero()[:, 0]
        if hit.numel() == 0:
            continue
        d, px, py, t0 = d[hit], px[hit], py[hit], t0[hit]
        size = (t1[hit] - t0) / steps
        u = torch.full_like(t0, 0.5)
        if jitter_frame >= 0:
            if prm["jitter_mode"] == "frame":
                px, py = torch.zeros_like(px), torch.zeros_like(py)
            frame = torch.full_like(px, jitter_frame)
            u = (_hash4(px, py, frame, key) >> 8).double() / 16777216.0
        mu = d @ sun
        phase = (1.0 - g * g) / (4.0 * math.pi) * (1.0 + g * g - 2.0 * g * mu) ** -1.5
        tau, rgb = torch.zeros_like(t0), torch.zeros((t0.numel(), 3), **_D)
        live = torch.arange(t0.numel(), device="cuda")
        for i in range(steps):
            live = live[tau[live] < tau_max]
            if live.numel() == 0:
                break
            p = origin + (t0[live] + (i + u[live]) * size[live])[:, None] * d[live]
            rho = _density(desc, tiles, p[:, 0], p[:, 1], p[:, 2])
            dense = (rho > 0.0).nonzero()[:, 0]
            if dense.numel() == 0:
                continue
            on, p, rho = live[dense], p[dense], rho[dense]
            q = (p[:, None, :] + away[None, :, None] * sun).reshape(-1, 3)
            shade = torch.zeros_like(rho)
            if light_steps:
                shade = _density(desc, tiles, q[:, 0], q[:, 1], q[:, 2]).reshape(-1, light_steps).sum(1)
            light = torch.exp(-alpha * prm["light_step"] * shade) * phase[on]
            light = light[:, None] * radiance + ambient
            depth = alpha * rho * size[on]
            if integration == "analytic":
                weight = torch.exp(-tau[on]) * -torch.expm1(-depth)
            else:
                weight = torch.exp(-(tau[on] + depth)) * depth
            rgb[on] += weight[:, None] * light
            tau[on] += depth
        flat = out.view(-1, 4)[first * width:(first + count) * width]
        flat[hit] = torch.cat([rgb, -torch.expm1(-tau)[:, None]], dim=1)
    return out


def _exact_motion(desc: dict, prm: dict, prev: dict, cur: dict, width: int, rows: int) -> torch.Tensor:
    d, px, py = _rays(cur, width, rows, 0, rows)
    t0, _, hit = _clip(desc, prm, cur["pos"][2], d[:, 2])
    t = torch.where(hit & (t0 > 0.0), t0, torch.full_like(t0, prm["t_max"]))
    q = torch.tensor(cur["pos"], **_D) - torch.tensor(prev["pos"], **_D) + t[:, None] * d
    qx, qy, qz = (q @ torch.tensor(prev[k], **_D) for k in ("right", "up", "forward"))
    tan = prev["tan_half_fovy"]
    safe = torch.where(qz > 0.0, qz, torch.ones_like(qz))
    mx = px.double() + 0.5 - (qx / (safe * (width / rows) * tan) + 1.0) * (width / 2.0)
    my = py.double() + 0.5 - (1.0 - qy / (safe * tan)) * (rows / 2.0)
    far = torch.full_like(mx, 1e9)
    m = torch.stack([torch.where(qz > 0.0, mx, far), torch.where(qz > 0.0, my, far)], dim=1)
    return m.reshape(rows, width, 2)


def _bilinear(image: torch.Tensor, x: torch.Tensor, y: torch.Tensor) -> torch.Tensor:
    """image (h, w, 4) at texel-centre coordinates, clamped to the edge."""
    h, w = image.shape[:2]
    x0, y0 = torch.floor(x), torch.floor(y)
    fx, fy = (x - x0)[..., None], (y - y0)[..., None]
    xa, xb = x0.long().clamp(0, w - 1), (x0.long() + 1).clamp(0, w - 1)
    ya, yb = y0.long().clamp(0, h - 1), (y0.long() + 1).clamp(0, h - 1)
    top = image[ya, xa] * (1.0 - fx) + image[ya, xb] * fx
    bottom = image[yb, xa] * (1.0 - fx) + image[yb, xb] * fx
    return top * (1.0 - fy) + bottom * fy


def _exact_resolve(history: torch.Tensor, current: torch.Tensor, motion: torch.Tensor,
                   blend: float = 0.1) -> torch.Tensor:
    history, current = history.double(), current.double()
    h, w = current.shape[:2]
    y = torch.arange(h, **_D)[:, None] + 0.5
    x = torch.arange(w, **_D)[None, :] + 0.5
    qx, qy = x - motion[..., 0].double(), y - motion[..., 1].double()
    on = (qx >= 0.0) & (qx <= w) & (qy >= 0.0) & (qy <= h)
    old = _bilinear(history, torch.where(on, qx, x) - 0.5, torch.where(on, qy, y) - 0.5)
    pad = torch.nn.functional.pad(current.permute(2, 0, 1)[None], (1, 1, 1, 1), mode="replicate")[0]
    near = [pad[:, 1 + dy:1 + dy + h, 1 + dx:1 + dx + w] for dy in (-1, 0, 1) for dx in (-1, 0, 1)]
    near = torch.stack(near)
    low, high = near.amin(0).permute(1, 2, 0), near.amax(0).permute(1, 2, 0)
    old = torch.minimum(torch.maximum(old, low), high)
    return torch.where(on[..., None], old + blend * (current - old), current)


def exact(case: dict, seed: int):
    kind = case["kind"]
    if kind == "composite":
        cloud, background = _composite_inputs(case, seed)
        sw, sh, w, h = case["cloud_width"], case["cloud_rows"], case["width"], case["rows"]
        x = (torch.arange(w, **_D) + 0.5) * (sw / w) - 0.5
        y = (torch.arange(h, **_D) + 0.5) * (sh / h) - 0.5
        c = _bilinear(cloud.double(), x[None, :].expand(h, w), y[:, None].expand(h, w))
        return c + (1.0 - c[..., 3:]) * background.double()
    desc, prm = _descriptor(case, seed), _params(case)
    if kind in ("views", "batch"):
        return [_march(desc, prm, v["camera"], v["width"], v["height"], v["steps"], 6,
                       v["jitter_frame"], "analytic") for v in _views(case, seed, kind == "views")]
    prev, cam = _cameras(case, seed)
    w, h = case["width"], case["rows"]
    image = None
    if kind in ("render", "frame"):
        image = _march(desc, prm, cam, w, h, case["steps"], case["light_steps"],
                       _jitter_frame(case, seed), case["integration"])
    if kind == "render":
        return image
    history, current = _frame_buffers(case, seed)
    motion = _exact_motion(desc, prm, prev, cam, w, h)
    if kind == "frame":
        return dict(image=image, resolved=_exact_resolve(history, image, motion))
    if kind == "resolve":
        return _exact_resolve(history, current, motion)
    given = _motion_field(_generator(seed + 1), h, w)
    return dict(motion=motion, resolved=_exact_resolve(history, current, given))
