"""The work that users of this rasterizer have it do, for timing and for comparing results.

Each case is one pass through the public entry points of paper_1908_02681_gb300.pcr: frames along a camera
path, a key buffer for later depth queries, batched views replayed from a graph, a burst of served requests, a
frame from host memory, the per-point projection. The scenes follow this repository's generators (a uniform
cube; scanned terrain with box buildings over 1 km, and a 10 km city seen from street level), made here on the
GPU from the seed. All results are whole numbers and are compared exactly.
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_1908_02681_gb300 import pcr

BACKGROUND = 0xFF301810
EPS = (1, 100)  # the band of high-quality splatting: 1 % of linear depth
LINEAR, METRIC, PIECEWISE = pcr.PCR_DEPTH_LINEAR, pcr.PCR_DEPTH_METRIC, pcr.PCR_DEPTH_PIECEWISE
# nanometres to 10 m, micrometres to 10 km, millimetres beyond
RANGES = ((0.0, 10.0, 1e9), (10.0, 10010.0, 1e6), (10010.0, 1010010.0, 1e3))


# ------------------------------------------------------------------------------------------------- the cases

def listed():
    return [
        # someone turns a small scan in a viewer: four frames, the camera moved before each
        {"name": "path_40k_320x240", "kind": "path", "cloud": "lidar", "n": 40_001, "order": "scan", "views": 4,
         "w": 320, "h": 240, "hq": False, "depth": LINEAR},
        # the unit cube at 640 x 480: one small frame from a fixed camera
        {"name": "cube_1m_640x480", "kind": "path", "cloud": "cube", "n": 1_000_000, "order": "scan", "views": 1,
         "w": 640, "h": 480, "hq": False, "depth": LINEAR},
        # a turntable of a few million points in a window of odd size, high-quality, millimetre depth codes
        {"name": "path_2m7_1013x771_hq_mm", "kind": "path", "cloud": "lidar", "n": 2_700_001, "order": "scan",
         "views": 3, "w": 1013, "h": 771, "hq": True, "depth": METRIC},
        # an ordinary scan at full HD that arrives in pinned host memory, high-quality, images back to the host
        {"name": "host_20m_1080p_hq", "kind": "host", "cloud": "lidar", "n": 20_000_000, "order": "scan", "views": 1,
         "w": 1920, "h": 1080, "hq": True, "depth": LINEAR},
        # the benchmark's frame: 100M scanned points, basic and high-quality images
        {"name": "lidar_100m_1080p_hq", "kind": "path", "cloud": "lidar", "n": 100_000_000, "order": "scan",
         "views": 1, "w": 1920, "h": 1080, "hq": True, "depth": LINEAR},
        # merged scans whose points come in no order, high-quality
        {"name": "shuffled_37m_1600x900_hq", "kind": "path", "cloud": "lidar", "n": 37_000_003, "order": "shuffled",
         "views": 1, "w": 1600, "h": 900, "hq": True, "depth": LINEAR},
        # a city from street level at 4K, most of it outside the view; the keys are kept for depth queries
        {"name": "city_400m_4k_keys", "kind": "keys", "cloud": "city", "n": 400_000_000, "order": "scan", "views": 1,
         "w": 3840, "h": 2160, "hq": False, "depth": LINEAR},
        # depth at nanometres near the eye and micrometres farther out
        {"name": "piecewise_50m_720p_keys", "kind": "keys", "cloud": "lidar", "n": 50_000_000, "order": "scan",
         "views": 1, "w": 1280, "h": 720, "hq": False, "depth": PIECEWISE},
        # 16 cameras around one resident cloud, mixed resolutions, a captured frame with new views each time
        {"name": "batch_16v_20m", "kind": "batch", "cloud": "lidar", "n": 20_000_000, "order": "scan", "views": 16,
         "w": 0, "h": 0, "hq": False, "depth": LINEAR},
        # the same, high-quality, a smaller cloud
        {"name": "batch_12v_6m_hq", "kind": "batch", "cloud": "lidar", "n": 6_000_037, "order": "scan", "views": 12,
         "w": 0, "h": 0, "hq": True, "depth": LINEAR},
        # a burst of requests to a server: 720p to 4K, 70 % basic and 30 % high-quality
        {"name": "serve_20_requests_10m", "kind": "serve", "cloud": "lidar", "n": 10_000_000, "order": "scan",
         "views": 20, "w": 0, "h": 0, "hq": False, "depth": LINEAR},
        # every point's own pixel and key (picking, visibility queries)
        {"name": "project_6m_1080p", "kind": "project", "cloud": "lidar", "n": 6_000_011, "order": "scan", "views": 1,
         "w": 1920, "h": 1080, "hq": False, "depth": LINEAR},
    ]


def _log_between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["path", "path", "path", "keys", "batch", "serve", "host", "project"])
    w, h = _log_between(rng, 200, 3840), _log_between(rng, 150, 2160)
    depth = rng.choice([LINEAR, LINEAR, METRIC])
    case = {"kind": kind, "cloud": "lidar", "order": rng.choice(["scan", "scan", "scan", "shuffled"]), "views": 1,
            "w": w, "h": h, "hq": rng.random() < 0.5, "depth": depth}
    if kind == "path":
        case["views"] = rng.randint(1, 4)
        case["n"] = _log_between(rng, 20_000, 100_000_000 // case["views"])
        case["cloud"] = rng.choice(["lidar", "lidar", "cube"])
    elif kind == "keys":
        case["n"] = _log_between(rng, 100_000, 200_000_000)
        case["cloud"] = rng.choice(["lidar", "city"])
        case["hq"] = False
        case["depth"] = rng.choice([LINEAR, METRIC, PIECEWISE])
    elif kind == "batch":
        case["views"] = rng.randint(2, 24)
        case["n"] = _log_between(rng, 200_000, 240_000_000 // case["views"])
    elif kind == "serve":
        case["views"] = rng.randint(4, 24)
        case["n"] = _log_between(rng, 200_000, 120_000_000 // case["views"])
        case["hq"] = False  # each request says for itself
    elif kind == "host":
        case["n"] = _log_between(rng, 100_000, 30_000_000)
    else:
        case["n"] = _log_between(rng, 100_000, 60_000_000)
        case["hq"] = False
        case["depth"] = rng.choice([LINEAR, METRIC, PIECEWISE])
    return case


# ------------------------------------------------------------------------------------------ points and cameras

CHUNK = 1 << 23


def _ramp(t):
    """Height ramp colours (dark blue, green, yellow, red, white) of t in [0, 1] as RGBA8 words."""
    stops = torch.tensor([[26, 38, 115], [38, 140, 51], [230, 217, 64], [204, 64, 38], [247, 247, 247]],
                         dtype=torch.float32, device=t.device)
    s = t.float().clamp(0, 1) * 4
    k = s.long().clamp(max=3)
    c = torch.lerp(stops[k], stops[k + 1], (s - k).unsqueeze(1)).round().to(torch.int32)
    return c[:, 0] | (c[:, 1] << 8) | (c[:, 2] << 16) | (-1 << 24)


class _Scene:
    """Sin-sum terrain with axis-aligned box buildings; city: ten times as wide, with street-level detail."""

    def __init__(self, city, rnd):
        self.city = city
        self.lo, self.hi = (-5000.0, 5000.0) if city else (0.0, 1000.0)
        amp, wav = (0.25, 10.0) if city else (1.0, 1.0)
        self.waves = [(a * amp, lam * wav, rnd.uniform(0, 2 * math.pi), rnd.uniform(0, 2 * math.pi))
                      for a, lam in zip((40, 20, 10, 5, 2.5, 1.25), (500, 250, 120, 60, 30, 15))]
        boxes = []
        for _ in range(8000 if city else 200):
            fx, fy, hh = rnd.uniform(10, 40), rnd.uniform(10, 40), rnd.uniform(5, 60)
            cx = rnd.uniform(self.lo + fx / 2, self.hi - fx / 2)
            cy = rnd.uniform(self.lo + fy / 2, self.hi - fy / 2)
            if city and math.hypot(cx, cy) < 30 + (fx + fy) / 2:
                continue  # the eye's own street stays free
            boxes.append((cx, cy, fx, fy, self.height(cx, cy), hh))
        self.boxes = torch.tensor(boxes, dtype=torch.float64, device="cuda")

    def height(self, x, y):
        sin = torch.sin if torch.is_tensor(x) else math.sin
        return sum(a * sin(x * (2 * math.pi / lam) + p) * sin(y * (2 * math.pi / lam) + q)
                   for a, lam, p, q in self.waves)


def _scene_points(scene, n, gen, out):
    """Terrain in 1-m strips along y (alternating direction), then building by building, then the street."""
    def uni(m):
        return torch.rand(m, generator=gen, dtype=torch.float64, device="cuda")

    lo, size = scene.lo, scene.hi - scene.lo
    n_street = n // 50 if scene.city else 0
    b = scene.boxes
    roof, wall = b[:, 2] * b[:, 3], 2 * (b[:, 2] + b[:, 3]) * b[:, 5]
    area = torch.cat([torch.tensor([size * size], dtype=torch.float64, device="cuda"), roof + wall])
    first = (torch.cumsum(area, 0) / area.sum() * (n - n_street)).long()  # last index + 1 of terrain, box 0, ...
    n_terrain = int(first[0])
    strips = int(size)
    amp = sum(a for a, _, _, _ in scene.waves)
    for i0 in range(0, n, CHUNK):
        m = min(CHUNK, n - i0)
        i = torch.arange(i0, i0 + m, device="cuda")
        u, v = uni(m), uni(m)
        # terrain
        pos = i.double() * (strips / max(n_terrain, 1))
        k = pos.floor()
        along = (pos - k)
        x = lo + size * torch.where(k.long() % 2 == 1, 1 - along, along)
        y = lo + k + u
        if i0 + m > n_terrain and len(b):
            box = torch.searchsorted(first, i, right=True).clamp(1, len(b)) - 1
            cx, cy, fx, fy, base, hh = (b[box, j] for j in range(6))
            rf, wl = roof[box], wall[box]
            sel = uni(m) * (rf + wl)
            s = (sel - rf) / wl * 2 * (fx + fy)
            wx = torch.where(s < fx, s, torch.where(s < fx + fy, fx, torch.where(s < 2 * fx + fy, 2 * fx + fy - s,
                                                                                 torch.zeros_like(s))))
            wy = torch.where(s < fx, torch.zeros_like(s), torch.where(s < fx + fy, s - fx, torch.where(
                s < 2 * fx + fy, fy, 2 * (fx + fy) - s)))
            on_roof, building = sel < rf, (i >= n_terrain) & (i < n - n_street)
            x = torch.where(building, cx + torch.where(on_roof, (u - 0.5) * fx, wx - fx / 2), x)
            y = torch.where(building, cy + torch.where(on_roof, (v - 0.5) * fy, wy - fy / 2), y)
            if n_street:
                street, r, th = i >= n - n_street, 20 * torch.sqrt(u), 2 * math.pi * v
                x = torch.where(street, r * torch.cos(th), x)
                y = torch.where(street, r * torch.sin(th), y)
            z = scene.height(x, y)
            z = torch.where(building, base + torch.where(on_roof, hh, v * hh), z)
        else:
            z = scene.height(x, y)
        xyz = torch.stack([x, y, z], 1)
        xyz += 0.01 * torch.randn(xyz.shape, generator=gen, dtype=torch.float64, device="cuda")  # 1 cm noise
        out[i0:i0 + m, :3] = xyz.float().view(torch.int32)
        out[i0:i0 + m, 3] = _ramp((z + amp) / (2 * amp + 60))


def _points(case, seed):
    n = case["n"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    out = torch.empty((n, 4), dtype=torch.int32, device="cuda")
    if case["cloud"] == "cube":
        for i0 in range(0, n, CHUNK):
            m = min(CHUNK, n - i0)
            out[i0:i0 + m, :3] = (torch.rand((m, 3), generator=gen, device="cuda") - 0.5).view(torch.int32)
            out[i0:i0 + m, 3] = torch.randint(0, 1 << 24, (m,), generator=gen, device="cuda").int() | (-1 << 24)
        return out
    _scene_points(_Scene(case["cloud"] == "city", random.Random(seed)), n, gen, out)
    if case["order"] == "shuffled":
        out = out[torch.randperm(n, generator=gen, device="cuda")]
    return out


def _view(eye, target, up, width, height, near, far, depth):
    """An OpenGL-style camera: fov 60 degrees, row-major view-projection."""
    eye, target, up = (np.asarray(a, dtype=np.float64) for a in (eye, target, up))
    f = target - eye
    f /= math.sqrt(f @ f)
    s = np.cross(f, up)
    s /= math.sqrt(s @ s)
    u = np.cross(s, f)
    look = np.eye(4)
    for r, a in enumerate((s, u, -f)):
        look[r, :3], look[r, 3] = a, -(a @ eye)
    t = 1 / math.tan(math.radians(60) / 2)
    proj = np.zeros((4, 4))
    proj[0, 0], proj[1, 1] = t * height / width, t
    proj[2, 2], proj[2, 3], proj[3, 2] = (far + near) / (near - far), 2 * far * near / (near - far), -1.0
    v = SimpleNamespace(view_proj=proj @ look, near=near, far=far, width=width, height=height, depth_mode=depth,
                        metric_scale=1000.0)
    if depth == PIECEWISE:
        v.ranges = RANGES
    return v


def _views(case, seed):
    rnd = random.Random(seed * 7919 + 1)
    w, h, depth = case["w"], case["h"], case["depth"]
    jit = [rnd.uniform(-1, 1) for _ in range(3)]
    if case["kind"] in ("batch", "serve"):  # seeded orbit poses
        sizes = (((640, 480), (1920, 1080), (3840, 2160)) if case["kind"] == "batch" else
                 ((1280, 720), (1920, 1080), (2560, 1440), (3840, 2160)))
        views = []
        for i in range(case["views"]):
            az, el = rnd.uniform(0, 2 * math.pi), math.radians(rnd.uniform(15, 75))
            rad = rnd.uniform(300, 1500)
            t = np.array([500 + rnd.uniform(-100, 100), 500 + rnd.uniform(-100, 100), 0.0])
            eye = t + rad * np.array([math.cos(el) * math.cos(az), math.cos(el) * math.sin(az), math.sin(el)])
            views.append(_view(eye, t, (0, 0, 1), *sizes[i % len(sizes)], 0.1, 3000.0, depth))
        return views
    if case["cloud"] == "cube":
        return [_view((0.3 * i + 0.02 * jit[0], 0.02 * jit[1], 3.0), (0, 0, 0), (0, 1, 0), w, h, 0.1, 10.0, depth)
                for i in range(case["views"])]
    if case["cloud"] == "city":  # 1.7 m above the street
        z = _Scene(True, random.Random(seed)).height(0.0, 0.0) + 1.7
        return [_view((0, 0, z), (100.0, 37.0 + jit[0], z), (0, 0, 1), w, h, 0.01, 10000.0, depth)]
    return [_view((-150 + 12 * i + jit[0], -150 - 9 * i + jit[1], 350 + jit[2]), (500, 500, 0), (0, 0, 1), w, h, 0.1,
                  3000.0, depth) for i in range(case["views"])]


def _serve_modes(case, seed):
    rnd = random.Random(seed * 31 + 5)
    return [rnd.random() < 0.3 for _ in range(case["views"])]


# ------------------------------------------------------------------------------------------ preparing, running

def _images(n, case):
    return [torch.zeros(case["w"] * case["h"], dtype=torch.int32, device="cuda") for _ in range(n)]


def prepare(case, seed):
    kind, hq = case["kind"], case["hq"]
    pts, views = _points(case, seed), _views(case, seed)
    st = SimpleNamespace(case=case, pts=pts, views=views)
    flags = pcr.PCR_FB_HQ if hq else 0
    if kind in ("path", "keys"):
        st.fb = pcr.pcr_create_framebuffer(case["w"], case["h"], flags)
        if kind == "keys":
            st.keys = pcr.pcr_framebuffer_keys(st.fb)[0]
        else:
            st.basic, st.hq = _images(len(views), case), _images(len(views) if hq else 0, case)
    elif kind == "batch":
        st.cloud = pcr.pcr_cloud_create(pts)
        st.fbs = [pcr.pcr_create_framebuffer(v.width, v.height, flags) for v in views]
        st.outs = [torch.zeros(v.width * v.height, dtype=torch.int32, device="cuda") for v in views]
        st.batch = pcr.pcr_batch_create(st.cloud, st.fbs, st.outs, hq, *EPS, BACKGROUND, True)
        pcr.pcr_batch_set_views(st.batch, views)
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        pcr.pcr_batch_capture(st.batch, side)
        torch.cuda.current_stream().wait_stream(side)
    elif kind == "serve":
        torch.cuda.synchronize()  # the server's streams do not wait for the one that made the points
        st.server = pcr.pcr_server_create(streams=4, max_batch_views=16, framebuffer_budget_bytes=4 << 30)
        cid = pcr.pcr_server_add_cloud(st.server, pts)
        st.outs = [torch.zeros(v.width * v.height, dtype=torch.int32, device="cuda") for v in views]
        st.requests = [{"cloud": cid, "view": v, "out": o, "hq": q, "background_rgba": BACKGROUND}
                       for v, o, q in zip(views, st.outs, _serve_modes(case, seed))]
        torch.cuda.synchronize()
    elif kind == "host":
        st.h_pts = pts.cpu().pin_memory()
        st.fb = pcr.pcr_create_framebuffer(case["w"], case["h"], flags)
        st.d_pts = torch.empty_like(pts)
        st.d_images = torch.empty(2 * case["w"] * case["h"], dtype=torch.int32, device="cuda")
        st.h_images = [torch.zeros(case["w"] * case["h"], dtype=torch.int32).pin_memory() for _ in range(2 if hq else 1)]
        del st.pts
    elif kind == "project":
        st.pixel = torch.empty(case["n"], dtype=torch.int32, device="cuda")
        st.key = torch.empty(case["n"], dtype=torch.int64, device="cuda")
    return st


def run(st):
    kind, hq = st.case["kind"], st.case["hq"]
    if kind == "path":
        for i, v in enumerate(st.views):
            if hq:
                pcr.pcr_render_hq_splat(st.fb, st.pts, v, *EPS)
                pcr.pcr_resolve_both(st.fb, st.basic[i], st.hq[i], BACKGROUND)
            else:
                pcr.pcr_render_atomicmin(st.fb, st.pts, v)
                pcr.pcr_resolve(st.fb, st.basic[i], BACKGROUND, clear_after=True)
        return st.basic + st.hq
    if kind == "keys":
        pcr.pcr_clear(st.fb)
        pcr.pcr_render_atomicmin(st.fb, st.pts, st.views[0])
        return st.keys
    if kind == "batch":
        pcr.pcr_batch_set_views(st.batch, st.views)
        pcr.pcr_batch_launch(st.batch)
        return st.outs
    if kind == "serve":
        left = len(pcr.pcr_server_submit_many(st.server, st.requests))
        while left:
            for c in pcr.pcr_server_poll(st.server, wait_ms=1000):
                if c["status"] != pcr.PCR_OK:
                    raise RuntimeError(f"request {c['id']}: {pcr.pcr_status_string(c['status'])}")
                left -= 1
        return st.outs
    if kind == "host":
        pcr.pcr_render_frame_host(st.fb, st.h_pts, st.views[0], st.d_pts, st.d_images, st.h_images[0],
                                  st.h_images[1] if hq else None, *EPS, BACKGROUND)
        return st.h_images
    return pcr.pcr_project_points(st.pts, st.views[0], st.pixel, st.key)


def work(case):
    """Each point read once and each image, key or fragment written once; 32 operations per point and view (three
    clip rows, the division, pixel, depth code) and 6 more for the band test and sums."""
    n, v = case["n"], case["views"]
    if case["kind"] in ("batch", "serve"):
        px = sum(x.width * x.height for x in _views(case, 0))
        out = 4 * px
    else:
        out = case["w"] * case["h"] * v * (8 if case["kind"] == "keys" else 4 * (2 if case["hq"] else 1))
        if case["kind"] == "project":
            out = 12 * n
    reads = v if case["kind"] == "path" else 1  # each frame of a path is a call of its own
    return {"bytes": 16 * n * reads + out, "flops": (38 if case["hq"] else 32) * n * v}


def tolerance(case):
    return "exact"  # images, keys and pixels are whole numbers, fixed by the definition


# --------------------------------------------------------------------------------- the definition in 64 bits

def _fma(a, x, c):
    """a * x + c rounded once to 64 bits: a a Python double, x a tensor of float32 values held as doubles, c a
    double or tensor. The product is two exact doubles (a split in halves of 26 and 27 bits); their sum with c is
    rounded through one odd-rounded intermediate, as Boldo and Melquiond (2008) prove correct."""
    g = a * 134217729.0
    hi = g - (g - a)
    p, q = x * hi, x * (a - hi)
    s = p + q
    t = s - p
    r = (p - (s - t)) + (q - t)  # s + r = a * x exactly
    u = s + c
    t = u - s
    e = (s - (u - t)) + (c - t)  # u + e = s + c exactly
    v = r + e
    t = v - r
    f = (r - (v - t)) + (e - t)  # v + f = r + e exactly
    bits = v.view(torch.int64)
    even = (bits & 1) == 0
    step = torch.where((f > 0) == (v > 0), 1, -1)
    odd = torch.where((f != 0) & even, bits + step, bits).view(torch.float64)
    return u + odd


def _project(pts, view):
    """Per point: the pixel (-1 when culled) and the depth code."""
    xyz = pts[:, :3].contiguous().view(torch.float32).double()
    x, y, z = xyz[:, 0], xyz[:, 1], xyz[:, 2]
    m = [[float(a) for a in row] for row in view.view_proj]
    cx, cy, w = (_fma(m[r][2], z, _fma(m[r][1], y, _fma(m[r][0], x, torch.full_like(x, m[r][3])))) for r in (0, 1, 3))
    near, far, width, height = view.near, view.far, view.width, view.height
    ok = (w >= near) & (w < far)
    fw = w.float()
    fx = ((cx.float() / fw) * 0.5 + 0.5) * float(width)
    fy = ((cy.float() / fw) * 0.5 + 0.5) * float(height)
    ok &= (fx >= 0) & (fx < width) & (fy >= 0) & (fy < height)
    if view.depth_mode == LINEAR:
        t = (w - near) * (1099511627776.0 / (far - near))
    elif view.depth_mode == METRIC:
        t = w * view.metric_scale
    else:
        t, base, inside = torch.zeros_like(w), 0.0, torch.zeros_like(ok)
        for lo, hi, res in view.ranges:
            here = (w >= lo) & (w < hi)
            t = torch.where(here, base + torch.floor((w - lo) * res), t)
            inside |= here
            base += math.ceil((hi - lo) * res)
        ok &= inside
    q = torch.floor(torch.where(ok, t, torch.zeros_like(t))).clamp(max=float((1 << 40) - 2)).long()
    pix = torch.where(ok, fy.nan_to_num(0).clamp(0, height).long() * width + fx.nan_to_num(0).clamp(0, width).long(),
                      torch.full_like(q, -1))
    return pix, q


def _parts(pts, view):
    for i0 in range(0, len(pts), CHUNK):
        p = pts[i0:i0 + CHUNK]
        yield (p[:, 3].long() & 0xFFFFFF, *_project(p, view))


SIGN = -(1 << 63)


def _keys(pts, view):
    """The smallest key of each pixel, as int64 bit patterns of unsigned words (-1: empty)."""
    keys = torch.full((view.width * view.height,), -1 ^ SIGN, dtype=torch.int64, device=pts.device)
    for rgb, pix, q in _parts(pts, view):
        vis = pix >= 0
        keys.scatter_reduce_(0, pix[vis], ((q << 24) | rgb)[vis] ^ SIGN, "amin")
    return keys ^ SIGN


def _signed(x):
    return x - (1 << 32) if x >= 1 << 31 else x


def _basic_image(keys):
    rgba = torch.where(keys == -1, _signed(BACKGROUND), (keys & 0xFFFFFF) | (-1 << 24))
    return rgba.to(torch.int32)


def _hq_image(pts, view, keys):
    nq = math.floor(view.near * (1099511627776.0 / (view.far - view.near))) if view.depth_mode == LINEAR else 0
    qmin = (keys >> 24) & ((1 << 40) - 1)
    sums = torch.zeros((4, len(keys)), dtype=torch.int64, device=pts.device)
    num, den = EPS
    for rgb, pix, q in _parts(pts, view):
        vis = pix >= 0
        rgb, pix, q = rgb[vis], pix[vis], q[vis]
        near = qmin[pix]
        take = den * (q - near) <= num * (near + nq)
        rgb, pix = rgb[take], pix[take]
        for c in range(3):
            sums[c].index_add_(0, pix, (rgb >> (8 * c)) & 255)
        sums[3].index_add_(0, pix, torch.ones_like(pix))
    n = sums[3].clamp(min=1)
    r, g, b = ((sums[c] + sums[3] // 2) // n for c in range(3))
    return torch.where(sums[3] == 0, _signed(BACKGROUND), r | (g << 8) | (b << 16) | (-1 << 24)).to(torch.int32)


def exact(case, seed):
    kind = case["kind"]
    pts, views = _points(case, seed), _views(case, seed)
    if kind == "project":
        pix, key = [], []
        for rgb, p, q in _parts(pts, views[0]):
            pix.append(p.int())
            key.append(torch.where(p >= 0, (q << 24) | rgb, torch.full_like(q, -1)))
        return torch.cat(pix), torch.cat(key)
    if kind == "keys":
        return _keys(pts, views[0])
    if kind in ("batch", "serve"):
        modes = _serve_modes(case, seed) if kind == "serve" else [case["hq"]] * len(views)
        return [_hq_image(pts, v, k) if q else _basic_image(k) for v, q in zip(views, modes) for k in [_keys(pts, v)]]
    basic, hq = [], []
    for v in views:
        keys = _keys(pts, v)
        basic.append(_basic_image(keys))
        if case["hq"]:
            hq.append(_hq_image(pts, v, keys))
    out = basic + hq
    return [o.cpu() for o in out] if kind == "host" else out
