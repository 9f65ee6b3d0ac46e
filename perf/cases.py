"""Performance cases of the library: what its users have it do, over the sizes they do it at.

Every case goes through the public entry points of paper_1711_07793_gb300 (api and surrogate).  The scenes are those
of the repository's workloads in kind and proportion (rotated rectangles, tilted fence bars and spheres over a ground
plane, a perspective camera over a window of the ground), drawn here with torch on the GPU so that fresh inputs are
quick to make.

Kinds of case
  single    rbsm_visibility / rsmss_filter: one shadow map, one set of fragments (a renderer with one light)
  batch     rbsm_batch_run: several maps and views in one launch (cascades, several lights, frames)
  gbuffer   rbsm_visibility_gbuffer: fragments projected from depth buffers (a deferred renderer)
  rpcf      rbsm_rpcf: PCF over the filtered answer
  light     rbsm_shadow_maps: the light pass from analytic occluders
  learned   rbsm_batch_run with the guarded surrogate
  train     Surrogate.train_step: one minibatch of surrogate training
  host      Stager.run: maps, fragments and answers in page-locked host memory
"""
import math
import os
import random

import numpy as np
import torch

from paper_1711_07793_gb300 import api
from paper_1711_07793_gb300 import surrogate as sg

DEV = "cuda"
PACKAGE = os.path.dirname(os.path.abspath(api.__file__))
CHECKPOINT = os.path.join(PACKAGE, "weights", "surrogate_c4.npz")
GUARD_TAU = 0.01            # the guard the committed checkpoint's error bound is stated for
RECEIVER_OFFSET = 1e-3      # fragments on a sphere lie this far in front of the stored depth
SILHOUETTE, FILTER, BOTH = 1, 2, 3


# ------------------------------------------------------------------ cases --

def _case(name, kind, **kw):
    c = {"kind": kind, "scene": "fence", "map_w": 1024, "map_h": 1024, "screen_w": 640, "screen_h": 360, "frames": 1,
         "mode": BOTH, "codes": False, "texture": True, "shift": 0, "max_dist": 16, "k": 0, "batch": 0}
    unknown = set(kw) - set(c)
    assert not unknown, unknown
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest scene (320x240 over a 256^2 map): a call whose latency counts, on a map without a texture.
        _case("filter_320x240", "single", scene="rects", map_w=256, map_h=256, screen_w=320, screen_h=240, mode=FILTER,
              texture=False),
        # Odd sizes, planes off the 16-byte grid, codes asked for: a debug view, or a compacted list of fragments.
        _case("visibility_odd_codes", "single", map_w=1531, map_h=997, screen_w=1277, screen_h=719, mode=SILHOUETTE,
              codes=True, texture=False, shift=1),
        # Hard shadows of a 1080p frame.
        _case("visibility_1080p", "single", map_w=2048, map_h=2048, screen_w=1920, screen_h=1080, mode=SILHOUETTE),
        # Soft shadows of a 4K frame.
        _case("filter_4k", "single", map_w=4096, map_h=4096, screen_w=3840, screen_h=2160, mode=FILTER),
        # Cascades: 4 lights x 4 cascades (4096^2 .. 512^2) against views of uneven size, one job per view, light and
        # cascade (64 jobs, both answers).
        _case("batch_cascades", "batch", scene="cascades", map_w=4096, map_h=4096, screen_w=3840, screen_h=2160,
              frames=4),
        # A moving light: 8 frames of 3840x2160 fragments on 8192^2 maps in one launch (the benchmark's workload, a
        # quarter of its frames).
        _case("batch_frames_4k", "batch", scene="mixed", map_w=8192, map_h=8192, screen_w=3840, screen_h=2160,
              frames=8),
        # The same frames from depth buffers.
        _case("gbuffer_4k", "gbuffer", scene="mixed", map_w=8192, map_h=8192, screen_w=3840, screen_h=2160, frames=4),
        # PCF over the filtered answer, 3x3 samples.
        _case("rpcf3_4k", "rpcf", scene="mixed", map_w=8192, map_h=8192, screen_w=3840, screen_h=2160, mode=FILTER,
              k=3),
        # The light pass of four frames.
        _case("light_8192", "light", scene="mixed", map_w=8192, map_h=8192, frames=4),
        # The guarded surrogate on a 4K frame.
        _case("learned_4k", "learned", map_w=4096, map_h=4096, screen_w=3840, screen_h=2160, mode=FILTER),
        # A training step of the surrogate at the trainer's minibatch.
        _case("train_8192", "train", batch=8192),
        # A 1080p frame whose inputs and answers are in host memory.
        _case("host_1080p", "host", map_w=2048, map_h=2048, screen_w=1920, screen_h=1080, texture=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges, sizes log-uniform, odd ones among them."""
    kind = rng.choice(["single", "single", "single", "batch", "batch", "gbuffer", "gbuffer", "rpcf", "rpcf", "light",
                       "learned", "train", "host"])
    odd = rng.random() < 0.3
    size = _log(rng, 256, 8192)
    mw = size if odd else max(256, size // 64 * 64)
    mh = max(200, int(mw * rng.uniform(0.5, 1.0))) if odd else mw
    sw = _log(rng, 320, 3840)
    sh = max(100, int(sw * rng.choice([0.5625, 0.75, 0.4219])))
    if not odd:
        sw, sh = max(320, sw // 16 * 16), max(100, sh // 4 * 4)
    kw = dict(scene=rng.choice(["rects", "fence", "mixed"]), map_w=mw, map_h=mh, screen_w=sw, screen_h=sh,
              texture=rng.random() < 0.7, max_dist=rng.choice([8, 16, 16, 16, 32, 64]))
    if kind == "single":
        return _case(None, kind, mode=rng.choice([SILHOUETTE, FILTER]), codes=rng.random() < 0.3,
                     shift=1 if odd and rng.random() < 0.5 else 0, **kw)
    if kind == "batch":
        if rng.random() < 0.4:
            kw["scene"] = "cascades"
            kw["map_w"] = kw["map_h"] = max(512, mw // 64 * 64 // 2)
        return _case(None, kind, mode=rng.choice([SILHOUETTE, FILTER, BOTH, BOTH]), codes=rng.random() < 0.25,
                     frames=rng.randint(1, 4), **kw)
    if kind == "gbuffer":
        return _case(None, kind, mode=rng.choice([SILHOUETTE, FILTER, BOTH]), codes=rng.random() < 0.25,
                     frames=rng.randint(1, 4), **kw)
    if kind == "rpcf":
        return _case(None, kind, mode=FILTER, k=rng.choice([1, 3, 3, 5, 7]), **kw)
    if kind == "light":
        return _case(None, kind, scene=kw["scene"], map_w=mw, map_h=mh, frames=rng.randint(1, 4))
    if kind == "learned":
        kw["max_dist"] = 16
        return _case(None, kind, mode=FILTER, **kw)
    if kind == "train":
        return _case(None, kind, batch=_log(rng, 256, 65536))
    kw.update(texture=False, screen_w=min(sw, 1920), screen_h=min(sh, 1080), map_w=min(mw, 2048), map_h=min(mh, 2048))
    return _case(None, kind, frames=rng.randint(1, 3), **kw)


# ----------------------------------------------------------------- scenes --

def _axis(r, max_deg=180.0):
    a = math.radians(r.uniform(-max_deg, max_deg))
    return math.sin(a), math.cos(a)


def _rects(r, n, w, h, lo, hi, d_lo, d_hi):
    out = []
    for _ in range(n):
        ux, uy = _axis(r)
        out.append((r.uniform(0, w), r.uniform(0, h), ux, uy, r.uniform(lo, hi) / 2, r.uniform(lo, hi) / 2,
                    float(np.float32(r.uniform(d_lo, d_hi)))))
    return out


def _bars(r, n, w, h, w_lo, w_hi, l_lo, l_hi):
    out = []
    for _ in range(n):
        ux, uy = _axis(r, 30.0)
        out.append((r.uniform(0, w), r.uniform(0, h), ux, uy, r.uniform(l_lo, l_hi) / 2, r.uniform(w_lo, w_hi) / 2,
                    float(np.float32(r.uniform(0.05, 0.2)))))
    return out


def _spheres(r, n, w, h, lo, hi):
    out = []
    for _ in range(n):
        rad = r.uniform(lo, hi)
        out.append((r.uniform(0, w), r.uniform(0, h), rad, r.uniform(0.4, 0.8)))
    return out


def _occluders(scene, r, w, h):
    """(rects (cx cy ux uy ha hb depth), spheres (cx cy radius centre-depth)), in proportion to the map's size."""
    size = max(w, h)
    if scene == "rects":
        return _rects(r, 24, w, h, size / 32, size / 4, 0.2, 0.8), []
    if scene == "fence":
        s = size / 2048.0
        n = 80 if size >= 4096 else 40
        return _bars(r, n, w, h, max(1.0, s), 6 * s + 1, 256 * s, 2048 * s), _spheres(r, n * 3 // 4, w, h, 10 * s, 120 * s)
    s = size / 8192.0
    rects = _rects(r, 70, w, h, 64 * s, 512 * s, 0.2, 0.8) + _bars(r, 70, w, h, max(1.0, 2 * s), 24 * s + 1, 1024 * s,
                                                                   8192 * s)
    return rects, _spheres(r, 60, w, h, 40 * s, 480 * s)


def _shifted(occ, du):
    """The light moves: every occluder shifts along u by its height."""
    rects, spheres = occ
    return ([(c[0] + du * (1.0 - c[6]),) + c[1:] for c in rects], [(c[0] + du * (1.0 - c[3]),) + c[1:] for c in spheres])


def _box(c0, c1, n):
    return max(0, min(n, int(math.floor(c0)) - 1)), max(0, min(n, int(math.ceil(c1)) + 1))


def _raster(occ, depth, zscale, dtype=torch.float32):
    """The smallest depth of the occluders covering each texel centre, else 1 (the ground), into `depth`."""
    rects, spheres = occ
    h, w = depth.shape
    depth.fill_(1.0)
    ic = torch.arange(w, device=DEV, dtype=dtype) + 0.5
    jc = (torch.arange(h, device=DEV, dtype=dtype) + 0.5)[:, None]
    for cx, cy, ux, uy, ha, hb, d in rects:
        ex, ey = abs(ux) * ha + abs(uy) * hb, abs(uy) * ha + abs(ux) * hb
        i0, i1 = _box(cx - ex, cx + ex, w)
        j0, j1 = _box(cy - ey, cy + ey, h)
        if i0 >= i1 or j0 >= j1:
            continue
        px, py = ic[i0:i1] - cx, jc[j0:j1] - cy
        inside = ((px * ux + py * uy).abs() <= ha) & (((-px) * uy + py * ux).abs() <= hb)
        sub = depth[j0:j1, i0:i1]
        sub.copy_(torch.where(inside & (sub > d), d, sub))
    for cx, cy, rad, c in spheres:
        i0, i1 = _box(cx - rad, cx + rad, w)
        j0, j1 = _box(cy - rad, cy + rad, h)
        if i0 >= i1 or j0 >= j1:
            continue
        dx, dy = ic[i0:i1] - cx, jc[j0:j1] - cy
        left = rad * rad - (dx * dx + dy * dy)
        cap = (c - left.clamp_min(0).sqrt() / zscale).to(depth.dtype)
        sub = depth[j0:j1, i0:i1]
        sub.copy_(torch.where((left >= 0) & (cap < sub), cap, sub))
    return depth


def _map(occ, w, h, zscale, texture):
    """A shadow map as a program keeps it: rows padded to 128 bytes where a texture reads it, else dense."""
    pitch = (w + 31) // 32 * 32 if texture else w
    return _raster(occ, torch.empty((h, pitch), dtype=torch.float32, device=DEV)[:, :w], zscale)


def _camera(r, w, h, zoom=(0.2, 0.4)):
    """3x3 homography from the unit screen to texels: a randomly turned trapezoid whose far edge is twice as wide."""
    side = r.uniform(*zoom) * min(w, h)
    half = side / 2
    reach = half * math.sqrt(2.0)
    cx, cy = r.uniform(reach, w - reach), r.uniform(reach, h - reach)
    ux, uy = _axis(r)
    wrow = np.array([0.0, 1.0, 1.0])                         # w = 1 + v
    xl, yl = np.array([side, 0.0, -half]), np.array([0.0, 3 * half, -half])
    return np.stack([cx * wrow + ux * xl - uy * yl, cy * wrow + uy * xl + ux * yl, wrow])


def _pixels(hom, sw, sh):
    """The homography over pixel indices (px + 1/2, py + 1/2, 1)."""
    return hom * np.array([1.0 / sw, 1.0 / sh, 1.0])


def _fragments(hom, sw, sh, w, h, spheres, zscale):
    """Light-space planes (x, y, z) of every pixel: the ground at depth 1, or the nearest sphere under it."""
    m = _pixels(hom, sw, sh)
    u = torch.arange(sw, device=DEV, dtype=torch.float64) + 0.5
    v = (torch.arange(sh, device=DEV, dtype=torch.float64) + 0.5)[:, None]
    ww = m[2, 0] * u + m[2, 1] * v + m[2, 2]
    X = ((m[0, 0] * u + m[0, 1] * v + m[0, 2]) / ww).reshape(-1)
    Y = ((m[1, 0] * u + m[1, 1] * v + m[1, 2]) / ww).reshape(-1)
    z = torch.full((sw * sh,), 2.0, dtype=torch.float32, device=DEV)
    Xf, Yf = X.float(), Y.float()
    lo_x, hi_x, lo_y, hi_y = (float(t) for t in (Xf.min(), Xf.max(), Yf.min(), Yf.max()))
    for cx, cy, rad, c in spheres:
        if cx + rad < lo_x or cx - rad > hi_x or cy + rad < lo_y or cy - rad > hi_y:
            continue
        left = rad * rad - ((Xf - cx) ** 2 + (Yf - cy) ** 2)
        z = torch.where(left >= 0, torch.minimum(z, c - left.clamp_min(0).sqrt() / zscale - RECEIVER_OFFSET), z)
    z = torch.where(z == 2.0, 1.0, z)
    return (X / w).float(), (Y / h).float(), z


def _shift(t, by):
    """A copy of a plane that starts `by` elements past an aligned address."""
    if not by:
        return t
    s = torch.empty(t.numel() + by, dtype=t.dtype, device=t.device)[by:]
    return s.copy_(t)


def _frames(case, seed):
    """[(occluders, map, fragments, homography)] of a moving light over one camera."""
    r = random.Random(seed)
    w, h, sw, sh = case["map_w"], case["map_h"], case["screen_w"], case["screen_h"]
    zscale = float(max(w, h))
    base, hom = _occluders(case["scene"], r, w, h), _camera(r, w, h)
    out = []
    for f in range(case["frames"]):
        occ = _shifted(base, 0.25 * zscale * math.tan(math.radians(0.5 * f)))
        out.append((occ, _map(occ, w, h, zscale, case["texture"]), _fragments(hom, sw, sh, w, h, occ[1], zscale), hom))
    return out


CASCADE_VIEWS = [(1.0, 1.0), (0.75, 0.8), (0.5, 0.5), (1 / 3, 1 / 3)]    # of the screen


def _cascades(case, seed):
    """(maps, [(map index, x, y, z)]): 4 lights x 4 cascades, every view's bands against every light."""
    r = random.Random(seed)
    sizes = [max(128, case["map_w"] >> c) for c in range(4)]
    maps, jobs = [], []
    for _ in range(4):
        for size in sizes:
            maps.append(_map(_occluders("fence", r, size, size), size, size, float(size), case["texture"]))
    for sx, sy in CASCADE_VIEWS[:case["frames"]]:
        sw, sh = max(16, int(case["screen_w"] * sx)), max(16, int(case["screen_h"] * sy))
        for light in range(4):
            for c, size in enumerate(sizes):
                rows = sh - c * sh // 4 - (sh - (c + 1) * sh // 4)
                jobs.append((light * 4 + c,) + _fragments(_camera(r, size, size, (0.25, 0.5)), sw, rows, size, size, [],
                                                          float(size)))
    return maps, jobs


# ---------------------------------------------------------------- prepare --

def _answer_planes(case, sizes):
    """One plane per kind of answer for all jobs, and each job's views of them (16-byte aligned starts)."""
    starts, total = [], 0
    for n in sizes:
        starts.append(total)
        total += (n + 7) // 8 * 8
    planes = {}
    if case["mode"] & SILHOUETTE:
        planes["silhouette"] = torch.zeros(total, dtype=torch.float32, device=DEV)
    if case["mode"] & FILTER:
        planes["filter"] = torch.zeros(total, dtype=torch.float32, device=DEV)
    if case["codes"]:
        planes["codes"] = torch.zeros(total, dtype=torch.int16, device=DEV)
    views = [{k: p[s:s + n] for k, p in planes.items()} for s, n in zip(starts, sizes)]
    return planes, views


def _texture(case, depth):
    return api.MapTexture(depth) if case["texture"] else depth


def _gbuffer(hom, sw, sh, w, h, z):
    """(depth buffer, 4x4 float32 screen-to-light matrix) whose projection gives the fragments of `hom` with depths z."""
    p = _pixels(hom, sw, sh)
    m = np.zeros((4, 4))
    m[0, [0, 1, 3]], m[1, [0, 1, 3]], m[2, 2], m[3, [0, 1, 3]] = p[0] / w, p[1] / h, 1.0, p[2]
    m = m.astype(np.float32)
    u = torch.arange(sw, device=DEV, dtype=torch.float32) + 0.5
    v = (torch.arange(sh, device=DEV, dtype=torch.float32) + 0.5)[:, None]
    ww = (u * float(m[3, 0]) + v * float(m[3, 1])) + 0.0
    ww = ww + float(m[3, 3])
    return (z.view(sh, sw) * ww).contiguous(), m


def _samples(case, seed):
    """Packed training samples around straight edges, initial weights and one minibatch order."""
    g = np.random.default_rng(seed)
    n = 1 << 17
    ang, off = g.uniform(0, 2 * math.pi, n), g.uniform(-0.9, 0.9, n)
    nx, ny = np.cos(ang), np.sin(ang)
    bits = np.zeros(n, np.uint32)
    for dy in range(-2, 3):
        for dx in range(-2, 3):
            bits |= ((nx * dx + ny * dy + off) > 0).astype(np.uint32) << np.uint32((dy + 2) * 5 + dx + 2)
    fx, fy = g.random(n, dtype=np.float32), g.random(n, dtype=np.float32)
    feat = {"bits": bits, "fx": fx, "fy": fy, "gap": g.uniform(0.0, 0.9, n).astype(np.float32)}
    label = np.clip(0.5 + nx * (fx - 0.5) + ny * (fy - 0.5) + off, 0, 1).astype(np.float32)

    def he(fan_in, shape):
        return (g.standard_normal(shape) * math.sqrt(2.0 / fan_in)).astype(np.float32)

    params = {"W1": he(28, (32, 64)), "b1": np.zeros(64, np.float32), "W2": he(64, (64, 64)),
              "b2": np.zeros(64, np.float32), "W3": he(64, (64, 2)) * np.float32(0.1),
              "b3": np.array([0.5, 0.05], np.float32)}
    return feat, label, params, g.integers(0, n, case["batch"]).astype(np.int32)


def _device_occluders(occ):
    rects, spheres = occ
    r = np.array([c[:6] for c in rects], np.float64).reshape(-1, 6)
    return api.DeviceOccluders(r, np.array([c[6] for c in rects], np.float32),
                               np.array(spheres, np.float64).reshape(-1, 4))


def prepare(case, seed):
    kind, st = case["kind"], {"case": case}
    if kind == "train":
        feat, label, params, order = _samples(case, seed)
        st["net"] = sg.Surrogate(params)
        st["samples"], _ = sg.Surrogate.pack(feat, label)
        st["order"] = torch.from_numpy(order).to(DEV)
        return st
    if kind == "light":
        r = random.Random(seed)
        w, h = case["map_w"], case["map_h"]
        base = _occluders(case["scene"], r, w, h)
        st["occ"] = [_device_occluders(_shifted(base, 0.25 * max(w, h) * math.tan(math.radians(0.5 * f))))
                     for f in range(case["frames"])]
        st["maps"] = [torch.empty((h, w), dtype=torch.float32, device=DEV) for _ in st["occ"]]
        return st
    if kind == "batch" and case["scene"] == "cascades":
        maps, jobs = _cascades(case, seed)
    else:
        frames = _frames(case, seed)
        maps, jobs = [f[1] for f in frames], [(k,) + f[2] for k, f in enumerate(frames)]
    if kind in ("single", "rpcf"):
        st["map"] = _texture(case, maps[0])
        st["xyz"] = [_shift(t, case["shift"]) for t in jobs[0][1:]]
        return st
    if kind == "host":
        pin = lambda t: t.cpu().pin_memory()  # noqa: E731
        st["maps"] = [pin(m) for m in maps]
        st["jobs"] = [api.Job(j[0], pin(j[1]), pin(j[2]), pin(j[3]), mode=case["mode"]) for j in jobs]
        st["stager"] = api.Stager(max(j[1].numel() for j in jobs), case["map_w"], case["map_h"])
        return st
    if kind == "gbuffer":
        st["jobs"] = []
        st["out"], views = _answer_planes(case, [j[1].numel() for j in jobs])
        for f, v in zip(frames, views):
            d, m = _gbuffer(f[3], case["screen_w"], case["screen_h"], case["map_w"], case["map_h"], f[2][2])
            st["jobs"].append(api.GBufferJob(_texture(case, f[1]), d, m, mode=case["mode"], codes=v.get("codes"),
                                             vis_silhouette=v.get("silhouette"), vis_filter=v.get("filter")))
        return st
    st["out"], views = _answer_planes(case, [j[1].numel() for j in jobs])
    made = [api.Job(j[0], j[1], j[2], j[3], mode=case["mode"], codes=v.get("codes"), vis_silhouette=v.get("silhouette"),
                    vis_filter=v.get("filter")) for j, v in zip(jobs, views)]
    if kind == "learned":
        st["net"] = sg.Surrogate.from_checkpoint(CHECKPOINT)
        st["batch"] = api.Batch([_texture(case, m) for m in maps], made, max_dist=case["max_dist"],
                                surrogate=st["net"], guard_tau=GUARD_TAU)
    else:
        st["batch"] = api.Batch([_texture(case, m) for m in maps], made, max_dist=case["max_dist"])
    return st


# -------------------------------------------------------------------- run --

def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "single":
        fn = api.rsmss_filter if case["mode"] == FILTER else api.rbsm_visibility
        return fn(st["map"], *st["xyz"], codes=case["codes"], max_dist=case["max_dist"])
    if kind == "rpcf":
        return api.rbsm_rpcf(st["map"], *st["xyz"], k=case["k"], max_dist=case["max_dist"])
    if kind in ("batch", "learned"):
        api.rbsm_batch_run(st["batch"])
        return st["out"]
    if kind == "gbuffer":
        api.rbsm_visibility_gbuffer(st["jobs"], mode=case["mode"], max_dist=case["max_dist"])
        return st["out"]
    if kind == "light":
        return api.rbsm_shadow_maps(st["occ"], case["map_w"], case["map_h"], float(max(case["map_w"], case["map_h"])),
                                    outs=st["maps"])
    if kind == "train":
        st["net"].train_step(st["samples"], st["order"], 1e-3)
        return st["net"].state[:sg.N_PARAMS]         # the float32 parameters lead the state block
    st["stager"].run(st["maps"], st["jobs"], max_dist=case["max_dist"])
    return [[j.vis_silhouette, j.vis_filter] for j in st["jobs"]]


# ------------------------------------------------------------------- work --

def _job_sizes(case):
    """[(fragments, map width, map height, window as a share of the map's smaller side squared)]"""
    if case["kind"] == "batch" and case["scene"] == "cascades":
        out = []
        for sx, sy in CASCADE_VIEWS[:case["frames"]]:
            sw, sh = max(16, int(case["screen_w"] * sx)), max(16, int(case["screen_h"] * sy))
            for c in range(4):
                size = max(128, case["map_w"] >> c)
                out += [(sw * (sh - c * sh // 4 - (sh - (c + 1) * sh // 4)), size, size, 0.375)] * 4
        return out
    return [(case["screen_w"] * case["screen_h"], case["map_w"], case["map_h"], 0.3)] * case["frames"]


def work(case):
    kind = case["kind"]
    if kind == "train":
        # three products forward, their two backward counterparts each, 2 operations per weight and sample
        return {"bytes": case["batch"] * (20.0 + 4.0) + 6402 * 4 * 8.0, "flops": case["batch"] * 6.0 * 6272}
    if kind == "light":
        return {"bytes": 4.0 * case["map_w"] * case["map_h"] * case["frames"], "flops": 0.0}
    per = 4.0 if kind == "gbuffer" else 12.0
    per += 4.0 * ((case["mode"] & 1) + (case["mode"] >> 1 & 1)) + (2.0 if case["codes"] else 0.0)
    total = 0.0
    for n, w, h, zoom in _job_sizes(case):
        # the fragments, and each texel under them once (a trapezoid of three quarters of the window's square)
        total += n * per + 4.0 * min(n, 0.75 * (zoom * min(w, h)) ** 2)
    return {"bytes": total, "flops": 0.0}


def tolerance(case):
    kind = case["kind"]
    if kind == "light" or (case["mode"] == SILHOUETTE and kind != "train"):
        return "exact"                       # hard shadows, codes and the light pass are defined to the bit
    if kind == "train":
        # Adam's first step moves every weight by the learning rate in the sign of its gradient, which 16-bit operands
        # leave open where the gradient is near zero (measured against 64 bits: 3.8e-4)
        return {"rel": 1.5e-3, "max": 0.05}
    if kind == "learned":
        # another order of the network's float32 sums moves its estimates by 16-bit roundings of the hidden units and
        # can flip the guard's choice between an estimate and the exact walk (both within the stated bound of 0.1)
        return {"rel": 1e-3, "max": 0.15}
    # one rounded divide and add per axis (measured: 1.5e-9 to 6e-9; most answers are 0 or 1), and for RPCF the samples'
    # rounding to 2^-20 .. 2^-24 (measured: 1.2e-8)
    return {"rel": 5e-8, "max": 2e-6}


# ------------------------------------------------------------------ exact --

def _walk(lit, s0, i, j, di, dj, use_a, use_b, w, h, max_dist):
    """The steps of one walk: +k for an end at step k, -k where the edge is left, -(max_dist + 1) for neither."""
    r = torch.zeros_like(i)
    for k in range(1, max_dist + 1):
        ci, cj = (i + k * di).clamp(0, w - 1), (j + k * dj).clamp(0, h - 1)
        end = lit(ci, cj) != s0
        a = lit((ci + abs(dj)).clamp(0, w - 1), (cj + abs(di)).clamp(0, h - 1)) != s0
        b = lit((ci - abs(dj)).clamp(0, w - 1), (cj - abs(di)).clamp(0, h - 1)) != s0
        on = (use_a & a) | (use_b & b)
        r = torch.where((r == 0) & end, k, torch.where((r == 0) & ~on, -k, r))
        if bool((r != 0).all()):
            break
    return torch.where(r == 0, -(max_dist + 1), r)


def _position(rn, rp, f, dtype):
    """Normalised position along an axis, in `dtype`."""
    f = f.to(dtype)
    length = (rn.abs() + rp.abs() - 1).to(dtype)
    neg, pos = (rn > 0) & (rp <= 0), (rp > 0) & (rn <= 0)
    one = torch.ones_like(f)
    return torch.where(neg, ((rn - 1).to(dtype) + f) / length, torch.where(pos, ((rp - 1).to(dtype) + (one - f)) / length, one))


def _exact_texel(depth, u, v, z, max_dist, want):
    """{silhouette, filter (float64), codes of each mode} for float32 texel-space positions: texels, tests, walks and the
    hard decision in the float32 operations that define them, the filtered value in 64 bits."""
    h, w = depth.shape

    def cell(t, n):
        fl = torch.floor(t)
        return fl.clamp(0, n - 1).nan_to_num(0.0).long(), t - fl

    i, fx = cell(u, w)
    j, fy = cell(v, h)
    lit_at = lambda zz: (lambda a, b: ~(zz > depth[b, a]))  # noqa: E731
    lit = lit_at(z)
    s0 = lit(i, j)
    dl, dr = lit((i - 1).clamp_min(0), j) != s0, lit((i + 1).clamp_max(w - 1), j) != s0
    du, dd = lit(i, (j + 1).clamp_max(h - 1)) != s0, lit(i, (j - 1).clamp_min(0)) != s0
    code = dl.int() | (dr.int() << 1) | (du.int() << 2) | (dd.int() << 3) | ((~s0).int() << 4)
    at = torch.nonzero(dl | dr | du | dd).reshape(-1)
    i, j, fx, fy, s, z, dl, dr, du, dd = (t[at] for t in (i, j, fx, fy, s0, z, dl, dr, du, dd))
    lit = lit_at(z)
    rxn, rxp = (_walk(lit, s, i, j, d, 0, du, dd, w, h, max_dist) for d in (-1, 1))
    ryn, ryp = (_walk(lit, s, i, j, 0, d, dr, dl, w, h, max_dist) for d in (-1, 1))
    ex, ey = (rxn > 0).int() + (rxp > 0).int(), (ryn > 0).int() + (ryp > 0).int()
    out = {}
    walked = code.clone()
    walked[at] |= (ex << 5) | (ey << 7) | (1 << 9)
    if "silhouette" in want:
        nx, ny = _position(rxn, rxp, fx, torch.float32), _position(ryn, ryp, fy, torch.float32)
        val = (~(ny < 1.0 - nx)).double()
        val = torch.where((ex == 0) | (ey == 0), 1.0, val)
        val = torch.where((dl & dr) | (du & dd) | (ex == 2) | (ey == 2) | ~s, 0.0, val)
        sil = s0.double()
        sil[at] = val
        out["silhouette"] = sil
        out["codes1"] = torch.where(s0, walked, code)          # shadowed fragments do not walk
    if "filter" in want:
        nx, ny = _position(rxn, rxp, fx, torch.float64), _position(ryn, ryp, fy, torch.float64)
        dz = (~s).double()
        sx, sy = torch.where(s, nx, -nx), torch.where(s, ny, -ny)
        val = (dz + sy + sx).clamp(0.0, 1.0)
        val = torch.where((ex == 0) | (ey == 0), 1.0 - dz, val)
        val = torch.where(ey == 2, dz + sx, val)
        val = torch.where(ex == 2, dz + sy, val)
        val = torch.where(((dl & dr) & (du & dd)) | ((ex == 2) & (ey == 2)), dz, val)
        fil = s0.double()
        fil[at] = val
        out["filter"] = fil
        out["codes2"] = walked
    return out


def _exact_job(case, depth, x, y, z):
    h, w = depth.shape
    want = [n for n, bit in (("silhouette", SILHOUETTE), ("filter", FILTER)) if case["mode"] & bit]
    got = _exact_texel(depth, x * float(w), y * float(h), z, case["max_dist"], want)
    if case["codes"]:
        got["codes"] = (got["codes2"] if case["mode"] & FILTER else got["codes1"]).to(torch.int16)
    return {k: got[k] for k in want + (["codes"] if case["codes"] else [])}


def _exact_train(case, seed):
    """The parameters after the first step, without any 16-bit rounding."""
    feat, label, params, order = _samples(case, seed)
    X = np.zeros((case["batch"], 32))
    for b in range(25):
        X[:, b] = (feat["bits"][order] >> b) & 1
    for c, key in enumerate(("fx", "fy", "gap")):
        X[:, 25 + c] = feat[key][order]
    X, t = torch.from_numpy(X).to(DEV), torch.from_numpy(label[order].astype(np.float64)).to(DEV)
    p = [torch.from_numpy(params[k].astype(np.float64)).to(DEV).requires_grad_() for k in ("W1", "b1", "W2", "b2", "W3", "b3")]
    y = torch.relu(torch.relu(X @ p[0] + p[1]) @ p[2] + p[3]) @ p[4] + p[5]
    err = (y[:, 0].detach().clamp(0, 1) - t).abs()
    (((y[:, 0] - t) ** 2).mean() + ((y[:, 1] - err) ** 2).mean()).backward()
    return torch.cat([(q.detach() - 1e-3 * q.grad / (q.grad.abs() + 1e-8)).reshape(-1) for q in p])


def exact(case, seed):
    kind = case["kind"]
    if kind == "learned":
        return None                          # no 64-bit value: 16-bit operands decide which fragments are estimated
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "light":
        r = random.Random(seed)
        w, h = case["map_w"], case["map_h"]
        base = _occluders(case["scene"], r, w, h)
        return [_raster(_shifted(base, 0.25 * max(w, h) * math.tan(math.radians(0.5 * f))),
                        torch.empty((h, w), dtype=torch.float32, device=DEV), float(max(w, h)), torch.float64)
                for f in range(case["frames"])]
    if kind == "batch" and case["scene"] == "cascades":
        maps, jobs = _cascades(case, seed)
    else:
        frames = _frames(case, seed)
        maps, jobs = [f[1] for f in frames], [(k,) + f[2] for k, f in enumerate(frames)]
    if kind == "gbuffer":
        jobs = []
        for k, f in enumerate(frames):
            sw, sh = case["screen_w"], case["screen_h"]
            d, m = _gbuffer(f[3], sw, sh, case["map_w"], case["map_h"], f[2][2])
            u = torch.arange(sw, device=DEV, dtype=torch.float32) + 0.5
            v = (torch.arange(sh, device=DEV, dtype=torch.float32) + 0.5)[:, None]
            rows = [(u * float(m[q, 0]) + v * float(m[q, 1])) + d * float(m[q, 2]) for q in range(4)]
            rows = [t + float(m[q, 3]) for q, t in enumerate(rows)]
            jobs.append((k,) + tuple((t / rows[3]).reshape(-1) for t in rows[:3]))
    if kind == "rpcf":
        _, x, y, z = jobs[0]
        h, w = maps[0].shape
        u, v, half = x * float(w), y * float(h), (case["k"] - 1) // 2
        total = 0.0
        for b in range(-half, half + 1):
            for a in range(-half, half + 1):
                total = total + _exact_texel(maps[0], u + float(a), v + float(b), z, case["max_dist"], ["filter"])["filter"]
        return total / case["k"] ** 2
    got = [_exact_job(case, maps[j[0]], *j[1:]) for j in jobs]
    if kind == "single":
        name = "filter" if case["mode"] == FILTER else "silhouette"
        return got[0][name], got[0].get("codes")
    if kind == "host":
        return [[g["silhouette"], g["filter"]] for g in got]
    planes = {}
    for key in got[0]:
        parts = []
        for g in got:
            n = g[key].numel()
            parts += [g[key], torch.zeros((n + 7) // 8 * 8 - n, dtype=g[key].dtype, device=DEV)]
        planes[key] = torch.cat(parts)
    return planes
