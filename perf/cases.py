"""Performance cases of the renderer: what its users call, over the sizes they call it with.

    listed()               the named cases
    draw(rng)              one more case of the same ranges
    prepare(case, seed)    what a program holds before the call (scene, cameras, buffers, server)
    run(state)             one pass through the public entry points; returns its outputs
    work(case)             bytes and floating-point operations that a pass cannot do without
    exact(case, seed)      the same outputs in 64 bits from plain torch, where that is quick

Every scene is generated from the seed (geometry, albedo and pose), with the library's default tuning; only the
sizes of batched views and of served requests are those of the repository's own fixed mixes.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2312_12392_gb300 import rcp, scenes

EYE, TARGET, DEPTH, IMAGE, NORMAL = (rcp.RCP_MAP_EYE, rcp.RCP_MAP_TARGET, rcp.RCP_MAP_DEPTH, rcp.RCP_MAP_IMAGE,
                                     rcp.RCP_MAP_NORMAL)
SORT_BITS = 30


def _frame(name, scene, size, width, height, passes, mapping, spp=0, continued=False):
    c = {"kind": "frame", "scene": scene, "size": size, "width": width, "height": height, "passes": passes,
         "mapping": mapping, "spp": spp, "continued": continued}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a thumbnail of a handful of primitives, where launches and latency count
        _frame("tiny_eye_128", "tiny", 5, 128, 128, 6, EYE),
        # the headline: one walk-through frame of the 133k-triangle terrain, the paper's K = 6, on the device
        _frame("terrain_eye_1080p", "terrain", 256, 1920, 1080, 6, EYE),
        # an odd-sized window, normal-driven cameras, continued from the previous frame's image (temporal feedback)
        _frame("terrain_normal_1283x717", "terrain", 256, 1283, 717, 5, NORMAL, continued=True),
        # anti-aliased frames: four jittered samples per pixel, the paper's displaced targets
        _frame("terrain_jitter4_720p", "terrain", 256, 1280, 720, 6, TARGET, spp=4),
        # the image-space reduction at 4K: one traced pass, then gathers
        _frame("terrain_image_2160p", "terrain", 256, 3840, 2160, 6, IMAGE),
        # a frame of the 1.07M-triangle forest, in the build advised for many separate objects
        _frame("forest_eye_1080p", "forest", 2000, 1920, 1080, 6, EYE),
        # many uneven views of one scene in one call (stereo pairs, light-field and dataset renders)
        {"name": "forest_batch16", "kind": "batch", "scene": "forest", "size": 2000, "views": 16, "passes": 6,
         "mapping": EYE},
        # an animated frame: 3.07M swaying triangles refitted, then rendered at 4K with K = 8
        {"name": "forest_moving_2160p", "kind": "moving", "scene": "forest", "size": 6000, "width": 3840,
         "height": 2160, "passes": 8, "mapping": EYE},
        # a frame delivered to host memory, depth-driven cameras
        {"name": "terrain_host_1440p", "kind": "host", "scene": "terrain", "size": 221, "width": 2560, "height": 1440,
         "passes": 4, "mapping": DEPTH},
        # opening a scene: 1M triangles from host arrays to the first preview image
        {"name": "terrain_load_1m", "kind": "load", "scene": "terrain", "size": 706, "width": 480, "height": 270,
         "mapping": EYE},
        # the render server: a burst of requests of mixed sizes and K over two resident scenes
        {"name": "serve_mix12", "kind": "serve", "size": 221, "size2": 706, "requests": 12},
        # the allocation-free sort at its real-time loop's usual full load
        {"name": "sort_1m", "kind": "sort", "pairs": 1000003},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "frame", "frame", "image", "batch", "moving", "host", "load", "serve", "sort"])
    mapping = rng.choice([EYE, EYE, TARGET, DEPTH, NORMAL])
    w, h = _log(rng, 160, 2560), _log(rng, 120, 1440)
    if kind == "frame":
        scene = rng.choice(["tiny", "terrain", "terrain", "forest"])
        if scene == "tiny":
            return _frame(None, "tiny", 5, _log(rng, 48, 640), _log(rng, 48, 480), rng.randint(1, 8), mapping,
                          rng.choice([0, 0, 4]), rng.random() < 0.3)
        size = _log(rng, 64, 706) if scene == "terrain" else _log(rng, 50, 3000)
        spp = rng.choice([0, 0, 0, 1, 2, 4])
        return _frame(None, scene, size, w, h, rng.randint(1, 8 if spp < 2 else 6), mapping, spp, rng.random() < 0.3)
    if kind == "image":
        return _frame(None, "terrain", _log(rng, 64, 400), _log(rng, 320, 3840), _log(rng, 180, 2160),
                      rng.randint(2, 8), IMAGE)
    if kind == "batch":
        return {"kind": "batch", "scene": rng.choice(["terrain", "forest"]), "size": _log(rng, 100, 700),
                "views": rng.randint(2, 20), "passes": rng.randint(1, 6), "mapping": mapping}
    if kind == "moving":
        return {"kind": "moving", "scene": "forest", "size": _log(rng, 30, 5000), "width": w, "height": h,
                "passes": rng.randint(1, 8), "mapping": mapping}
    if kind == "host":
        return {"kind": "host", "scene": rng.choice(["terrain", "forest"]), "size": _log(rng, 100, 700), "width": w,
                "height": h, "passes": rng.randint(1, 8), "mapping": mapping}
    if kind == "load":
        scene = rng.choice(["terrain", "forest"])
        return {"kind": "load", "scene": scene, "size": _log(rng, 64, 706) if scene == "terrain" else _log(rng, 50, 1500),
                "width": _log(rng, 160, 640), "height": _log(rng, 120, 360), "mapping": mapping}
    if kind == "serve":
        return {"kind": "serve", "size": _log(rng, 100, 300), "size2": _log(rng, 300, 706),
                "requests": rng.randint(3, 12)}
    return {"kind": "sort", "pairs": _log(rng, 1000, 1 << 20)}


# ------------------------------------------------------------------ inputs

def _scene(kind, size, seed):
    if kind == "tiny":
        return scenes.tiny_scene(seed + 1)
    if kind == "terrain":
        return scenes.terrain_scene(size, seed + 2)
    return scenes.forest_scene(size, seed + 3)


def _options(kind):
    """Build options: the defaults for terrains, the advised ones for many separate objects."""
    return (rcp.RCP_COLLAPSE_SAH, rcp.RCP_SPLIT_MAX) if kind == "forest" else (None, 0)


def _jitter(spp, rng):
    """Stratified sample offsets."""
    if not spp:
        return None
    return np.stack([(np.arange(spp) + rng.random(spp)) / spp, rng.permutation((np.arange(spp) + rng.random(spp)) / spp)],
                    axis=1).astype(np.float32) * np.float32(0.9999)


def _params(mapping, sc, spp=0, rng=None, k_frac=None, width=0):
    diam = sc.diameter()
    f = 6.0 if sc.name == "tiny" else 0.1 * diam
    k = (k_frac if k_frac is not None else 0.05 if sc.name == "tiny" else 0.02) * diam
    if mapping == IMAGE:
        k = 0.02 * width  # pixels
    elif mapping == DEPTH:
        k *= 0.05  # multiplies |z - z0|
    return rcp.make_params(mapping, k, f, z0=f, jitter=_jitter(spp, rng))


class _State:
    """A case's inputs; destroys its scenes and server when it goes."""

    def __init__(self, case):
        self.case = case
        self.scenes = []
        self.server = None

    def add(self, sc, kind):
        self.scenes.append(rcp.scene_from(sc, *_options(kind)))
        return self.scenes[-1]

    def __del__(self):
        if self.server:
            rcp.rcp_server_destroy(self.server)
        for g in self.scenes:
            rcp.rcp_scene_destroy(g)


def _image(h, w):
    return torch.empty((h, w, 4), dtype=torch.float32, device="cuda")


def prepare(case, seed):
    rng = np.random.default_rng(seed + 77)
    s = _State(case)
    kind = case["kind"]
    if kind == "sort":
        g = torch.Generator(device="cuda").manual_seed(seed)
        n = case["pairs"]
        s.keys = torch.randint(0, 1 << SORT_BITS, (n,), dtype=torch.int32, device="cuda", generator=g)
        s.values = torch.arange(n, dtype=torch.int32, device="cuda")
        s.out_keys, s.out_values = torch.empty_like(s.keys), torch.empty_like(s.values)
        return s
    if kind == "serve":
        host = [_scene("terrain", case["size"], seed), _scene("terrain", case["size2"], seed)]
        handles = [s.add(sc, "terrain") for sc in host]
        s.requests = []
        for q in scenes.served_requests(case["requests"], 2, 64):  # the mix; poses and strengths from the seed
            i, w, h = q["scene"], q["width"], q["height"]
            s.requests.append((handles[i], rcp.camera_from(host[i].poses[int(rng.integers(0, 64))]), w, h, q["K"],
                               _params(EYE, host[i], k_frac=float(rng.uniform(0.0, 0.05))),
                               np.zeros((h, w, 3), np.float32)))
        s.server = rcp.rcp_server_create(8 << 30, 16)
        return s
    sc = _scene(case["scene"], case["size"], seed)
    poses = [rcp.camera_from(sc.poses[int(p)]) for p in rng.integers(0, len(sc.poses), case.get("views", 1) + 1)]
    s.cam = poses[0]
    s.params = _params(case["mapping"], sc, case.get("spp", 0), rng, width=case.get("width", 0))
    if kind == "load":
        s.source = sc
        return s
    s.scene = s.add(sc, case["scene"])
    if kind == "batch":
        sizes = scenes.batched_view_sizes(case["views"])
        s.cams, s.widths, s.heights = poses[1:], [w for w, _ in sizes], [h for _, h in sizes]
        s.outs = [_image(h, w) for w, h in sizes]
        return s
    w, h = case["width"], case["height"]
    if kind == "host":
        s.rgb = np.zeros((h, w, 3), np.float32)
        return s
    s.out = _image(h, w)
    s.ids = torch.empty((h, w), dtype=torch.int32, device="cuda") if case["mapping"] != IMAGE else None
    s.previous = None
    if case.get("continued"):  # the previous frame, from the pose before
        s.previous = _image(h, w)
        rcp.rcp_render_device(s.scene, poses[1], w, h, 1, s.params, None, s.previous, None, torch.cuda.current_stream())
    if kind == "moving":  # this frame's vertices: wind sway, as a simulation leaves them on the device
        v = torch.from_numpy(sc.tris).cuda().view(-1, 3, 3).clone()
        amp = torch.from_numpy(sc.sway_amp).cuda()
        angle = torch.from_numpy(sc.sway_phase).cuda()[:, None] + 2 * math.pi * 0.5 * (seed % 60) / 60.0
        v[:, :, 0] += amp * torch.sin(angle)
        v[:, :, 2] += amp * torch.cos(angle)
        s.vertices = v.reshape(-1, 9).contiguous()
    return s


# ------------------------------------------------------------------ one pass

def _split(image, mapping):
    """An rgbz image's outputs: colour, and the fourth lane (z-depth; the normal mapping's is a 32-bit code)."""
    last = image[..., 3]
    if mapping == NORMAL:
        last = last.view(torch.int32) if isinstance(last, torch.Tensor) else np.ascontiguousarray(last).view(np.int32)
    return {"rgb": image[..., :3], "lane": last}


def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "sort":
        s.out_keys.copy_(s.keys)
        s.out_values.copy_(s.values)
        rcp.rcp_sort_pairs_static(s.out_keys, s.out_values, c["pairs"], SORT_BITS, torch.cuda.current_stream())
        return [s.out_keys, s.out_values]
    if kind == "serve":
        tickets = [rcp.rcp_server_submit(s.server, *q) for q in s.requests]
        for t in tickets:
            rcp.rcp_server_wait(s.server, t, 60.0)
        return [q[-1] for q in s.requests]
    if kind == "load":
        g = rcp.scene_from(s.source, *_options(c["scene"]))
        ids = np.empty((c["height"], c["width"]), np.int32)
        image = rcp.rcp_render_pass(g, s.cam, c["width"], c["height"], s.params, out_prim=ids)
        diam = rcp.rcp_scene_get_info(g).diam
        rcp.rcp_scene_destroy(g)
        return {**_split(image, c["mapping"]), "ids": ids, "diam": diam}
    if kind == "host":
        return rcp.rcp_render(s.scene, s.cam, c["width"], c["height"], c["passes"], s.params, s.rgb)
    stream = torch.cuda.current_stream()
    if kind == "batch":
        rcp.rcp_render_batch_device(s.scene, s.cams, s.widths, s.heights, c["passes"], s.params, s.outs, stream)
        return [_split(o, c["mapping"]) for o in s.outs]
    if kind == "moving":
        rcp.rcp_scene_update_vertices_device(s.scene, s.vertices, stream)
    rcp.rcp_render_device(s.scene, s.cam, c["width"], c["height"], c["passes"], s.params, s.previous, s.out, s.ids,
                          stream)
    out = _split(s.out, c["mapping"])
    return out if s.ids is None else {**out, "ids": s.ids}


# ------------------------------------------------------------------ what a pass cannot do without

def _triangles(kind, size):
    return 2 if kind == "tiny" else 2 * size * size + 2400 if kind == "terrain" else 65522 + 500 * size


def _rays(scene, size, samples):
    """Operations of tracing `samples` camera samples: a primary and about 0.5 shadow rays each, a ray testing the
    boxes on one path from the root of an 8-wide tree (14 operations a box) and one triangle (34); 40 to make the
    camera and shade."""
    levels = 1 + math.ceil(math.log(max(_triangles(scene, size) / 3, 1), 8))
    return samples * (1.5 * (levels * 8 * 14 + 34) + 40)


def work(case):
    kind = case["kind"]
    if kind == "sort":
        return {"bytes": 16 * case["pairs"], "flops": 0}
    if kind == "serve":
        mix = scenes.served_requests(case["requests"], 2, 64)
        return {"bytes": sum(12 * q["width"] * q["height"] for q in mix),
                "flops": sum(_rays("terrain", (case["size"], case["size2"])[q["scene"]], q["K"] * q["width"] * q["height"])
                             for q in mix)}
    if kind == "batch":
        pixels = sum(w * h for w, h in scenes.batched_view_sizes(case["views"]))
    else:
        pixels = case["width"] * case["height"]
    triangles = _triangles(case["scene"], case["size"])
    if kind == "load":  # vertices and albedo in, tree and image out: 48 bytes a record and a node's share of 26
        return {"bytes": triangles * (36 + 12 + 48 + 26) + 20 * pixels, "flops": _rays(case["scene"], case["size"], pixels)}
    traced = 1 if case["mapping"] == IMAGE else case["passes"]
    flops = _rays(case["scene"], case["size"], pixels * traced * max(1, case.get("spp", 0)))
    moved = pixels * (12 if kind == "host" else 20 if kind in ("frame", "moving") else 16)
    if case.get("spp", 0) or case["mapping"] == IMAGE:  # neighbours' values: every pass's image is written and read
        moved += pixels * (case["passes"] - 1) * (48 if case["mapping"] == IMAGE else 32)
    if kind == "moving":  # vertices in, records and boxes out
        moved += triangles * (36 + 48 + 26)
    return {"bytes": moved, "flops": flops}


# ------------------------------------------------------------------ 64-bit values

def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _closest(o, d, tmin, tmax, tris, spheres):
    """Closest hit of rays o + t d, t in (tmin, tmax), by testing every primitive: t (inf: none), id (-1)."""
    t = torch.full_like(o[:, 0], math.inf)
    ids = torch.full_like(t, -1, dtype=torch.int64)
    for i in range(len(tris)):
        v0, e1, e2 = tris[i, 0], tris[i, 1] - tris[i, 0], tris[i, 2] - tris[i, 0]
        p = torch.linalg.cross(d, e2.expand_as(d))
        det = (p * e1).sum(-1)
        q = torch.linalg.cross(o - v0, e1.expand_as(d))
        u, v, th = (p * (o - v0)).sum(-1) / det, (d * q).sum(-1) / det, (q * e2).sum(-1) / det
        ok = (u >= 0) & (v >= 0) & (u + v <= 1) & (th > tmin) & (th < tmax) & (th < t)
        t, ids = torch.where(ok, th, t), torch.where(ok, torch.full_like(ids, i), ids)
    for i in range(len(spheres)):
        oc = o - spheres[i, :3]
        b = (oc * d).sum(-1)
        disc = b * b - (oc * oc).sum(-1) + spheres[i, 3] ** 2
        root = disc.clamp(min=0).sqrt()
        th = torch.where(-b - root > tmin, -b - root, -b + root)
        ok = (disc >= 0) & (th > tmin) & (th < tmax) & (th < t)
        t, ids = torch.where(ok, th, t), torch.where(ok, torch.full_like(ids, len(tris) + i), ids)
    return t, ids


def _exact_frame(case, sc, cam, params):
    """K passes in 64 bits: I_n from I_{n-1}, every ray tested against every primitive."""
    f64 = {"dtype": torch.float64, "device": "cuda"}
    tris = torch.tensor(sc.tris, **f64).view(-1, 3, 3)
    spheres, albedo = torch.tensor(sc.spheres, **f64), torch.tensor(sc.albedo, **f64)
    light, a = torch.tensor([float(np.float32(x)) for x in sc.light.v], **f64), float(np.float32(sc.light.ambient))
    diam, inf = sc.diameter(), math.inf
    eye, at, up = (torch.tensor(list(v), **f64) for v in (cam.eye, cam.look_at, cam.up))
    fwd = _unit(at - eye)
    right = _unit(torch.linalg.cross(fwd, up))
    upward = torch.linalg.cross(right, fwd)
    w, h = case["width"], case["height"]
    tan = math.tan(cam.fov_y_deg * math.pi / 360)
    y, x = torch.meshgrid(torch.arange(h, **f64), torch.arange(w, **f64), indexing="ij")
    sx, sy = ((2 * x + 1 - w) / w * tan * w / h).reshape(-1, 1), ((h - 2 * y - 1) / h * tan).reshape(-1, 1)
    focal = params.focal_dist * (fwd + sx * right + sy * upward)
    rgb, z = torch.full((w * h, 3), 0.5, **f64), torch.zeros(w * h, **f64)
    for _ in range(case["passes"]):
        c = 2 * rgb - 1
        v = params.k * (c[:, :1] * right + c[:, 1:2] * upward + c[:, 2:] * fwd)
        if case["mapping"] == EYE:
            o, d = eye + v, _unit(focal - v)
        else:
            m = (z - params.z0).abs()[:, None] if case["mapping"] == DEPTH else 1.0
            o, d = eye.expand_as(focal), _unit(focal + m * v)
        t, ids = _closest(o, d, 1e-6 * diam, inf, tris, spheres)
        hit = ids >= 0
        p = o + torch.where(hit, t, 0.0)[:, None] * d
        normals = [torch.linalg.cross(tr[1] - tr[0], tr[2] - tr[0]).expand_as(p) for tr in tris]
        normals += [p - sp[:3] for sp in spheres]
        n = _unit(torch.stack(normals)[ids.clamp(min=0), torch.arange(w * h, device="cuda")])
        n = torch.where((n * d).sum(-1, keepdim=True) > 0, -n, n)
        ndl = (n * _unit(light - p)).sum(-1)
        so = p + 1e-4 * diam * n
        dist = (light - so).norm(dim=-1)
        blocked = _closest(so, _unit(light - so), 0.0, dist, tris, spheres)[1] >= 0
        lit = torch.where((ndl > 0) & ~blocked, a + (1 - a) * ndl, a)
        s = 0.5 * (d[:, 1:2] + 1)
        sky = (1 - s) + s * torch.tensor([[0.5, 0.7, 1.0]], **f64)
        rgb = torch.where(hit[:, None], albedo[ids.clamp(min=0)] * lit[:, None], sky).clamp(0, 1)
        z = torch.where(hit, t * (d * fwd).sum(-1), 0.0)
    return {"rgb": rgb.view(h, w, 3), "lane": z.view(h, w), "ids": None}


def exact(case, seed):
    if case["kind"] == "sort":
        s = prepare(case, seed)
        keys, order = torch.sort(s.keys.long(), stable=True)
        return [keys, order]
    # scenes of more than a few primitives take too long against every one of them
    if case["kind"] != "frame" or case["scene"] != "tiny" or case["spp"] or case["continued"] or case["mapping"] == NORMAL:
        return None
    rng = np.random.default_rng(seed + 77)
    sc = _scene("tiny", 5, seed)
    cam = rcp.camera_from(sc.poses[int(rng.integers(0, 1, 2)[0])])
    return _exact_frame(case, sc, cam, _params(case["mapping"], sc))
