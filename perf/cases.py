"""The calls by which this library's speed is judged, with their inputs and values.

A case is one kind of use at one size; `prepare` makes what a program holds
before the call, `run` makes the call through the package's public entry
points, and `exact` gives the same outputs from the definitions in 64 bits.

Kinds:
  view      trace a camera view (camera rays in, Eq. 8 sums out)
  step      one optimisation step of the tracer: the geometry has moved, so the
            hierarchy is rebuilt, then rays are traced and run backwards
  refit     the geometry has moved a little: refit, then trace a view
  raster    rasterise a G-buffer image
  shade     Monte Carlo shading of G-buffer points
  shade_step  the same, differentiated (the second training stage)
  relight   relighting of G-buffer points under a kept environment
  new_env   a new environment arrives: pre-integrate it, then relight
  serve     a burst of requests through the batching server
"""
import math

import numpy as np
import torch

import paper_2412_15867_gb300 as irgs
from paper_2412_15867_gb300 import serve

ALPHA_MIN = 1.0 / 255.0
DEV = "cuda:0"


def listed():
    return [
        # a unit-test-sized call: a tiny cloud and a 64 x 64 view, all latency
        {"name": "view_tiny", "kind": "view", "cloud": True, "surfels": 1024, "width": 64, "height": 64, "cams": 1,
         "k": 8, "channels": 3, "tiles": False},
        # one evaluation image of an object scene with all its channels
        {"name": "view_800", "kind": "view", "cloud": False, "surfels": 300000, "width": 800, "height": 800,
         "cams": 1, "k": 16, "channels": 10, "tiles": True},
        # a large optimisation batch over whole views, hit lists kept for the backward
        {"name": "step_views", "kind": "step", "surfels": 300000, "width": 800, "height": 800, "cams": 25,
         "pixels": 0, "channels": 10, "saved_hits": 96},
        # a small optimisation batch of random pixels with the default options
        # (no hit lists); odd counts, and the rebuild is a large part of it
        {"name": "step_pixels", "kind": "step", "surfels": 100003, "width": 800, "height": 800, "cams": 100,
         "pixels": 32769, "channels": 10, "saved_hits": 0},
        # a preview while a large scene is animated
        {"name": "refit_view", "kind": "refit", "surfels": 1000000, "width": 512, "height": 384, "channels": 3},
        # a G-buffer image of the first training stage
        {"name": "raster_800", "kind": "raster", "surfels": 300000, "width": 800, "height": 800, "channels": 10},
        # the shading of a full batch of primary hits, half cosine and half GGX samples
        {"name": "shade_640k", "kind": "shade", "surfels": 1000000, "points": 640000, "diffuse": 32, "spec": 32,
         "mode": "split", "aux": False},
        # an interactive preview with the stratified uniform estimator and the light split's maps
        {"name": "shade_preview", "kind": "shade", "surfels": 300000, "points": 4097, "diffuse": 63, "spec": 0,
         "mode": "uniform", "aux": True},
        # a mini-batch of the second training stage
        {"name": "shade_step", "kind": "shade_step", "surfels": 300000, "points": 16384, "diffuse": 32, "spec": 32,
         "mode": "split"},
        # an evaluation image relit
        {"name": "relight_100k", "kind": "relight", "surfels": 1000000, "points": 100000, "samples": 64},
        # a new environment map comes in and a thumbnail is relit under it
        {"name": "new_env", "kind": "new_env", "surfels": 100000, "points": 4096, "samples": 64, "env_h": 256},
        # a burst of render and relight requests for two resident scenes
        {"name": "serve_burst", "kind": "serve", "surfels": 100000, "requests": 6, "side": 256, "spp": 16},
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["view", "view", "step", "step", "refit", "raster", "shade", "shade_step", "relight", "new_env",
                       "serve"])
    c = {"kind": kind}
    if kind == "view":
        c["cloud"] = rng.random() < 0.3
        c["surfels"] = log_int(200, 8000) if c["cloud"] else log_int(20000, 1000000)
        c["width"], c["height"] = (log_int(16, 128), log_int(16, 128)) if c["cloud"] else (log_int(100, 1200), log_int(100, 1000))
        c["cams"] = rng.choice([1, 1, 2, 5])
        c["k"] = rng.choice([8, 16])
        c["channels"] = 3 if c["cloud"] else rng.choice([3, 7, 10])
        c["tiles"] = rng.random() < 0.5
    elif kind == "step":
        c["surfels"] = log_int(20000, 1000000)
        whole = rng.random() < 0.4
        c["width"], c["height"] = (log_int(100, 800), log_int(100, 800)) if whole else (800, 800)
        c["cams"] = rng.randint(1, 8) if whole else 100
        c["pixels"] = 0 if whole else log_int(1000, 300000)
        c["channels"] = rng.choice([3, 10])
        c["saved_hits"] = rng.choice([0, 32, 96])
    elif kind in ("refit", "raster"):
        c["surfels"] = log_int(20000, 2000000)
        c["width"], c["height"] = log_int(100, 1200), log_int(100, 1000)
        c["channels"] = rng.choice([3, 7, 10])
    elif kind in ("shade", "shade_step"):
        c["surfels"] = log_int(50000, 1000000)
        c["points"] = log_int(300, 100000 if kind == "shade" else 40000)
        c["mode"] = rng.choice(["split", "split", "uniform"])
        c["diffuse"] = rng.randint(4, 64)
        c["spec"] = 0 if c["mode"] == "uniform" else rng.randint(0, 64)
        if kind == "shade":
            c["aux"] = rng.random() < 0.5
    elif kind == "relight":
        c["surfels"] = log_int(50000, 1000000)
        c["points"] = log_int(300, 100000)
        c["samples"] = rng.randint(8, 96)
    elif kind == "new_env":
        c["surfels"] = log_int(20000, 300000)
        c["points"] = log_int(300, 20000)
        c["samples"] = rng.randint(8, 96)
        c["env_h"] = rng.randint(32, 300)
    else:
        c["surfels"] = log_int(50000, 300000)
        c["requests"] = rng.randint(2, 10)
        c["side"] = rng.choice([128, 200, 256, 400])
        c["spp"] = rng.randint(1, 48)
    return c


# ---------------------------------------------------------------------------
# Inputs (made on the GPU; distributions as in the synth module's scenes)

SPHERE_C, SPHERE_R = (-1.1, 0.0, 1.0), 1.0
TORUS_C, TORUS_R, TORUS_r = (1.1, 0.0, 0.25), 0.7, 0.25
GROUND = 2.5


class _Rng:
    def __init__(self, seed):
        self.g = torch.Generator(device=DEV).manual_seed(seed)

    def uniform(self, *shape, lo=0.0, hi=1.0):
        return lo + (hi - lo) * torch.rand(shape, generator=self.g, device=DEV, dtype=torch.float64)

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device=DEV, dtype=torch.float64)


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _f32(*ts):
    return tuple(t.to(torch.float32).contiguous() for t in ts)


def _surface(rng, n):
    """n points on a sphere, a torus and a ground square, allocated by area, with their normals."""
    areas = (4 * math.pi * SPHERE_R ** 2, 4 * math.pi ** 2 * TORUS_R * TORUS_r, (2 * GROUND) ** 2)
    ns = int(round(n * areas[0] / sum(areas)))
    nt = int(round(n * areas[1] / sum(areas)))
    ng = n - ns - nt
    a = _unit(rng.normal(ns, 3))
    u = rng.uniform(nt) * 2 * math.pi
    # the torus' minor angle has density ~ R + r cos v: invert its cdf v + (r/R) sin v by Newton steps
    t = rng.uniform(nt) * 2 * math.pi
    v = t.clone()
    for _ in range(20):
        v = v - (v + TORUS_r / TORUS_R * torch.sin(v) - t) / (1 + TORUS_r / TORUS_R * torch.cos(v))
    cu, su, cv, sv = torch.cos(u), torch.sin(u), torch.cos(v), torch.sin(v)
    tn = torch.stack([cv * cu, cv * su, sv], 1)
    tp = torch.stack([(TORUS_R + TORUS_r * cv) * cu, (TORUS_R + TORUS_r * cv) * su, TORUS_r * sv], 1)
    gp = torch.cat([rng.uniform(ng, 2, lo=-GROUND, hi=GROUND), torch.zeros(ng, 1, device=DEV, dtype=torch.float64)], 1)
    gn = torch.zeros(ng, 3, device=DEV, dtype=torch.float64)
    gn[:, 2] = 1.0
    c = lambda p: torch.tensor(p, device=DEV, dtype=torch.float64)
    return torch.cat([c(SPHERE_C) + SPHERE_R * a, c(TORUS_C) + tp, gp]), torch.cat([a, tn, gn])


def _object_scene(rng, n):
    """Surfels tangent to the surfaces, in no particular order: means, quats,
    scales, opacity, features (radiance, albedo, roughness, normal)."""
    p, nrm = _surface(rng, n)
    order = torch.argsort(rng.uniform(n))
    p, nrm = p[order], _unit(nrm[order] + 0.01 * rng.normal(n, 3))
    half = rng.uniform(n) * math.pi
    # the shortest rotation from z to the normal, after a turn about z
    w = 1 + nrm[:, 2]
    flip = w < 1e-9
    w, x, y = torch.where(flip, 0 * w, w), torch.where(flip, 0 * w + 1, -nrm[:, 1]), torch.where(flip, 0 * w, nrm[:, 0])
    c, s = torch.cos(half), torch.sin(half)
    q = _unit(torch.stack([w * c, x * c + y * s, y * c - x * s, w * s], 1))
    scales = torch.exp(math.log(0.01 * math.sqrt(300000.0 / n)) + 0.5 * rng.normal(n, 2))
    opacity = (rng.uniform(n) ** 0.2).clamp(1e-4, 1 - 1e-6)   # Beta(5, 1)
    feats = torch.cat([rng.uniform(n, 3), rng.uniform(n, 3, lo=0.05, hi=0.95), rng.uniform(n, 1, lo=0.05), nrm], 1)
    return _f32(p, q, scales, opacity, feats)


def _cloud(rng, n):
    return _f32(rng.uniform(n, 3, lo=-1.0), _unit(rng.normal(n, 4)),
                torch.exp(rng.uniform(n, 2, lo=math.log(0.02), hi=math.log(0.2))),
                rng.uniform(n, lo=0.05, hi=0.95), rng.uniform(n, 3))


def _eyes(rng, n, radius=4.0):
    z = rng.uniform(n, lo=math.sin(math.radians(5.0)))
    phi = rng.uniform(n) * 2 * math.pi
    r = torch.sqrt(1 - z * z)
    return radius * torch.stack([r * torch.cos(phi), r * torch.sin(phi), z], 1)


TAN_HALF = math.tan(math.radians(60.0) / 2)


def _frame(eye):
    """View direction, image right and image up of cameras at eye [..., 3] that look at the origin."""
    fw = _unit(-eye)
    up = torch.zeros_like(fw)
    steep = fw[..., 2].abs() > 0.99
    up[..., 2] = (~steep).double()
    up[..., 0] = steep.double()
    rt = _unit(torch.linalg.cross(fw, up))
    return fw, rt, torch.linalg.cross(rt, fw)


def _pixel_dirs(eye, px, py, width, height):
    fw, rt, up = _frame(eye)
    x = ((px + 0.5) / width * 2 - 1) * (TAN_HALF * width / height)
    y = (1 - (py + 0.5) / height * 2) * TAN_HALF
    return _unit(fw + x[..., None] * rt + y[..., None] * up)


def _view_rays(eyes, width, height, tiles):
    """All pixels of every camera, row by row or in 4 x 8 tiles."""
    py, px = torch.meshgrid(torch.arange(height, device=DEV), torch.arange(width, device=DEV), indexing="ij")
    if tiles:
        key = ((py // 8) * ((width + 3) // 4) + px // 4) * 32 + (py % 8) * 4 + px % 4
        order = torch.argsort(key.reshape(-1))
        px, py = px.reshape(-1)[order], py.reshape(-1)[order]
    px, py = px.reshape(-1).double(), py.reshape(-1).double()
    o = torch.empty(eyes.shape[0], px.numel(), 3, device=DEV)
    d = torch.empty_like(o)
    for i, e in enumerate(eyes):
        o[i] = e.float()
        d[i] = _pixel_dirs(e, px, py, width, height).float()
    return o.reshape(-1, 3), d.reshape(-1, 3)


def _pixel_rays(rng, eyes, count, width, height):
    """Random pixels of random cameras."""
    eye = eyes[(rng.uniform(count) * eyes.shape[0]).long()]
    px, py = torch.floor(rng.uniform(count) * width), torch.floor(rng.uniform(count) * height)
    return _f32(eye, _pixel_dirs(eye, px, py, width, height))


def _gbuffer(rng, points):
    """Surface points with a camera that sees their side: x, n, albedo, rough, wo."""
    p, nrm = _surface(rng, 3 * points + 64)
    p, nrm = p[(order := torch.argsort(rng.uniform(p.shape[0])))], nrm[order]
    eyes = _eyes(rng, 100)
    wo = _unit(eyes[(rng.uniform(p.shape[0]) * 100).long()] - p)
    keep = torch.nonzero((wo * nrm).sum(1) > 0.05).reshape(-1)[:points]
    return _f32(p[keep], nrm[keep], rng.uniform(points, 3, lo=0.05, hi=0.95), rng.uniform(points, lo=0.05), wo[keep])


def _env_map(rng, h):
    """An equirect HDR map [h, 2h, 3]: log-normal texels and three bright lobes."""
    w = 2 * h
    env = torch.exp(rng.normal(h, w, 1)) * rng.uniform(h, w, 3, lo=0.8, hi=1.2)
    th = (torch.arange(h, device=DEV, dtype=torch.float64) + 0.5) / h * math.pi
    ph = (torch.arange(w, device=DEV, dtype=torch.float64) + 0.5) / w * 2 * math.pi - math.pi
    dirs = torch.stack([th.sin()[:, None] * ph.cos(), th.sin()[:, None] * ph.sin(), th.cos()[:, None].expand(h, w)], -1)
    lobes = _eyes(rng, 3, 1.0)
    for c in lobes:
        ang = torch.arccos((dirs @ c).clamp(-1, 1)) / math.radians(3.0)
        env = env + 50.0 * torch.exp(-0.5 * ang ** 2)[..., None]
    return _f32(env)[0]


def _inputs(case, seed):
    """The tensors of a case, from the seed alone."""
    rng = _Rng(seed * 7919 + 17)
    kind = case["kind"]
    s = {}
    cloud = bool(case.get("cloud"))
    s["surfels"] = (_cloud if cloud else _object_scene)(rng, case["surfels"])
    if kind in ("view", "refit"):
        eyes = _eyes(rng, case.get("cams", 1), 3.0 if cloud else 4.0)
        s["rays"] = _view_rays(eyes, case["width"], case["height"], bool(case.get("tiles")))
    if kind == "refit":   # the surfels of the hierarchy's last build, a little away from today's
        m, q, sc, op, f = s["surfels"]
        s["old"] = _f32(m + 0.002 * rng.normal(*m.shape), q, sc, op, f)
    if kind == "step":
        eyes = _eyes(rng, case["cams"])
        s["rays"] = (_pixel_rays(rng, eyes, case["pixels"], case["width"], case["height"]) if case["pixels"]
                     else _view_rays(eyes, case["width"], case["height"], True))
        n = s["rays"][0].shape[0]
        g = torch.Generator(device=DEV).manual_seed(seed + 5)
        s["up"] = tuple(torch.randn(sh, generator=g, device=DEV) for sh in ((n, case["channels"]), (n,), (n,)))
    if kind == "raster":
        s["eye"] = [float(v) for v in _eyes(rng, 1)[0]]
    if kind in ("shade", "shade_step", "relight", "new_env"):
        s["gbuffer"] = _gbuffer(rng, case["points"])
        s["env"] = _env_map(rng, case.get("env_h", 256))
        s["seed"] = seed * 1000003 + 11
    if kind == "shade_step":
        s["up"] = _f32(rng.normal(case["points"], 3))[0]
    if kind == "serve":
        s["second"] = _object_scene(rng, 3 * case["surfels"])
        s["env"] = _env_map(rng, 256)
        s["eyes"] = [tuple(float(v) for v in e) for e in _eyes(rng, case["requests"])]
        s["seed"] = seed * 1000003 + 11
    return s


def _sides(case):
    """Image sides of a burst's requests, spread around the case's; renders and relights take turns."""
    return [case["side"] * (1 + i % 3) // 2 // 8 * 8 for i in range(case["requests"])]


def _requests(case, s):
    got = []
    for i, (eye, side) in enumerate(zip(s["eyes"], _sides(case))):
        if i % 2 == 0:
            got.append(serve.RenderRequest(scene=i // 2 % 2, eye=eye, width=side, height=side))
        else:
            got.append(serve.RelightRequest(scene=i // 2 % 2, eye=eye, width=side, height=side, spp=case["spp"],
                                            env=s["env"], seed=s["seed"] + i))
    return got


def _shade_params():
    return irgs.TraceParams(k=16, feat_count=3, t_min=1e-3)


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    if kind in ("step", "shade_step"):
        s["surfels"] = tuple(t.requires_grad_(True) for t in s["surfels"])
    s["scene"] = irgs.Scene(*(s["old"] if kind == "refit" else s["surfels"]), alpha_min=ALPHA_MIN)
    if kind in ("view", "step", "refit", "raster"):
        s["params"] = irgs.TraceParams(k=case.get("k", 16), feat_count=case["channels"])
    if kind == "raster":
        s["cam"] = serve.make_camera(s["eye"], case["width"], case["height"])
        s["params"] = irgs.TraceParams(feat_count=case["channels"], t_min=0.2)
    if kind == "shade_step":
        s["leaves"] = [t.requires_grad_(True) for t in (s["gbuffer"][2], s["gbuffer"][3], s["env"])]
    if kind == "relight":
        s["map"] = irgs.EnvMap(s["env"])
    if kind == "serve":
        s["scenes"] = [s["scene"], irgs.Scene(*s["second"], alpha_min=ALPHA_MIN)]
        s["server"] = serve.Server(s["scenes"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "view":
        return irgs.trace_forward(s["scene"], *s["rays"], s["params"])
    if kind == "step":
        s["scene"].update()   # the optimiser wrote new values into the scene's tensors
        feat, depth, opacity, n_hits = irgs.trace(s["scene"], *s["rays"], s["params"], case["saved_hits"])
        g = torch.autograd.grad((feat, depth, opacity), s["surfels"], s["up"])
        return {"feat": feat.detach(), "depth": depth.detach(), "opacity": opacity.detach(), "n_hits": n_hits,
                "means": g[0], "quats": g[1], "scales": g[2], "op": g[3], "features": g[4]}
    if kind == "refit":
        s["scene"].refit(*s["surfels"])
        return irgs.trace_forward(s["scene"], *s["rays"], s["params"])
    if kind == "raster":
        return irgs.rasterize(s["scene"], s["cam"], s["params"])
    if kind == "shade":
        x, n, albedo, rough, wo = s["gbuffer"]
        return irgs.shade_mc(s["scene"], x, n, albedo, rough, wo, s["env"], case["diffuse"], case["spec"], s["seed"],
                             _shade_params(), want_aux=case["aux"], mode=case["mode"])
    if kind == "shade_step":
        x, n, albedo, rough, wo = s["gbuffer"]
        rgb = irgs.shade(s["scene"], x, n, albedo, rough, wo, s["env"], case["diffuse"], case["spec"], s["seed"],
                         _shade_params(), mode=case["mode"])
        g = torch.autograd.grad(rgb, list(s["surfels"]) + s["leaves"], s["up"])
        return dict(zip(("means", "quats", "scales", "op", "features", "albedo", "rough", "env"), g), rgb=rgb.detach())
    if kind in ("relight", "new_env"):
        x, n, albedo, rough, wo = s["gbuffer"]
        env = s["map"] if kind == "relight" else irgs.EnvMap(s["env"])
        params = irgs.TraceParams(k=16, feat_offset=3, feat_count=7, t_min=1e-3)
        return irgs.relight(s["scene"], env, x, n, albedo, rough, wo, case["samples"], s["seed"], params, want_aux=True)
    server = s["server"]
    handles = [server.submit(r) for r in _requests(case, s)]
    server.run_until_idle()
    server.finished.clear()
    return [h.out if "feat" in h.out else {"rgb": h.out["rgb"], **serve.gbuffer_views(h.out["gbuffer"], h.request.pixels())}
            for h in handles]


def work(case):
    """Bytes that have to move (each input and output once) and arithmetic of
    the blended hits alone: 45 operations a test, two a blended channel, and
    one descent of the hierarchy a ray."""
    kind, n = case["kind"], case["surfels"]
    scene = 4 * n * 20
    descent = 40 * math.ceil(math.log2(n))

    def ray(hits, channels):
        return hits * (48 + 2 * (channels + 2)) + descent

    if kind in ("view", "refit", "raster"):
        r = case["width"] * case["height"] * case.get("cams", 1)
        b = scene * (2 if kind == "refit" else 1) + r * (4 * (case["channels"] + 3) + (0 if kind == "raster" else 24))
        return {"bytes": b, "flops": r * ray(22, case["channels"])}
    if kind == "step":
        r = case["pixels"] or case["width"] * case["height"] * case["cams"]
        return {"bytes": 3 * scene + r * (24 + 8 * (case["channels"] + 3)), "flops": 4 * r * ray(22, case["channels"])}
    if kind == "serve":
        px = [side * side for side in _sides(case)]
        shade = sum(px[1::2]) * case["spp"]
        return {"bytes": 4 * scene + 60 * sum(px), "flops": sum(px) * ray(22, 10) + shade * ray(9, 3)}
    p = case["points"]
    env = 12 * 2 * case.get("env_h", 256) ** 2
    if kind in ("relight", "new_env"):
        r, f = p * case["samples"], 0
        if kind == "new_env":   # half the sphere of texels, for each texel of the pre-integrated maps
            f = case["env_h"] ** 2 * (5 * 64 * 128 + 32 * 64) * 12
        return {"bytes": scene + env + p * 72, "flops": f + r * ray(18, 7)}
    r = p * (case["diffuse"] + case["spec"])
    k = 4 if kind == "shade_step" else 1
    return {"bytes": (scene + env) * (2 if k == 4 else 1) + p * (44 + 28 * (1 if k == 1 else 2)), "flops": k * r * ray(9, 3)}


# ---------------------------------------------------------------------------
# The same outputs from the definitions, in 64 bits

T_MIN = float(np.float32(1e-4))
A_MIN = float(np.float32(ALPHA_MIN))
A_MAX = float(np.float32(0.99))
MOST_RAYS = 7_000_000


def _tangents(q):
    w, x, y, z = _unit(q).unbind(-1)
    tu = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + w * z), 2 * (x * z - w * y)], -1)
    tv = torch.stack([2 * (x * y - w * z), 1 - 2 * (x * x + z * z), 2 * (y * z + w * x)], -1)
    nn = torch.stack([2 * (x * z + w * y), 2 * (y * z - w * x), 1 - 2 * (x * x + y * y)], -1)
    return tu, tv, nn


class _Exact:
    """Every hit of a set of rays, found through bounding spheres."""

    def __init__(self, surfels, inflate=None):
        self.p = [t.detach().double() for t in surfels]
        mu, q, sc, op, _ = self.p
        self.rc2 = torch.clamp(2 * torch.log(op / A_MIN), max=9.0)
        rad = torch.sqrt(self.rc2.clamp(min=0.0)) * sc.max(1).values * 1.001 + 1e-5
        self.rad = rad if inflate is None else rad + inflate
        cell = ((mu - mu.min(0).values) / (mu.max(0).values - mu.min(0).values + 1e-12) * 1023).long()
        key = torch.zeros(mu.shape[0], device=DEV, dtype=torch.int64)
        for b in range(10):
            for a in range(3):
                key |= ((cell[:, a] >> b) & 1) << (3 * b + a)
        order = torch.argsort(key)
        pad = -order.numel() % 32
        self.group = torch.cat([order, order[-1:].expand(pad)]).reshape(-1, 32)
        self.real = torch.arange(self.group.numel(), device=DEV).reshape(-1, 32) < order.numel()
        box = mu[self.group]
        self.c = (box.min(1).values + box.max(1).values) / 2
        self.r = ((box - self.c[:, None]).norm(dim=2) + self.rad[self.group]).max(1).values

    def near(self, o, d):
        """(ray, surfel) of every surfel whose sphere the ray's line crosses ahead of it."""
        of, df, c, r = o.float(), _unit(d).float(), self.c.float(), self.r.float()
        mid = c.mean(0)
        c, oc = c - mid, of - mid
        t = df @ c.T - (oc * df).sum(1)[:, None]
        d2 = (c * c).sum(1)[None] + (oc * oc).sum(1)[:, None] - 2 * (oc @ c.T) - t * t
        ray, grp = torch.nonzero((d2 <= r * r + 2e-4) & (t > -r - 1e-3), as_tuple=True)
        out = []
        mu, rad = self.p[0].float(), self.rad.float()
        for a in range(0, ray.numel(), 1 << 21):
            g = grp[a:a + (1 << 21)]
            sid, rid = self.group[g], ray[a:a + (1 << 21), None]
            w = mu[sid] - of[rid]
            dd = df[rid]
            t = (w * dd).sum(2)
            ok = ((w - t[..., None] * dd).norm(dim=2) <= rad[sid] + 1e-5) & self.real[g]
            i, j = torch.nonzero(ok, as_tuple=True)
            out.append(torch.stack([rid[i, 0], sid[i, j]]))
        return torch.cat(out, 1) if out else torch.zeros(2, 0, device=DEV, dtype=torch.int64)

    def geometry(self, o, d, ray, sid, p=None):
        """tau and the squared local radius of each pair (differentiable in p)."""
        mu, q, sc = (self.p if p is None else p)[:3]
        tu, tv, nn = _tangents(q[sid])
        oo, dd = o[ray], d[ray]
        den = (nn * dd).sum(1)
        tau = (nn * (mu[sid] - oo)).sum(1) / den
        e = oo + tau[:, None] * dd - mu[sid]
        u, v = (e * tu).sum(1) / sc[sid, 0], (e * tv).sum(1) / sc[sid, 1]
        return tau, u * u + v * v, den

    def hits(self, o, d, t_min):
        """Accepted (ray, surfel) pairs in blend order."""
        ray, sid = self.near(o, d)
        tau, rho2, den = self.geometry(o, d, ray, sid)
        alpha = torch.clamp(self.p[3][sid] * torch.exp(-rho2 / 2), max=A_MAX)
        ok = (rho2 <= self.rc2[sid]) & (alpha >= A_MIN) & (tau > t_min) & (den.abs() >= 1e-8 * d[ray].norm(dim=1))
        ray, sid, tau = ray[ok], sid[ok], tau[ok]
        return self.sort(ray, sid, tau)

    @staticmethod
    def sort(ray, sid, depth):
        i = torch.argsort(sid, stable=True)
        i = i[torch.argsort(depth[i], stable=True)]
        i = i[torch.argsort(ray[i], stable=True)]
        return ray[i], sid[i]


def _blend(rays, ray, alpha, depth, feats):
    """Front-to-back blend of sorted pairs: feat, depth, opacity, hits."""
    count = torch.bincount(ray, minlength=rays)
    start = torch.cumsum(count, 0) - count
    width = max(1, int(count.max()) if count.numel() else 1)
    slot = ray * width + torch.arange(ray.numel(), device=DEV) - start[ray]
    grid = lambda v: torch.zeros(rays * width, device=DEV, dtype=torch.float64).index_copy(0, slot, v).reshape(rays, width)
    a = grid(alpha)
    through = torch.cumprod(1 - a, 1)
    before = torch.cat([torch.ones(rays, 1, device=DEV, dtype=torch.float64), through[:, :-1]], 1)
    live = (before >= T_MIN).detach()
    w = (before * a * live).reshape(-1)[slot]
    add = lambda v: torch.zeros((rays,) + v.shape[1:], device=DEV, dtype=torch.float64).index_add(0, ray, v)
    n_hits = add(live.reshape(-1)[slot].double())
    last = torch.cumprod(torch.where(live, 1 - a, torch.ones_like(a)), 1)[:, -1]
    return add(w[:, None] * feats), add(w * depth), 1 - last, n_hits


def _trace64(ex, o, d, channels, offset=0, t_min=0.0, up=None, step=None):
    """Trace64 of rays (o, d): feat, depth, opacity, n_hits; with `up` also the
    gradients of the surfel tensors."""
    o, d = o.double(), d.double()
    step = step or max(256, min(1 << 15, int(3e8 / ex.group.shape[0])))
    outs, grads = [], None
    p = ex.p
    if up is not None:
        p = [t.clone().requires_grad_(True) for t in ex.p]
        grads = [torch.zeros_like(t) for t in p]
    for a in range(0, o.shape[0], step):
        oc, dc = o[a:a + step], d[a:a + step]
        with torch.no_grad():
            ray, sid = ex.hits(oc, dc, t_min)
        with torch.set_grad_enabled(up is not None):
            tau, rho2, _ = ex.geometry(oc, dc, ray, sid, p)
            alpha = torch.clamp(p[3][sid] * torch.exp(-rho2 / 2), max=A_MAX)
            out = _blend(oc.shape[0], ray, alpha, tau, p[4][sid, offset:offset + channels])
            if up is not None:
                got = torch.autograd.grad(out[:3], p, [u[a:a + step].double() for u in up])
                for g, x in zip(grads, got):
                    g += x
        outs.append([t.detach() for t in out])
    return [torch.cat(t) for t in zip(*outs)], grads


def _uniforms(seed, first, count):
    """SplitMix64 outputs first .. first + count of the stream, as [0, 1) values."""
    def signed(v):
        v &= (1 << 64) - 1
        return v - (1 << 64) if v >= 1 << 63 else v

    def shift(z, b):
        return (z >> b) & ((1 << (64 - b)) - 1)

    z = (torch.arange(first, first + count, device=DEV) + 1) * signed(0x9E3779B97F4A7C15) + signed(seed)
    z = (z ^ shift(z, 30)) * signed(0xBF58476D1CE4E5B9)
    z = (z ^ shift(z, 27)) * signed(0x94D049BB133111EB)
    z = z ^ shift(z, 31)
    return shift(z, 40).double() / 16777216.0


def _lookup(img, w):
    """Bilinear equirect lookup (differentiable in img)."""
    h, wd = img.shape[:2]
    x = (torch.atan2(w[..., 1], w[..., 0]) + math.pi) / (2 * math.pi) * wd - 0.5
    y = torch.atan2(torch.sqrt(w[..., 0] ** 2 + w[..., 1] ** 2), w[..., 2]) / math.pi * h - 0.5
    x0, y0 = torch.floor(x), torch.floor(y)
    fx, fy = (x - x0)[..., None], (y - y0)[..., None]
    c = [(x0.long() + i) % wd for i in (0, 1)]
    r = [(y0.long() + i).clamp(0, h - 1) for i in (0, 1)]
    flat = img.reshape(-1, img.shape[2])
    top = (1 - fx) * flat[r[0] * wd + c[0]] + fx * flat[r[0] * wd + c[1]]
    low = (1 - fx) * flat[r[1] * wd + c[0]] + fx * flat[r[1] * wd + c[1]]
    return (1 - fy) * top + fy * low


def _dot(a, b):
    return (a * b).sum(-1)


def _point_frame(n, wo):
    n, wo = _unit(n.double()), _unit(wo.double())
    no = _dot(n, wo)
    n = torch.where((no <= 0)[:, None], -n, n)
    s = torch.where(n[:, 2] >= 0, 1.0, -1.0).double()
    a = -1 / (s + n[:, 2])
    b = n[:, 0] * n[:, 1] * a
    b1 = torch.stack([1 + s * n[:, 0] ** 2 * a, s * b, -s * n[:, 0]], 1)
    b2 = torch.stack([b, s + n[:, 1] ** 2 * a, -n[:, 1]], 1)
    return n, wo, no.abs(), b1, b2


def _ggx(r, nh, oh, ni, no):
    """ln of D G1(w_i) G1(w_o), and the Fresnel term."""
    a2, k = r ** 4, r ** 2 / 2
    ln = torch.log(a2 / (math.pi * ((1 - nh ** 2) + nh ** 2 * a2) ** 2))
    ln = ln + torch.log(ni / (ni * (1 - k) + k)) + torch.log(no / (no * (1 - k) + k))
    return ln, 0.04 + 0.96 * (1 - oh) ** 5


def _shade64(case, s, up=None):
    x, n, albedo, rough, wo = (t.detach() for t in s["gbuffer"])
    P, nd, ns = case["points"], case["diffuse"], case["spec"]
    S, split = nd + ns, case["mode"] == "split"
    ex = _Exact(s["surfels"])
    leaves = [t.double().clone().requires_grad_(up is not None) for t in (albedo, rough, s["env"].detach())]
    total = {"rgb": [], "vis": [], "ind": []}
    scene_g = [torch.zeros_like(t) for t in ex.p]
    leaf_g = [torch.zeros_like(t) for t in leaves]
    step = max(1, int(3e6 / S))
    for a in range(0, P, step):
        sl = slice(a, min(P, a + step))
        m = sl.stop - a
        u = _uniforms(s["seed"], a * S * 2, m * S * 2).reshape(m, S, 2)
        N, W, no, b1, b2 = _point_frame(n[sl], wo[sl])
        N, W, b1, b2, no = N[:, None], W[:, None], b1[:, None], b2[:, None], no[:, None]
        r0 = rough[sl].double()[:, None]
        c, q = torch.cos(2 * math.pi * u[..., 1]), torch.sin(2 * math.pi * u[..., 1])
        place = lambda rr, z: _unit((rr * c)[..., None] * b1 + (rr * q)[..., None] * b2 + z[..., None] * N)
        is_d = torch.zeros(m, S, device=DEV, dtype=torch.bool)
        if split:
            is_d[:, :nd] = True
            a2 = r0 ** 4
            inv = 1 / (a2 * u[..., 0] + 1 - u[..., 0])
            h = place(torch.sqrt(a2 * u[..., 0] * inv), torch.sqrt((1 - u[..., 0]) * inv))
            spec = _unit(2 * _dot(W, h)[..., None] * h - W)
            wi = torch.where(is_d[..., None], place(torch.sqrt(u[..., 0]), torch.sqrt(1 - u[..., 0])), spec)
        else:
            z = (torch.arange(S, device=DEV)[None] + u[..., 0]) / S
            wi = place(torch.sqrt((1 - z * z).clamp(min=0)), z)
            h = _unit(wi + W)
        oh, nh, ni = _dot(W, h), _dot(N, h), _dot(N, wi)
        ok = is_d | ((oh > 0) & (ni > 0)) if split else ni > 0
        idx = torch.nonzero(ok.reshape(-1)).reshape(-1)
        ro = x[sl].double()[:, None].expand(m, S, 3).reshape(-1, 3)[idx]
        rd = wi.reshape(-1, 3)[idx]

        def estimate(C, V, lv):
            al, rr, env = lv[0][sl], lv[1][sl], lv[2]
            at = lambda v: v.expand(m, S).reshape(-1)[idx]
            Li = V[:, None] * _lookup(env, rd) + C
            dif, pt = at(is_d), idx // S
            safe = lambda v: torch.where(dif, torch.ones_like(v), v)
            nh_, oh_, ni_, no_ = safe(at(nh)), safe(at(oh)), safe(at(ni)), at(no)
            ln, F = _ggx(rr[pt], nh_, oh_, ni_, no_)
            if split:
                k = rough[sl].double()[pt] ** 2 / 2
                G = ni_ / (ni_ * (1 - k) + k) * (no_ / (no_ * (1 - k) + k))
                ws = F * G * oh_ / (no_ * nh_) / max(1, ns) * torch.exp(ln - ln.detach())
                wgt = torch.where(dif[:, None], al[pt] / max(1, nd), ws[:, None].expand(-1, 3))
            else:
                wgt = 2 * al[pt] * ni_[:, None] / S + (2 * math.pi / S * torch.exp(ln) * F / (4 * no_))[:, None]
            return torch.zeros(m, 3, device=DEV, dtype=torch.float64).index_add(0, pt, wgt * Li)

        tm = float(np.float32(1e-3))
        (C, _, O, _), _ = _trace64(ex, ro, rd, 3, t_min=tm)
        total["rgb"].append(estimate(C, 1 - O, leaves).detach())
        over = torch.nonzero((is_d if split else ok).reshape(-1)[idx]).reshape(-1)
        pt = idx[over] // S
        cnt = torch.bincount(pt, minlength=m).clamp(min=1).double()
        mean = lambda v: torch.zeros((m,) + v.shape[1:], device=DEV, dtype=torch.float64).index_add(0, pt, v)
        total["vis"].append(mean((1 - O)[over]) / cnt)
        total["ind"].append(mean(C[over]) / cnt[:, None])
        if up is not None:
            C, V = C.requires_grad_(True), (1 - O).requires_grad_(True)
            g = torch.autograd.grad(estimate(C, V, leaves), [C, V] + leaves, up[sl].double(), allow_unused=True)
            for t, v in zip(leaf_g, g[2:]):
                t += 0 if v is None else v
            _, gs = _trace64(ex, ro, rd, 3, t_min=tm, up=(g[0], torch.zeros_like(V), -g[1]))
            for t, v in zip(scene_g, gs):
                t += v
    out = {k: torch.cat(v) for k, v in total.items()}
    return out, scene_g + leaf_g


def _maps64(env):
    """Irradiance, prefiltered levels, BRDF table and sampling cdfs of an environment."""
    H, W = env.shape[:2]
    E = env.double()
    f = lambda n: torch.arange(n, device=DEV, dtype=torch.float64) + 0.5

    def dirs(h, w):
        th, ph = f(h) / h * math.pi, f(w) / w * 2 * math.pi - math.pi
        return torch.stack([th.sin()[:, None] * ph.cos(), th.sin()[:, None] * ph.sin(), th.cos()[:, None].expand(h, w)], -1).reshape(-1, 3)

    edge = torch.arange(H + 1, device=DEV, dtype=torch.float64) / H * math.pi
    area = ((torch.cos(edge[:-1]) - torch.cos(edge[1:])) * 2 * math.pi / W)[:, None].expand(H, W).reshape(-1)
    wt, Ef = dirs(H, W), E.reshape(-1, 3)
    val = torch.cat([Ef, torch.ones_like(Ef[:, :1])], 1) * area[:, None]
    irr = torch.cat([(d @ wt.T).clamp(min=0) @ val[:, :3] for d in dirs(32, 64).split(256)]) / math.pi
    levels = [E]
    sums = [[] for _ in range(5)]
    for d in dirs(64, 128).split(256):
        cs = (d @ wt.T).clamp(min=0)
        x2 = ((d[:, None] - wt[None]) ** 2).sum(2) / 4    # |R x h|^2 = |w - R|^2 / 4, (R.h)^2 = 1 - that
        for l in range(1, 6):
            a2 = (l / 5) ** 4
            g = (cs * a2 / (x2 + (1 - x2) * a2) ** 2) @ val
            sums[l - 1].append(g[:, :3] / g[:, 3:])
    levels += [torch.cat(v).reshape(64, 128, 3) for v in sums]
    mu, rho = f(32)[:, None, None] / 32, f(32)[None, :, None] / 32
    k = torch.arange(1024, device=DEV)
    rev = sum(((k >> b) & 1).double() / (2 << b) for b in range(10))[None, None]
    u1 = ((k.double() + 0.5) / 1024)[None, None]
    a2, kk = rho ** 4, rho ** 2 / 2
    inv = 1 / (a2 * u1 + 1 - u1)
    ct, st = torch.sqrt((1 - u1) * inv), torch.sqrt(a2 * u1 * inv)
    vh = torch.sqrt(1 - mu * mu) * st * torch.cos(2 * math.pi * rev) + mu * ct
    lz = 2 * vh * ct - mu
    gv = lz / (lz * (1 - kk) + kk) * (mu / (mu * (1 - kk) + kk)) * vh / (ct * mu) * ((lz > 0) & (vh > 0))
    fc = (1 - vh) ** 5
    lut = torch.stack([((1 - fc) * gv).mean(2), (fc * gv).mean(2)], -1)
    lum = (0.2126 * E[..., 0] + 0.7152 * E[..., 1] + 0.0722 * E[..., 2]) * torch.sin(f(H) / H * math.pi)[:, None]
    z = lambda t: torch.cat([torch.zeros_like(t[..., :1]), torch.cumsum(t, -1)], -1)
    col = z(lum)
    return {"levels": levels, "irr": irr.reshape(32, 64, 3), "lut": lut, "col": col, "row": z(col[:, -1])}


def _relight64(case, s):
    x, n, albedo, rough, wo = s["gbuffer"]
    P, S = case["points"], case["samples"]
    M, ex = _maps64(s["env"]), _Exact(s["surfels"])
    H, W = s["env"].shape[:2]
    out = {"rgb": [], "vis": [], "ind": []}
    step = max(1, int(3e6 / S))
    for a in range(0, P, step):
        sl = slice(a, min(P, a + step))
        m = sl.stop - a
        u = _uniforms(s["seed"], a * S * 2, m * S * 2).reshape(-1, 2)
        total = M["row"][H]
        t1 = u[:, 0] * total
        r = (torch.searchsorted(M["row"], t1, right=True) - 1).clamp(0, H - 1)
        cc = M["col"][r]
        t2 = u[:, 1] * cc[:, W]
        c = (torch.searchsorted(cc, t2[:, None], right=True) - 1).reshape(-1).clamp(0, W - 1)
        c0, c1 = cc.gather(1, c[:, None])[:, 0], cc.gather(1, c[:, None] + 1)[:, 0]
        th = (r + (t1 - M["row"][r]) / cc[:, W]) / H * math.pi
        ph = (c + (t2 - c0) / (c1 - c0)) / W * 2 * math.pi - math.pi
        w = torch.stack([torch.sin(th) * torch.cos(ph), torch.sin(th) * torch.sin(ph), torch.cos(th)], 1)
        pdf = (c1 - c0) / total * W * H / (2 * math.pi ** 2 * torch.sin(th))
        del cc
        pt = torch.arange(m, device=DEV).repeat_interleave(S)
        (C, _, O, _), _ = _trace64(ex, x[sl].double()[pt], w, 7, offset=3, t_min=float(np.float32(1e-3)))
        v, V = -w, 1 - O
        So = O.clamp(min=1e-300)[:, None]
        Rr = (C[:, 3] / So[:, 0])
        Nr = C[:, 4:7]
        Nr = torch.where((_dot(Nr, Nr) > 1e-24)[:, None], Nr / Nr.norm(dim=1, keepdim=True).clamp(min=1e-300), v)
        Nr = torch.where((_dot(Nr, v) < 0)[:, None], -Nr, Nr)
        mu = _dot(Nr, v).clamp(max=1.0)
        refl = 2 * mu[:, None] * Nr - v
        t = Rr.clamp(0, 1) * 5
        l0 = torch.floor(t).long().clamp(max=4)
        fr = (t - l0)[:, None]
        look = torch.stack([_lookup(im, refl) for im in M["levels"]], 1)
        pick = lambda l: look.gather(1, l[:, None, None].expand(-1, 1, 3))[:, 0]
        pf = (1 - fr) * pick(l0) + fr * pick(l0 + 1)
        gx, gy = (mu * 32 - 0.5).clamp(0, 31), (Rr * 32 - 0.5).clamp(0, 31)
        i0, j0 = torch.floor(gx).long().clamp(max=30), torch.floor(gy).long().clamp(max=30)
        fx, fy = (gx - i0)[:, None], (gy - j0)[:, None]
        L = M["lut"]
        ab = (1 - fx) * ((1 - fy) * L[i0, j0] + fy * L[i0, j0 + 1]) + fx * ((1 - fy) * L[i0 + 1, j0] + fy * L[i0 + 1, j0 + 1])
        ind = O[:, None] * (C[:, :3] / So * _lookup(M["irr"], Nr) + pf * (0.04 * ab[:, :1] + ab[:, 1:]))
        ind = torch.where((O > 0)[:, None], ind, torch.zeros_like(ind))
        N, Wo, no, _, _ = _point_frame(n[sl], wo[sl])
        N, Wo, no, r0 = N[pt], Wo[pt], no[pt], rough[sl].double()[pt]
        ni = _dot(N, w)
        h = _unit(w + Wo)
        up = ni > 0
        one = torch.ones_like(ni)
        ln, F = _ggx(r0, _dot(N, h), _dot(Wo, h), torch.where(up, ni, one), no)
        f = albedo[sl].double()[pt] / math.pi * ni[:, None] + (torch.exp(ln) * F / (4 * no))[:, None]
        Li = V[:, None] * _lookup(M["levels"][0], w) + ind
        term = torch.where(up[:, None], f * Li / pdf[:, None], torch.zeros_like(Li))
        mean = lambda q: q.reshape((m, S) + q.shape[1:]).mean(1)
        for k, q in (("rgb", term), ("vis", V), ("ind", ind)):
            out[k].append(mean(q))
    return {k: torch.cat(v) for k, v in out.items()}


def _raster64(case, s):
    W, H = case["width"], case["height"]
    eye = torch.tensor(s["eye"], device=DEV, dtype=torch.float64)
    fw, rt, up = _frame(eye)
    eye, fw, rt, up = (t.float().double() for t in (eye, fw, rt, up))
    tan = float(np.float32(TAN_HALF))
    mu = s["surfels"][0].double()
    px_size = 2 * tan / H
    ex = _Exact(s["surfels"], inflate=3.2 * px_size * 2 * (mu - eye).norm(dim=1))
    q = mu - eye
    z = q @ fw
    cx = ((q @ rt) / z / (tan * W / H) + 1) * 0.5 * W - 0.5
    cy = (1 - (q @ up) / z / tan) * 0.5 * H - 0.5
    py, px = torch.meshgrid(torch.arange(H, device=DEV).double(), torch.arange(W, device=DEV).double(), indexing="ij")
    px, py = px.reshape(-1), py.reshape(-1)
    d = _unit(fw + (((px + 0.5) / W * 2 - 1) * tan * W / H)[:, None] * rt + ((1 - (py + 0.5) / H * 2) * tan)[:, None] * up)
    outs = []
    near = float(np.float32(0.2))
    for a in range(0, W * H, 1 << 13):
        sl = slice(a, a + (1 << 13))
        dc = d[sl]
        oc = eye.expand(dc.shape[0], 3)
        ray, sid = ex.near(oc, dc)
        tau, rho3, den = ex.geometry(oc, dc, ray, sid)
        hit = (den.abs() >= 1e-8) & (tau > 0)
        rho3 = torch.where(hit, rho3, torch.full_like(rho3, math.inf))
        rho2 = 2 * ((px[sl][ray] - cx[sid]) ** 2 + (py[sl][ray] - cy[sid]) ** 2)
        rho = torch.minimum(rho3, rho2)
        alpha = torch.clamp(ex.p[3][sid] * torch.exp(-rho / 2), max=A_MAX)
        depth = torch.where(rho3 <= rho2, tau, ((mu - eye)[sid] * dc[ray]).sum(1))
        ok = (rho <= ex.rc2[sid]) & (alpha >= A_MIN) & (z[sid] > near)
        ray, sid, alpha, depth = ray[ok], sid[ok], alpha[ok], depth[ok]
        i = torch.argsort(sid, stable=True)
        i = i[torch.argsort(z[sid[i]], stable=True)]
        i = i[torch.argsort(ray[i], stable=True)]
        ray, sid, alpha, depth = ray[i], sid[i], alpha[i], depth[i]
        outs.append(_blend(dc.shape[0], ray, alpha, depth, ex.p[4][sid, :case["channels"]]))
    return [torch.cat(t) for t in zip(*outs)]


def _serve64(case, s):
    """The renders; the relights chain a thresholded G-buffer into shading and have no single value."""
    got = []
    scenes = [_Exact(s["surfels"]), _Exact(s["second"])]
    for j, (eye, side) in enumerate(zip(s["eyes"], _sides(case))):
        if j % 2:
            got.append(None)
            continue
        P = side * side
        eye = torch.tensor(eye, device=DEV, dtype=torch.float64)
        tw, th = 4, 8
        i = torch.arange(P, device=DEV)
        t, k = i // (tw * th), i % (tw * th)
        across = side // tw
        px, py = (t % across) * tw + k % tw, (t // across) * th + k // tw
        d = _pixel_dirs(eye, px.double(), py.double(), side, side)
        (feat, depth, opacity, _), _ = _trace64(scenes[j // 2 % 2], eye.expand(P, 3), d, 10)
        got.append({"feat": feat, "depth": depth, "opacity": opacity})
    return got


def exact(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    if kind in ("view", "refit", "step"):
        up = s.get("up")
        if s["rays"][0].shape[0] > (1_500_000 if up is None else 400_000):
            return None
        (feat, depth, opacity, _), g = _trace64(_Exact(s["surfels"]), *s["rays"], case["channels"], up=up)
        out = {"feat": feat, "depth": depth, "opacity": opacity, "n_hits": None}
        return out if g is None else dict(out, **dict(zip(("means", "quats", "scales", "op", "features"), g)))
    if kind == "raster":
        feat, depth, opacity, _ = _raster64(case, s)
        return {"feat": feat, "depth": depth, "opacity": opacity, "n_hits": None}
    if kind == "serve":
        return _serve64(case, s)
    if kind in ("relight", "new_env"):
        return _relight64(case, s) if case["points"] * case["samples"] <= MOST_RAYS else None
    rays = case["points"] * (case["diffuse"] + case["spec"])
    if rays > (MOST_RAYS if kind == "shade" else 1_500_000):
        return None
    out, g = _shade64(case, s, s.get("up"))
    if kind == "shade":
        return out if case["aux"] else {"rgb": out["rgb"]}
    return dict(zip(("means", "quats", "scales", "op", "features", "albedo", "rough", "env"), g), rgb=out["rgb"])
