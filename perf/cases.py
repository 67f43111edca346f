"""The performance cases of the renderer: what is timed, over which ranges, and what its results should be.

A case is a dict of plain values.  Its kind is what a program asks for:

  closest, any  a ray query (Scene.trace_closest / Scene.trace_any) over n rays of one sort:
                  pick    a few rays from the eye (selecting an object, a focus distance, a light meter)
                  camera  one ray per pixel of an image, row by row
                  bounce  diffuse bounces: from points on the scene's surfaces into the upper hemisphere, unbounded
                  sun     shadow rays: from such points toward the sun
                  ao      ambient occlusion: from such points into the upper hemisphere, of finite reach
  frame         one image (Scene.render), optionally a crop of a larger frame, with per-face textures, with key lights
  progressive   one sample per pixel of an image, added to the frames before it (Scene.render, api.accumulate)
  views         several small images in one captured graph (api.RenderGraph)
  train         an image, its loss against a target and the albedo's gradient (Scene.render, api.l2_loss, Scene.adjoint)

Scenes are the seeded ones of inputs.py: tiny (1 mesh, 256 instances), mid (5.7 M quads, 100 k instances; fits L2) and
island (the Moana-scale generator at a twentieth: 13 M quads, 2 M instances; larger than L2).  A program builds its scene
once and keeps it, so a process builds each once here; the seed makes the rays, cameras, random streams, albedo,
textures, lights and targets.
"""
import math

import numpy as np
import torch

from paper_2001_02620_gb300 import api, inputs

DEV = "cuda"
ISLAND_SCALE = 0.05
SUN = inputs.MID_SUN_DIR


def listed():
    return [
        # the smallest call: what the cursor points at, a handful of rays and one launch
        {"name": "pick_tiny", "kind": "closest", "scene": "tiny", "rays": "pick", "n": 37},
        # an image's visibility: coherent rays, odd image size
        {"name": "closest_camera_mid", "kind": "closest", "scene": "mid", "rays": "camera", "n": 1021 * 773, "w": 1021},
        # indirect light gathered by a program's own integrator: incoherent rays
        {"name": "closest_bounce_mid", "kind": "closest", "scene": "mid", "rays": "bounce", "n": 2000003},
        # shadow tests of a program's own integrator, parallel and unbounded
        {"name": "any_sun_mid", "kind": "any", "scene": "mid", "rays": "sun", "n": 1500007},
        # ambient occlusion of finite reach on a scene that does not fit L2
        {"name": "any_ao_island", "kind": "any", "scene": "island", "rays": "ao", "n": 1000003, "reach": 40.0},
        # a thumbnail: a whole render of a few thousand paths, where launches and the longest path count
        {"name": "frame_thumb_tiny", "kind": "frame", "scene": "tiny", "w": 61, "h": 47, "spp": 1, "depth": 3, "sun": True},
        # the interactive loop: one sample per pixel and frame, accumulated
        {"name": "progressive_mid", "kind": "progressive", "scene": "mid", "w": 1280, "h": 720, "depth": 5, "sun": True},
        # the benchmark's mid frame
        {"name": "frame_mid", "kind": "frame", "scene": "mid", "w": 1024, "h": 1024, "spp": 4, "depth": 5, "sun": True},
        # the benchmark's Moana-scale frame on the smaller island
        {"name": "frame_island", "kind": "frame", "scene": "island", "w": 960, "h": 540, "spp": 16, "depth": 8, "sun": True},
        # one worker's tile of a frame with textures and key lights
        {"name": "tile_rich_mid", "kind": "frame", "scene": "mid", "w": 1920, "h": 1080, "spp": 4, "depth": 5, "sun": True,
         "crop_x": 637, "crop_y": 411, "crop_w": 613, "crop_h": 389, "tex": 4, "lights": 23},
        # many small uneven views (a contact sheet, light probes) replayed as one graph
        {"name": "views_mid", "kind": "views", "scene": "mid", "n_views": 24, "side": 96, "spp": 3, "depth": 5, "sun": True},
        # a step of inverse rendering
        {"name": "train_mid", "kind": "train", "scene": "mid", "w": 512, "h": 512, "spp": 8, "depth": 4, "sun": True},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


#: Most paths times depth of a drawn case, and most rays of a drawn query.
MOST_PATHS, MOST_RAYS = 24_000_000, 4_000_000


def draw(rng):
    kind = rng.choice(["closest", "closest", "any", "any", "frame", "frame", "progressive", "views", "train"])
    scene = rng.choice(["tiny", "mid", "mid", "island"])
    if kind in ("closest", "any"):
        rays = rng.choice(["pick", "camera", "bounce", "sun", "ao"])
        c = {"kind": kind, "scene": scene, "rays": rays, "n": _log(rng, 1, 256) if rays == "pick" else _log(rng, 500, MOST_RAYS)}
        if rays == "camera":
            c["w"] = rng.randint(1, max(1, int(1.5 * math.sqrt(c["n"]))))
        if rays == "ao":
            c["reach"] = round(rng.uniform(2.0, 200.0), 2)
        return c
    depth = rng.randint(1, 8)
    c = {"kind": kind, "scene": scene, "depth": depth, "sun": rng.random() < 0.75}
    if kind == "views":
        return {**c, "n_views": rng.randint(2, 70), "side": _log(rng, 16, 160), "spp": rng.randint(1, 4)}
    spp = 1 if kind == "progressive" else rng.choice([1, 1, 2, 3, 4, 8, 16])
    most = MOST_PATHS // (depth * spp * (3 if kind == "train" else 1))
    w = _log(rng, 16, 1920)
    h = min(max(8, int(w * rng.uniform(0.4, 1.2))), max(8, most // w))
    c.update(w=w, h=h)
    if kind != "progressive":
        c["spp"] = spp
    if kind == "frame":
        if rng.random() < 0.3 and w >= 32 and h >= 32:
            cw, ch = rng.randint(8, w), rng.randint(8, h)
            c.update(crop_x=rng.randint(0, w - cw), crop_y=rng.randint(0, h - ch), crop_w=cw, crop_h=ch)
        if rng.random() < 0.25:
            c["tex"] = rng.choice([1, 2, 4])
        if rng.random() < 0.25:
            c["lights"] = rng.randint(1, 32)
    return c


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------
_scenes = {}


class _Built:
    """A scene, its handle, and its vertices on the GPU to start rays from."""

    def __init__(self, name):
        make = {"tiny": inputs.tiny_scene, "mid": inputs.mid_scene, "island": lambda: inputs.moana_scene(ISLAND_SCALE)}
        sc = make[name]()
        self.api = api.Scene(sc)
        self.verts = torch.from_numpy(np.concatenate([v for v, _ in sc.meshes])).to(DEV)
        counts = torch.tensor([v.shape[0] for v, _ in sc.meshes])
        self.first = (torch.cumsum(counts, 0) - counts).to(DEV)
        self.counts = counts.to(DEV)
        self.xforms = torch.from_numpy(sc.xforms.reshape(-1, 3, 4)).to(DEV)
        self.ids = torch.from_numpy(sc.mesh_ids.astype(np.int64)).to(DEV)
        self.extent = float(sc.meta.get("extent", 100.0))
        self.n_quads, self.n_inst = self.api.n_quads, self.api.n_instances
        # the ground's tiles are the last instances of the mid and island scenes
        self.ground = sc.meta["terrain_meshes"][1] if "terrain_meshes" in sc.meta else 0


def _scene(name):
    if name not in _scenes:
        _scenes[name] = _Built(name)
    return _scenes[name]


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _camera(name, extent, rng, far=False):
    """Eye, look and field of view around the scene's vista."""
    j = rng.uniform(-0.05, 0.05, size=6) * extent * (4.0 if far else 1.0)
    if name == "tiny":
        eye, look, fov = (50.0 + j[0], -120.0 + j[1], 50.0 + j[2]), (50.0 + j[3], 50.0, 50.0 + j[5]), 40.0
    elif name == "mid":
        eye, look, fov = (2048.0 + j[0], -300.0 + j[1], 450.0 + 0.3 * j[2]), (2048.0 + j[3], 1800.0 + j[4], 0.0), 50.0
    else:
        eye = (0.5 * extent + j[0], -0.07 * extent + j[1], 0.11 * extent + 0.2 * j[2])
        look, fov = (0.5 * extent + j[3], 0.45 * extent + j[4], 0.0), 50.0
    return tuple(float(np.float32(x)) for x in eye), tuple(float(np.float32(x)) for x in look), fov


def _basis(eye, look):
    eye, look = np.asarray(eye, dtype=np.float64), np.asarray(look, dtype=np.float64)
    f = (look - eye) / np.linalg.norm(look - eye)
    r = np.cross(f, (0.0, 0.0, 1.0))
    r /= np.linalg.norm(r)
    return f, r, np.cross(r, f)


def _surface_points(S, n, g):
    """Points at vertices of random instances (a third on the ground, where there is one), a little above the surface."""
    i = torch.randint(S.n_inst, (n,), generator=g, device=DEV)
    if S.ground:
        on = torch.rand(n, generator=g, device=DEV) < 1.0 / 3.0
        i = torch.where(on, S.n_inst - 1 - torch.randint(S.ground, (n,), generator=g, device=DEV), i)
    m = S.ids[i]
    k = S.first[m] + (torch.rand(n, generator=g, device=DEV, dtype=torch.float64) * S.counts[m]).long()
    A, v = S.xforms[i].double(), S.verts[k].double()
    p = (A[:, :, :3] * v[:, None, :]).sum(-1) + A[:, :, 3]
    p[:, 2] += 1e-3 + 1e-5 * p.abs().amax(1)
    # neighbours in memory are neighbours in space, as a renderer's queue has them
    cell = (p[:, :2] / (S.extent / 256.0)).floor().clamp(-4, 260).long() + 4
    return p[torch.argsort(cell[:, 0] * 512 + cell[:, 1], stable=True)]


def _hemisphere(n, g):
    d = torch.randn(n, 3, generator=g, device=DEV, dtype=torch.float64)
    d = d / d.norm(dim=1, keepdim=True)
    d[:, 2] += 1.0  # cosine-weighted about +z
    return d / d.norm(dim=1, keepdim=True).clamp_min(1e-6)


def _rays(case, seed):
    """float32 [n, 8] (o, tmin, d, tmax) on the GPU."""
    S, n, g = _scene(case["scene"]), int(case["n"]), _gen(seed)
    rng = np.random.default_rng(seed)
    tmax = float(case.get("reach", math.inf))
    if case["rays"] in ("pick", "camera"):
        eye, look, fov = _camera(case["scene"], S.extent, rng)
        f, r, u = (torch.from_numpy(x).to(DEV) for x in _basis(eye, look))
        if case["rays"] == "pick":
            w, x, y = 256, 128 + 48 * torch.randn(n, generator=g, device=DEV).double(), 128 + 48 * torch.randn(n, generator=g, device=DEV).double()
            h = 256
        else:
            w = int(case["w"])
            h = -(-n // w)
            k = torch.arange(n, device=DEV)
            x, y = (k % w).double() + 0.5, (k // w).double() + 0.5
        th = math.tan(math.radians(fov) / 2)
        d = f + ((2 * x / w - 1) * th * w / h)[:, None] * r + ((1 - 2 * y / h) * th)[:, None] * u
        d = d / d.norm(dim=1, keepdim=True)
        o = torch.tensor(eye, device=DEV, dtype=torch.float64).expand(n, 3)
    else:
        o = _surface_points(S, n, g)
        d = torch.tensor(SUN, device=DEV, dtype=torch.float64).expand(n, 3) if case["rays"] == "sun" else _hemisphere(n, g)
    a = torch.empty(n, 8, device=DEV)
    a[:, 0:3], a[:, 3], a[:, 4:7], a[:, 7] = o, 0.0, d, tmax
    return a


def _view(case, S, rng, **more):
    eye, look, fov = _camera(case["scene"], S.extent, rng, far=bool(more.pop("far", False)))
    crop = {k: int(case[k]) for k in ("crop_x", "crop_y", "crop_w", "crop_h") if k in case}
    size = {"w": int(case.get("w", 0)), "h": int(case.get("h", 0)), "spp": int(case.get("spp", 1)), **crop, **more}
    return inputs.View(eye=eye, look=look, up=(0.0, 0.0, 1.0), vfov_deg=fov, **size)


def _params(case, seed, S):
    p = inputs.Params(max_depth=int(case["depth"]), seed=1000 + int(seed), env=(1.0, 1.0, 1.0))
    if case.get("sun"):
        p.sun_dir, p.sun_E = SUN, (3.0, 3.0, 3.0)
    if case.get("tex"):
        r = int(case["tex"])
        p.tex = torch.rand(S.n_quads, r, r, 3, generator=_gen(seed + 7), device=DEV).mul_(0.6).add_(0.4)
    if case.get("lights"):
        e = S.extent
        p.lights = inputs.key_lights(int(case["lights"]), (0.1 * e, 0.1 * e), (0.9 * e, 0.9 * e), 0.03 * e, 0.15 * e + 60.0,
                                     (60.0, 55.0, 45.0), seed=int(seed) + 8)
    return p


def _albedo(S, seed):
    return torch.rand(S.n_quads, 3, generator=_gen(seed + 3), device=DEV).mul_(0.6).add_(0.2)


def prepare(case, seed):
    S, kind = _scene(case["scene"]), case["kind"]
    s = {"kind": kind, "scene": S.api}
    if kind in ("closest", "any"):
        return {**s, "rays": _rays(case, seed)}
    rng = np.random.default_rng(seed)
    s.update(albedo=_albedo(S, seed), params=_params(case, seed, S))
    if kind == "views":
        views, base = [], 0
        sizes = np.random.default_rng(int(case["n_views"]))  # the sizes are the case's, the cameras the seed's
        for _ in range(int(case["n_views"])):
            w, h = (int(x) for x in np.maximum(4, np.round(case["side"] * 2.0 ** sizes.uniform(-1.0, 1.0, size=2))))
            views.append(_view(case, S, rng, far=True, w=w, h=h, spp=int(sizes.integers(1, case["spp"] + 1)), pixel_base=base))
            base += w * h
        return {**s, "graph": api.RenderGraph(S.api, views, s["albedo"], s["params"])}
    view = _view(case, S, rng)
    w, h = view.region
    if kind == "progressive":
        k = 16  # frames already summed
        view.sample_base = k
        frames = torch.rand(h, w, 3, generator=_gen(seed + 5), device=DEV).mul_(2.0 * k)
        s.update(frames=k + 1, frame_sum=frames, mean=torch.empty_like(frames))
    if kind == "train":
        target = torch.rand(h, w, 3, generator=_gen(seed + 6), device=DEV).mul_(2.0)
        s.update(target=target, dimage=torch.empty_like(target))
    return {**s, "view": view}


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    kind, scene = s["kind"], s["scene"]
    if kind == "closest":
        hits = scene.trace_closest(s["rays"])
        return {"t": hits[:, 0].view(torch.float32), "id_uv": hits[:, 1:]}
    if kind == "any":
        return {"bits": scene.trace_any(s["rays"])}
    if kind == "views":
        return s["graph"].launch()
    (img,) = scene.render([s["view"]], s["albedo"], s["params"])
    if kind == "progressive":
        api.accumulate(s["frame_sum"], img, s["frames"], s["mean"])
        return {"frame": img, "sum": s["frame_sum"], "mean": s["mean"]}
    if kind == "train":
        loss = api.l2_loss(img, s["target"], s["dimage"])
        grad = torch.zeros_like(s["albedo"])
        scene.adjoint([s["view"]], s["albedo"], [s["dimage"]], grad, s["params"])
        return {"image": img, "loss": loss, "grad": grad}
    return {"image": img}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
#: quads, instances, quads of a typical mesh, and rays per path and depth that a render of the scene traces
_SIZES = {"tiny": (4096, 256, 4096, 0.6), "mid": (5.73e6, 1.0e5, 2.4e4, 0.6), "island": (13.1e6, 1.96e6, 2.1e3, 0.34)}


def work(case):
    """Rays and results once, and for each ray one descent through both levels of a four-wide tree (four boxes of 64 bytes
    and 24 multiply-adds a level), one instance (64 bytes) and one quad (48 bytes, about 100 operations); the scene's
    part no larger than the scene (each quad and instance with its share of the nodes once)."""
    quads, inst, mesh, share = _SIZES[case["scene"]]
    levels = math.log(inst, 4) + math.log(mesh / 2, 4)
    if case["kind"] in ("closest", "any"):
        rays, own = case["n"], case["n"] * (32 + (16 if case["kind"] == "closest" else 1 / 8))
        per_quad = 48
    else:
        if case["kind"] == "views":
            pixels = case["n_views"] * case["side"] ** 2
            paths = pixels * (case["spp"] + 1) / 2
        else:
            pixels = case.get("crop_w", case["w"]) * case.get("crop_h", case["h"])
            paths = pixels * case.get("spp", 1)
        rays = paths * (1 + share * (case["depth"] - 1) * (1 + bool(case["sun"]) + bool(case.get("lights"))) / 2)
        own = pixels * 12
        per_quad = 48 + 12 + 12 * case.get("tex", 0) ** 2
        if case["kind"] == "progressive":
            own += pixels * 36
        if case["kind"] == "train":
            rays *= 1.5  # the gradient's pass follows the paths, not the shadow rays
            own += pixels * 36 + quads * 12
    touched = min(rays * (levels * 64 + 64 + per_quad), quads * (per_quad + 20) + inst * (64 + 32))
    return {"bytes": own + touched, "flops": rays * (levels * 24 * 2 + 100)}


# ---------------------------------------------------------------------------
# the same in 64 bits, by brute force over every quad (tiny scene)
# ---------------------------------------------------------------------------

class _Brute:
    """World-space triangles of an instanced scene, each as the affine map that takes it to the unit triangle."""

    def __init__(self, sc):
        P, owner, quad = [], [], []
        for i, (x, m) in enumerate(zip(sc.xforms.reshape(-1, 3, 4).astype(np.float64), sc.mesh_ids)):
            v, q = sc.meshes[int(m)]
            P.append((v.astype(np.float64) @ x[:, :3].T + x[:, 3])[q])
            owner.append(np.full(len(q), i))
            quad.append(np.arange(len(q)))
        P = torch.from_numpy(np.concatenate(P)).to(DEV)  # [quads, 4, 3]
        self.normal = torch.linalg.cross(P[:, 2] - P[:, 0], P[:, 3] - P[:, 1])
        self.normal = self.normal / self.normal.norm(dim=1, keepdim=True)
        self.row = torch.from_numpy(np.concatenate(quad)).to(DEV)  # one mesh: its quad is the albedo's row
        tri = torch.stack([P[:, [0, 1, 2]], P[:, [0, 2, 3]]], 1).reshape(-1, 3, 3)
        e1, e2 = tri[:, 1] - tri[:, 0], tri[:, 2] - tri[:, 0]
        M = torch.linalg.inv(torch.stack([e1, e2, torch.linalg.cross(e1, e2)], 2))  # [tris, 3, 3]
        self.M = [M[:, k].T.contiguous() for k in range(3)]
        self.c = [-(M[:, k] * tri[:, 0]).sum(1) for k in range(3)]

    def closest(self, o, d, tmin, tmax):
        """Distances (tmax where nothing is hit) and quads of the nearest hits."""
        ts, qs = [], []
        for k in range(0, len(o), 96):
            a, b = o[k:k + 96], d[k:k + 96]
            t = -(a @ self.M[2] + self.c[2]) / (b @ self.M[2])
            u = a @ self.M[0] + self.c[0] + t * (b @ self.M[0])
            v = a @ self.M[1] + self.c[1] + t * (b @ self.M[1])
            hit = (u >= 0) & (v >= 0) & (u + v <= 1) & (t > tmin) & (t < tmax)
            best, at = torch.where(hit, t, math.inf).min(1)
            ts.append(torch.where(torch.isinf(best), torch.full_like(best, tmax), best))
            qs.append(torch.where(torch.isinf(best), -1, at // 2))
        return torch.cat(ts), torch.cat(qs)


def _philox(pixel, sample, bounce, seed):
    """Philox4x32-10 of (pixel, 0, sample, bounce), as uniforms in [0, 1) of 24 bits: [n, 2] (the first two words)."""
    full = 0xFFFFFFFF
    c = [pixel & full, pixel >> 32, sample, torch.full_like(pixel, bounce)]
    k0, k1 = seed & full, (seed >> 32) & full

    def mul(m, x):  # 32 x 32 -> high and low words, within 63 bits
        lo, hi = m * (x & 0xFFFF), m * (x >> 16)
        mid = hi + (lo >> 16)
        return mid >> 16, ((mid & 0xFFFF) << 16) | (lo & 0xFFFF)

    for _ in range(10):
        h0, l0 = mul(0xD2511F53, c[0])
        h1, l1 = mul(0xCD9E8D57, c[2])
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & full, (k1 + 0xBB67AE85) & full
    return (c[0] >> 8).double() * 2.0 ** -24, (c[1] >> 8).double() * 2.0 ** -24


def _exact_image(B, view, albedo, p):
    """The path-traced image of a view, environment and sun, in 64 bits."""
    rw, rh = view.region
    k = torch.arange(rw * rh * view.spp, device=DEV)
    pix, smp = k // view.spp, k % view.spp + view.sample_base
    x, y = pix % rw + view.crop_x, pix // rw + view.crop_y
    g = view.pixel_base + y * view.w + x
    j0, j1 = _philox(g, smp, 0, p.seed)
    f, r, u = (torch.from_numpy(a).to(DEV) for a in _basis(view.eye, view.look))
    th = math.tan(math.radians(view.vfov_deg) / 2)
    d = f + ((2 * (x + j0) / view.w - 1) * th * view.w / view.h)[:, None] * r + ((1 - 2 * (y + j1) / view.h) * th)[:, None] * u
    d = d / d.norm(dim=1, keepdim=True)
    o = torch.tensor(view.eye, device=DEV, dtype=torch.float64).expand_as(d)
    env, E = (torch.tensor(a, device=DEV, dtype=torch.float64) for a in (p.env, p.sun_E))
    sun = torch.tensor(p.sun_dir, device=DEV, dtype=torch.float64)
    sun = sun / sun.norm()
    L, beta, live = torch.zeros_like(d), torch.ones_like(d), k
    for i in range(1, p.max_depth + 1):
        t, q = B.closest(o, d, 0.0, math.inf)
        miss = q < 0
        L[live[miss]] += beta[live[miss]] * env
        live, o, d, t, q = live[~miss], o[~miss], d[~miss], t[~miss], q[~miss]
        if not len(live):
            break
        n = B.normal[q]
        n = torch.where((n * d).sum(1, keepdim=True) > 0, -n, n)
        h = o + t[:, None] * d
        o = h + (1e-4 + 1e-5 * h.abs().amax(1, keepdim=True)) * n
        a = albedo[B.row[q]].double()
        if p.sun_on:
            cos = n @ sun
            seen = (cos > 0).clone()
            at = torch.nonzero(seen)[:, 0]
            if len(at):
                seen[at] = B.closest(o[at], sun.expand(len(at), 3), 0.0, math.inf)[1] < 0
            L[live] += torch.where(seen[:, None], beta[live] * a / math.pi * E * cos[:, None], torch.zeros_like(a))
        beta[live] *= a
        x0, x1 = _philox(g[live], smp[live], i, p.seed)
        rad, phi = x0.sqrt(), 2 * math.pi * x1
        sg = torch.copysign(torch.ones_like(n[:, 2]), n[:, 2])
        c = -1.0 / (sg + n[:, 2])
        b = n[:, 0] * n[:, 1] * c
        b1 = torch.stack([1 + sg * n[:, 0] ** 2 * c, sg * b, -sg * n[:, 0]], 1)
        b2 = torch.stack([b, sg + n[:, 1] ** 2 * c, -n[:, 1]], 1)
        d = (rad * torch.cos(phi))[:, None] * b1 + (rad * torch.sin(phi))[:, None] * b2 + (1 - x0).clamp_min(0).sqrt()[:, None] * n
    return L.view(rh, rw, view.spp, 3).mean(2)


#: Most rays that brute force follows: about 0.1 ms each over the tiny scene's two million triangles.
_MOST_EXACT = 60_000


def exact(case, seed):
    if case["scene"] != "tiny" or case["kind"] not in ("closest", "frame"):
        return None
    if case["kind"] == "closest":
        if case["n"] > _MOST_EXACT:
            return None
        r = _rays(case, seed).double()
        t, _ = _Brute(inputs.tiny_scene()).closest(r[:, 0:3], r[:, 4:7], 0.0, float(case.get("reach", math.inf)))
        return {"t": t, "id_uv": None}
    paths = case.get("crop_w", case["w"]) * case.get("crop_h", case["h"]) * case["spp"]
    if case.get("tex") or case.get("lights") or paths * case["depth"] * (2 if case["sun"] else 1) > _MOST_EXACT:
        return None
    S = _scene("tiny")
    view, p = _view(case, S, np.random.default_rng(seed)), _params(case, seed, S)
    return {"image": _exact_image(_Brute(inputs.tiny_scene()), view, _albedo(S, seed), p)}
