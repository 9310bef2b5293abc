"""What a program that uses the cone tracer has it do, as cases that can be timed and compared.

A case is a dict of plain values.  Its "kind" is the path a program takes:

  frame     one rendered frame: vct.build_mips of this frame's level-0 grid, then vct.trace of one view
  views     vct.trace of many views over several pyramids that the program keeps, in one call
  train     one optimisation step of a learnable grid: build, trace, an L2 loss against target images, and
            the gradient with respect to the grid ("render": by autograd through vct.render, one view;
            "adjoint": vct.trace with its per-cone state and vct.trace_backward over all views)
  geometry  the passes before the cones, from a triangle mesh: vct.voxelize and vct.gbuffer
  build     vct.build_mips alone, every level returned
  host      a burst of frames whose inputs and outputs live in page-locked host memory (vct.Pipeline)

Scenes are seeded boxes, inside a room that is open above or free, Lambert-lit by one directional light
(opaque voxels, empty space zero), seen by a pinhole camera inside them (neighbouring pixels see
neighbouring surface points; pixels that see the sky are masked) or sampled at random surface points (as
probes, lightmap texels or training batches are).
"""
import math
import random

import numpy as np
import torch

import paper_2104_00618_gb300 as vct

DEV = "cuda"
RED, GREEN, GREY = (0.75, 0.2, 0.2), (0.2, 0.75, 0.2), (0.75, 0.75, 0.75)
SHADED = vct.FLAG_OCC_SMOOTH | vct.FLAG_SPEC_GRACE | vct.FLAG_DIFFUSE_FIRST_HIT | vct.FLAG_SHADE


def listed():
    return [
        # The smallest call in use: a coarse grid of free boxes and 16 K random surface points (probes).
        dict(name="frame probes 64", kind="frame", n=64, width=128, height=128, cones="ring6", dtype="f32",
             layout="dense", flags=0, masked=0.0, pixels="surface", boxes=12),
        # The standard frame: a room at 256^3, full HD, nine diffuse, one specular and one occlusion cone.
        dict(name="frame room 256 1080p", kind="frame", n=256, width=1920, height=1080, cones="room9", dtype="f32",
             layout="dense", flags=0, masked=0.0, pixels="camera", boxes=32),
        # Half-precision storage, an odd-sized window with pixels that see no surface.
        dict(name="frame f16 128 ragged", kind="frame", n=128, width=1111, height=699, cones="room9", dtype="f16",
             layout="dense", flags=0, masked=0.1, pixels="camera", boxes=32),
        # Directional mips (less light leaking), a quarter of full HD.
        dict(name="frame aniso 128", kind="frame", n=128, width=960, height=540, cones="room9", dtype="f32",
             layout="aniso", flags=0, masked=0.0, pixels="camera", boxes=32),
        # A large grid, stored as the bricks it occupies because a dense pyramid would waste memory.
        dict(name="frame bricks 512 720p", kind="frame", n=512, width=1280, height=720, cones="room9", dtype="f32",
             layout="bricks", flags=0, masked=0.0, pixels="camera", boxes=32),
        # The modified cones and the shaded radiance that a renderer shows.
        dict(name="frame shaded 256 720p", kind="frame", n=256, width=1280, height=720, cones="room9", dtype="f32",
             layout="dense", flags=SHADED, masked=0.0, pixels="camera", boxes=32),
        # Offline rendering of many cameras of mixed sizes over several half-precision scenes in one call.
        dict(name="views f16 18", kind="views", grids="64,128,256", views=6, lo=256, hi=1280, dtype="f16", boxes=32),
        # A step of fitting a grid to images: eight views of 512^2, all gradients in one adjoint call.
        dict(name="train 128 8x512", kind="train", how="adjoint", n=128, views=8, width=512, height=512, dtype="f32",
             layout="dense", deterministic=False),
        # The smallest step, through autograd, with the reproducible adjoint.
        dict(name="train 32 autograd", kind="train", how="render", n=32, views=1, width=97, height=61, dtype="f32",
             layout="dense", deterministic=True),
        # Dynamic geometry: a mesh of about 240 K triangles voxelized and drawn into the G-buffer.
        dict(name="geometry 256 1080p", kind="geometry", n=256, width=1920, height=1080, boxes=32, tess=24, spheres=4),
        # A large pyramid, built once per scene.
        dict(name="build 512", kind="build", n=512, dtype="f32", layout="dense", boxes=32),
        # A renderer on the host: four frames in flight through the pipeline.
        dict(name="host 128 720p x4", kind="host", n=128, width=1280, height=720, frames=4, boxes=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["frame", "frame", "frame", "views", "train", "train", "geometry", "build", "host"])
    if kind == "frame":
        layout = rng.choice(["dense", "dense", "dense", "bricks", "aniso"])
        dtype = "f32" if layout == "aniso" else rng.choice(["f32", "f32", "f16"])
        n = 2 ** rng.randint(4, 8 if layout == "aniso" else 9)
        hi = 1400 if layout == "aniso" else 1920
        return dict(kind=kind, n=n, width=_log(rng, 16, hi), height=_log(rng, 9, hi * 9 // 16),
                    cones=rng.choice(["room9", "ring6"]), dtype=dtype, layout=layout,
                    flags=rng.choice([0, 0, 0, SHADED, vct.FLAG_SHADE | vct.FLAG_SHADE_IMPL, vct.FLAG_PREMULTIPLIED]),
                    masked=rng.choice([0.0, 0.0, 0.1, 0.5]), pixels=rng.choice(["camera", "camera", "surface"]),
                    boxes=rng.randint(6, 40))
    if kind == "views":
        grids = ",".join(str(2 ** rng.randint(5, 8)) for _ in range(rng.randint(1, 4)))
        lo = _log(rng, 32, 512)
        return dict(kind=kind, grids=grids, views=rng.randint(1, 5), lo=lo, hi=_log(rng, lo, 1200),
                    dtype=rng.choice(["f32", "f16"]), boxes=rng.randint(6, 40))
    if kind == "train":
        how = rng.choice(["adjoint", "render"])
        layout = rng.choice(["dense", "dense", "aniso", "bricks"])
        dtype = "f32" if layout == "aniso" else rng.choice(["f32", "f32", "f16"])
        n = 2 ** rng.randint(4, 6 if layout == "aniso" else 7)
        side = 256 if layout == "aniso" else 512
        return dict(kind=kind, how=how, n=n, views=1 if how == "render" else rng.randint(1, 6),
                    width=_log(rng, 24, side), height=_log(rng, 17, side), dtype=dtype, layout=layout,
                    deterministic=rng.random() < 0.25)
    if kind == "geometry":
        return dict(kind=kind, n=2 ** rng.randint(5, 8), width=_log(rng, 64, 1920), height=_log(rng, 36, 1080),
                    boxes=rng.randint(4, 32), tess=rng.randint(1, 24), spheres=rng.randint(0, 4))
    if kind == "build":
        layout = rng.choice(["dense", "dense", "aniso"])
        return dict(kind=kind, n=2 ** rng.randint(3, 8 if layout == "aniso" else 9),
                    dtype="f32" if layout == "aniso" else rng.choice(["f32", "f16"]), layout=layout,
                    boxes=rng.randint(4, 40))
    return dict(kind=kind, n=2 ** rng.randint(4, 7), width=_log(rng, 64, 1280), height=_log(rng, 36, 720),
                frames=rng.randint(2, 6), boxes=rng.randint(4, 40))


# ---------------------------------------------------------------------------
# scenes, cameras, parameters
# ---------------------------------------------------------------------------
def _scene(n, count, rng, room=True):
    """Integer-voxel boxes (lo, hi, colour), a light, and the level-0 grid [n,n,n,4] (z, y, x, rgba)."""
    while True:
        light = rng.normal(size=3)
        light /= np.linalg.norm(light)
        if light[1] >= 0.3:
            break
    boxes = []
    for _ in range(count):
        size = rng.integers(max(1, n // 16), max(1, n // 4) + 1, size=3)
        lo = np.array([rng.integers(0, n - s + 1) for s in size])
        boxes.append((lo, lo + size, rng.random(3)))
    g = torch.zeros((n, n, n, 4), device=DEV)

    def face(axis, at, sign, colour, lo, hi):
        sl = [slice(int(lo[a]), int(hi[a])) for a in (2, 1, 0)]
        sl[2 - axis] = slice(at, at + 1)
        v = torch.tensor(np.asarray(colour) * max(0.0, sign * light[axis]), dtype=torch.float32, device=DEV)
        part = g[tuple(sl)]
        part[..., :3] = torch.maximum(part[..., :3], v)
        part[..., 3] = 1.0

    if room:  # open to the sky: the light comes from above, so that visibility takes every value
        for axis in range(3):
            face(axis, 0, 1, RED if axis == 0 else GREY, (0, 0, 0), (n, n, n))
            if axis != 1:
                face(axis, n - 1, -1, GREEN if axis == 0 else GREY, (0, 0, 0), (n, n, n))
    for lo, hi, colour in boxes:
        solid = g[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]]
        solid[..., :3] = 0.0
        solid[..., 3] = 1.0
        for axis in range(3):
            face(axis, int(lo[axis]), -1, colour, lo, hi)
            face(axis, int(hi[axis]) - 1, 1, colour, lo, hi)
    return dict(n=n, boxes=boxes, light=light, grid=g, room=room)


def _free_point(scene, rng):
    n = scene["n"]
    for _ in range(200):  # a crowded scene may have no free point at all: then the camera is inside a box
        p = 0.12 + 0.76 * rng.random(3)
        if not any(np.all(p * n >= lo - 2) and np.all(p * n <= hi + 2) for lo, hi, _ in scene["boxes"]):
            break
    return p


def _basis(eye, target):
    f = target - eye
    f /= np.linalg.norm(f)
    r = np.cross(f, (0.0, 1.0, 0.0))
    r /= np.linalg.norm(r)
    return f, r, np.cross(r, f)


def _camera(scene, rng):
    eye = _free_point(scene, rng)
    target = _free_point(scene, rng)
    while np.linalg.norm((target - eye) * (1, 0, 1)) < 0.1:
        target = rng.random(3)
    return eye, target


def _raycast(scene, width, height, eye, target):
    """Pinhole view (60 degrees) of the boxes and the room's inner faces: position, normal [H*W,3], mask
    (zero where the ray leaves through the open ceiling)."""
    n = scene["n"]
    f, r, u = (torch.tensor(v, device=DEV) for v in _basis(eye, target))
    th = math.tan(math.radians(30.0))
    sx = (2.0 * (torch.arange(width, device=DEV, dtype=torch.float64) + 0.5) / width - 1.0) * th * width / height
    sy = (1.0 - 2.0 * (torch.arange(height, device=DEV, dtype=torch.float64) + 0.5) / height) * th
    d = (f + sx[None, :, None] * r + sy[:, None, None] * u).reshape(-1, 3)
    d = torch.where(d == 0, torch.full_like(d, 1e-300), d / d.norm(dim=1, keepdim=True))
    o = torch.tensor(eye, device=DEV)
    best = torch.full((len(d),), math.inf, device=DEV, dtype=torch.float64)
    axis = torch.zeros(len(d), dtype=torch.int64, device=DEV)
    walls = [(torch.tensor(lo / n, device=DEV), torch.tensor(hi / n, device=DEV), False) for lo, hi, _ in scene["boxes"]]
    if scene["room"]:
        one = torch.ones(3, device=DEV, dtype=torch.float64)
        walls.append((one / n, one * (n - 1) / n, True))
    for lo, hi, inside in walls:
        t1, t2 = (lo - o) / d, (hi - o) / d
        near, a_near = torch.minimum(t1, t2).max(dim=1)
        far, a_far = torch.maximum(t1, t2).min(dim=1)
        t, a = (far, a_far) if inside else (near, a_near)
        hit = (t > 0) & (t < best)
        hit &= ~((a == 1) & (d[:, 1] > 0)) if inside else near <= far
        best, axis = torch.where(hit, t, best), torch.where(hit, a, axis)
    mask = best.isfinite()
    pos = o + torch.where(mask, best, torch.zeros_like(best))[:, None] * d
    nrm = torch.zeros_like(pos).scatter_(1, axis[:, None], -d.gather(1, axis[:, None]).sign())
    keep = mask[:, None].to(torch.float64)
    return (pos * keep).float(), (nrm * keep).float(), mask.to(torch.uint8)


def _surface(scene, count, rng):
    """Random points on exposed box faces (the voxel in front of the point is empty): position, normal."""
    n, pos, nrm = scene["n"], [], []
    size = np.array([hi - lo for lo, hi, _ in scene["boxes"]], dtype=np.float64)
    area = np.stack([size[:, (a + 1) % 3] * size[:, (a + 2) % 3] for a in range(3)], 1).repeat(2, 1).reshape(-1)
    alpha = scene["grid"][..., 3]
    while sum(map(len, pos)) < count:
        k = rng.choice(len(area), p=area / area.sum(), size=2 * count)
        b, a, s = k // 6, (k % 6) // 2, (k % 2) * 2 - 1
        lo = np.array([v[0] for v in scene["boxes"]])[b]
        q = lo + rng.random((len(k), 3)) * size[b]
        rows = np.arange(len(k))
        q[rows, a] = np.where(s < 0, lo[rows, a], lo[rows, a] + size[b, a])
        front = q.copy()
        front[rows, a] += 0.5 * s
        ok = np.all((front > 0) & (front < n), axis=1)
        v = torch.tensor(np.clip(front, 0, n - 1).astype(np.int64), device=DEV)
        ok &= (alpha[v[:, 2], v[:, 1], v[:, 0]] == 0).cpu().numpy()
        m = np.zeros((len(k), 3))
        m[rows, a] = s
        pos.append((q / n)[ok])
        nrm.append(m[ok])
    cat = lambda v: torch.tensor(np.concatenate(v)[:count], dtype=torch.float32, device=DEV)  # noqa: E731
    return cat(pos), cat(nrm)


def _sph(theta, phi):
    t, p = math.radians(theta), math.radians(phi)
    return math.sin(t) * math.cos(p), math.sin(t) * math.sin(p), math.cos(t)


def _cone_params(cones, light, flags=0):
    if cones == "ring6":  # a front cone and five at 60 degrees, cosine weights, a narrow specular cone
        dirs = [(0.0, 0.0, 1.0)] + [_sph(60.0, 72.0 * k) for k in range(5)]
        w = [1 / 3.5] + [0.5 / 3.5] * 5
        own = dict(diffuse_aperture=math.radians(60.0), spec_aperture_min=math.radians(10.0),
                   spec_aperture_max=math.radians(10.0), occ_enable=int(bool(flags)))
    else:  # "room9": a front cone, four at 45 and four at 90 degrees; the specular aperture follows roughness
        dirs = [(0.0, 0.0, 1.0)] + [_sph(t, 90.0 * k) for t in (45.0, 90.0) for k in range(4)]
        dirs = [tuple(0.0 if abs(c) < 1e-12 else c for c in v) for v in dirs]
        w = [1.0 / 9.0] * 9
        own = dict(diffuse_aperture=0.55, spec_aperture_min=math.radians(5.0), spec_aperture_max=math.radians(60.0),
                   occ_enable=1)
    return dict(own, n_diffuse=len(dirs), diffuse_dir=np.array(dirs, np.float32), diffuse_weight=np.array(w, np.float32),
                spec_enable=1, roughness_min=0.05, occ_aperture=0.55, light_dir=np.asarray(light, np.float32),
                beta=0.5, t0_voxels=1.0, normal_offset_voxels=1.0, t_max=1.0, flags=flags, shadow_str=1.0,
                occ_max_dist=0.3, shininess=32.0, shininess_falloff=2.0, diffuse_str=0.8, specular_str=0.6,
                light_color=(1.0, 0.9, 0.7))


def _make_view(scene, case, width, height, rng, pyramid=0):
    """A vct.View (outputs allocated) of the scene, with what the case's options ask for."""
    gen = torch.Generator(device=DEV).manual_seed(int(rng.integers(1 << 40)))
    eye, target = _camera(scene, rng)
    mask = None
    if case.get("pixels") == "surface":
        pos, nrm = _surface(scene, width * height, rng)
    else:
        pos, nrm, mask = _raycast(scene, width, height, eye, target)
    if case.get("masked"):
        keep = (torch.rand(width * height, device=DEV, generator=gen) >= case["masked"]).to(torch.uint8)
        mask = keep if mask is None else mask * keep
    rough = None
    if case.get("cones", "room9") == "room9":
        rough = 0.05 + 0.95 * torch.rand(width * height, device=DEV, generator=gen)
    v = vct.View(width, height, pos, nrm, tuple(float(np.float32(c)) for c in eye), rough, mask, pyramid)
    shade = bool(case.get("flags", 0) & vct.FLAG_SHADE)
    if shade:
        v.albedo = 0.2 + 0.8 * torch.rand((width * height, 3), device=DEV, generator=gen)
    return v.alloc_outputs(radiance=shade)


# ---------------------------------------------------------------------------
# meshes
# ---------------------------------------------------------------------------
def _mesh(case, rng):
    """Tessellated boxes, spheres and a room of a mesh scene in the unit cube; voxel-unaligned corners."""
    V, I, C, base = [], [], [], 0

    def add(p, nu, nv, colour):  # p: (nv + 1) x (nu + 1) grid of vertices
        nonlocal base
        a, b = np.meshgrid(np.arange(nu), np.arange(nv))
        i = (b * (nu + 1) + a).ravel() + base
        j, k, m = i + 1, i + nu + 2, i + nu + 1
        V.append(p.reshape(-1, 3))
        I.append(np.concatenate([np.stack([i, j, k], 1), np.stack([i, k, m], 1)]))
        C.append(np.broadcast_to(colour, (2 * nu * nv, 3)))
        base += len(V[-1])

    def box(lo, hi, colours, tess, inward):
        g = np.linspace(0.0, 1.0, tess + 1)
        for axis in range(3):
            u, v = (axis + 1) % 3, (axis + 2) % 3
            for side in (0, 1):
                p = np.zeros((tess + 1, tess + 1, 3))
                flip = (side == 0) != inward  # counter-clockwise seen from the side the face looks at
                s, t = (g[:, None], g[None, :]) if flip else (g[None, :], g[:, None])
                p[..., axis] = hi[axis] if side else lo[axis]
                p[..., u] = lo[u] + s * (hi[u] - lo[u])
                p[..., v] = lo[v] + t * (hi[v] - lo[v])
                add(p, tess, tess, colours[2 * axis + side])

    edge = 0.7 / case["n"]
    box(np.full(3, edge), np.full(3, 1 - edge), (RED, GREEN, GREY, GREY, GREY, GREY), case["tess"], True)
    solids = []
    for _ in range(case["boxes"]):
        size = rng.uniform(1 / 16, 1 / 4, size=3)
        lo = rng.uniform(edge, 1 - edge - size)
        solids.append((lo, lo + size))
        box(lo, lo + size, [rng.random(3)] * 6, case["tess"], False)
    for _ in range(case["spheres"]):
        r = rng.uniform(1 / 24, 1 / 10)
        c = rng.uniform(r + edge, 1 - r - edge, size=3)
        th, ph = np.meshgrid(np.linspace(math.pi, 0, 33), np.linspace(0, 2 * math.pi, 65), indexing="ij")
        add(c + r * np.stack([np.sin(th) * np.cos(ph), np.cos(th), np.sin(th) * np.sin(ph)], -1), 64, 32, rng.random(3))
        solids.append((c - r, c + r))
    for _ in range(200):
        eye, target = rng.uniform(0.1, 0.9, size=(2, 3))
        free = not any(np.all(eye > lo - 0.01) and np.all(eye < hi + 0.01) for lo, hi in solids)
        if free and np.linalg.norm((target - eye) * (1, 0, 1)) > 0.2:
            break
    f32 = lambda v: np.asarray(v, np.float32)  # noqa: E731
    f, r, u = _basis(eye, target)
    cam = dict(eye=f32(eye), forward=f32(f), right=f32(r), up=f32(u), tan_half=float(np.float32(math.tan(math.radians(30)))),
               width=case["width"], height=case["height"], frame_origin=f32((0, 0, 0)), frame_size=1.0)
    mesh = vct.Mesh.from_host({"vertices": np.concatenate(V), "indices": np.concatenate(I),
                               "colors": np.ascontiguousarray(np.concatenate(C))}, DEV)
    light = rng.normal(size=3)
    light[1] = abs(light[1]) + 0.3
    light = dict(light_dir=f32(light / np.linalg.norm(light)), light_color=(1.0, 0.9, 0.8), ambient=0.1, diffuse_str=0.9)
    return mesh, cam, light


# ---------------------------------------------------------------------------
# preparing and running
# ---------------------------------------------------------------------------
def prepare(case, seed):
    rng = np.random.default_rng([2104, seed])
    kind, st = case["kind"], {"case": case}
    if kind == "geometry":
        st["mesh"], st["cam"], st["light"] = _mesh(case, rng)
        n, w, h, nt = case["n"], case["width"], case["height"], st["mesh"].indices.shape[0]
        st["grid"] = torch.empty((n, n, n, 4), device=DEV)
        st["vws"], st["gws"] = vct.voxelize_workspace(n, nt), vct.gbuffer_workspace(w, h, nt)
        return st
    if kind == "views":
        st["scenes"] = [_scene(int(n), case["boxes"], rng) for n in case["grids"].split(",")]
        st["prm"] = _cone_params("room9", st["scenes"][0]["light"])
        sizes = np.random.default_rng([case["lo"], case["hi"]])  # the sizes are the case's, the rest the seed's
        side = lambda: int(sizes.integers(case["lo"], case["hi"] + 1))  # noqa: E731
        st["views"] = [_make_view(s, case, side(), max(1, side() * 9 // 16), rng, i)
                       for i, s in enumerate(st["scenes"]) for _ in range(case["views"])]
        st["pyramids"] = [vct.build_mips(s["grid"], dtype=case["dtype"]) for s in st["scenes"]]
        st["params"] = vct.make_params(st["prm"])
        return st
    if kind == "train":
        scene = _scene(case["n"], 16, rng)
        st["prm"] = dict(_cone_params("ring6", scene["light"]), occ_enable=1)
        st["params"] = vct.make_params(st["prm"])
        opts = dict(cones="ring6", pixels="camera")
        st["views"] = [_make_view(scene, opts, case["width"], case["height"], rng) for _ in range(case["views"])]
        vct.trace(vct.build_mips(scene["grid"]), st["views"], st["params"])
        st["targets"] = [(v.out_diffuse.clone(), v.out_specular.clone(), v.out_visibility.clone()) for v in st["views"]]
        for v in st["views"]:
            v.alloc_cone_state(st["params"])
        gen = torch.Generator(device=DEV).manual_seed(seed)
        st["grid"] = 0.05 + 0.1 * torch.rand((case["n"],) * 3 + (4,), device=DEV, generator=gen)
        if case["how"] == "render":
            st["grid"].requires_grad_(True)
        return st
    scene = _scene(case["n"], case["boxes"], rng, room=case.get("pixels") != "surface")
    st["grid"] = scene["grid"]
    if kind == "build":
        st["pyramid"] = vct.Pyramid(case["n"], dtype=case["dtype"], layout=case["layout"])
        return st
    st["prm"] = _cone_params(case.get("cones", "room9"), scene["light"], case.get("flags", 0))
    st["params"] = vct.make_params(st["prm"])
    st["view"] = v = _make_view(scene, case, case["width"], case["height"], rng)
    if kind == "host":
        host = lambda t: t.cpu().pin_memory()  # noqa: E731
        st["in"] = [host(t) for t in (scene["grid"], v.position, v.normal, v.roughness, v.mask)]
        st["out"] = [[torch.empty(s).pin_memory() for s in (v.out_diffuse.shape, v.out_specular.shape, v.out_visibility.shape)]
                     for _ in range(case["frames"])]
        st["pipeline"] = vct.Pipeline(case["n"], case["width"], case["height"], st["params"])
    elif case["layout"] != "bricks":  # a brick pyramid's size depends on the frame's grid: made anew each time
        st["pyramid"] = vct.Pyramid(case["n"], dtype=case["dtype"], layout=case["layout"])
    return st


def _outputs(v):
    out = {"diffuse": v.out_diffuse, "specular": v.out_specular, "visibility": v.out_visibility}
    if v.out_radiance is not None:
        out["radiance"] = v.out_radiance
    return out


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "frame":
        pyr = vct.build_mips(st["grid"], dtype=case["dtype"], layout=case["layout"], out=st.get("pyramid"))
        vct.trace(pyr, st["view"], st["params"])
        return _outputs(st["view"])
    if kind == "views":
        vct.trace(st["pyramids"], st["views"], st["params"])
        return [_outputs(v) for v in st["views"]]
    if kind == "train":
        if case["how"] == "render":
            st["grid"].grad = None
            out = vct.render(st["grid"], st["views"][0], st["params"], dtype=case["dtype"], layout=case["layout"],
                             deterministic=case["deterministic"])
            loss = sum(0.5 * (o - t).square().sum() for o, t in zip(out, st["targets"][0]))
            loss.backward()
            return {"outputs": [o.detach() for o in out], "grad": st["grid"].grad}
        pyr = vct.build_mips(st["grid"], dtype=case["dtype"], layout=case["layout"])
        vct.trace(pyr, st["views"], st["params"])
        diff = [(v.out_diffuse - t[0], v.out_specular - t[1], v.out_visibility - t[2])
                for v, t in zip(st["views"], st["targets"])]
        grad = vct.trace_backward(pyr, st["views"], diff, st["params"], deterministic=case["deterministic"])
        return {"outputs": [_outputs(v) for v in st["views"]], "grad": grad}
    if kind == "geometry":
        grid = vct.voxelize(st["mesh"], case["n"], light=st["light"], out=st["grid"], workspace=st["vws"])
        g = vct.gbuffer(st["mesh"], st["cam"], workspace=st["gws"])
        return {"grid": grid, **{k: g[k] for k in ("position", "normal", "albedo", "mask", "triangle")}}
    if kind == "build":
        pyr = vct.build_mips(st["grid"], dtype=case["dtype"], layout=case["layout"], out=st["pyramid"])
        return _levels(pyr, case)
    for out in st["out"]:
        st["pipeline"].submit(st["in"][0], st["in"][1], st["in"][2], st["view"].camera, *out, roughness=st["in"][3],
                              mask=st["in"][4])
    st["pipeline"].wait()
    return st["out"]


def _levels(pyr, case):
    """The stored texels of every level, in place (Morton order; six volumes per coarse anisotropic level)."""
    size = 8 if case["dtype"] == "f16" else 16
    kind = torch.float16 if case["dtype"] == "f16" else torch.float32
    out, at = [], 256
    for l in range(pyr.levels):
        nbytes = (pyr.n >> l) ** 3 * size * (6 if case["layout"] == "aniso" and l else 1)
        out.append(pyr.storage[at:at + nbytes].view(kind))
        at += (nbytes + 255) // 256 * 256
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _steps(gamma, n):
    """Samples of a cone that marches its whole length (t0 = 1 voxel to n voxels, t *= 1 + tan(gamma / 2))."""
    return math.log(n) / math.log1p(math.tan(gamma / 2)) + 1


def _march_flops(n, px, cones):
    """A sample: two trilinear lookups of four channels (7 lerps of 3 operations each), their blend, the
    compositing and the position: about 200 operations.  Most cones of these scenes march their whole length
    (the first-hit variant, where most stop early, is counted the same way)."""
    if cones == "ring6":
        steps = 6 * _steps(math.radians(60), n) + _steps(math.radians(10), n)
    else:
        steps = 10 * _steps(0.55, n) + _steps(math.radians(32.5), n)
    return 200.0 * px * steps


def _pyramid_bytes(n, dtype, layout="dense"):
    m = sum((n >> l) ** 3 * (6 if layout == "aniso" and l else 1) for l in range(n.bit_length()))
    return m * (8 if dtype == "f16" else 16)


def work(case):
    kind, n = case["kind"], case.get("n")
    px = case.get("width", 0) * case.get("height", 0)
    if kind == "build":
        return {"bytes": 16 * n ** 3 + _pyramid_bytes(n, case["dtype"], case["layout"]), "flops": 4.0 * n ** 3}
    if kind == "geometry":
        tris = 12 * (case["boxes"] + 1) * case["tess"] ** 2 + 4096 * case["spheres"]
        return {"bytes": 16 * n ** 3 + 41 * px + 36 * tris, "flops": 100.0 * tris + 50.0 * px}
    if kind == "views":
        grids = [int(v) for v in case["grids"].split(",")]
        each = case["views"] * ((case["lo"] + case["hi"]) / 2) ** 2 * 9 / 16  # of a scene, on average
        return {"bytes": sum(_pyramid_bytes(m, case["dtype"]) + 64 * each for m in grids),
                "flops": sum(_march_flops(m, each, "room9") for m in grids)}
    if kind == "train":
        px *= case["views"]
        # grid read and its gradient written; per pixel the view, the outputs, the targets
        return {"bytes": 32 * n ** 3 + px * (24 + 36 + 36), "flops": 3 * _march_flops(n, px, "ring6")}
    if kind == "host":
        return {"bytes": case["frames"] * (16 * n ** 3 + 64 * px), "flops": case["frames"] * _march_flops(n, px, "room9")}
    lit = 16 if case["flags"] & vct.FLAG_SHADE else 0
    return {"bytes": 16 * n ** 3 + px * (24 + 36 + 4 + lit), "flops": _march_flops(n, px, case["cones"])}


def tolerance(case):
    """About four times what the outputs were seen to differ from exact().  A traced pixel's largest difference
    is a specular cone with a step at t_max, taken on one side only (5e-3 in float32); half-precision storage
    rounds every texel (2^-11); gradients carry the rounding of small differences (outputs less targets)."""
    kind, half = case["kind"], case.get("dtype") == "f16"
    if kind == "build":
        return {"rel": 1e-4, "max": 2e-3} if half else {"rel": 1e-6, "max": 1e-6}
    if kind == "geometry":  # decisions are exact: the mask and the triangle of every pixel stay the same
        return {"rel": 1e-6, "max": 1e-5}
    if kind == "train":
        return {"rel": 3e-4, "max": 6e-3} if half else {"rel": 6e-5, "max": 1e-3}
    return {"rel": 3e-4, "max": 0.15} if half else {"rel": 3e-5, "max": 0.03}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _morton(m):
    c = torch.arange(m, device=DEV)
    s = sum(((c >> b) & 1) << (3 * b) for b in range(10))
    return (s[:, None, None] * 4 + s[None, :, None] * 2 + s[None, None, :]).reshape(-1)


def _mips(grid, layout):
    """Levels as [volumes, m, m, m, 4]: one volume, or six per level above 0 (+x, -x, +y, -y, +z, -z)."""
    levels = [grid[None].double()]
    while levels[-1].shape[1] > 1:
        g = levels[-1]
        if layout != "aniso":
            m = g.shape[1] // 2
            levels.append(g.reshape(1, m, 2, m, 2, m, 2, 4).mean(dim=(2, 4, 6)))
            continue
        vols = []
        for d in range(6):
            v = g[d if len(g) == 6 else 0]
            ax = 2 - d // 2  # of the array (z, y, x)
            f, b = (v.unflatten(ax, (-1, 2)).select(ax + 1, k) for k in ((1, 0) if d % 2 else (0, 1)))
            a = f[..., 3:] + (1 - f[..., 3:]) * b[..., 3:]
            c = (f[..., 3:] * f[..., :3] + (1 - f[..., 3:]) * b[..., 3:] * b[..., :3]) / torch.where(a > 0, a, torch.ones_like(a))
            p = torch.cat([torch.where(a > 0, c, torch.zeros_like(c)), a], -1)
            for o in [o for o in range(3) if o != ax]:
                p = p.unflatten(o, (-1, 2)).mean(dim=o + 1)
            vols.append(p)
        levels.append(torch.stack(vols))
    return levels


class _Sampler:
    def __init__(self, grid, layout):
        levels = _mips(grid, layout)
        self.n, self.top, self.aniso = grid.shape[0], len(levels) - 1, layout == "aniso"
        self.flat = torch.cat([g.reshape(-1, 4) for g in levels])
        sizes = [g[..., 0].numel() for g in levels]
        self.start = torch.tensor([sum(sizes[:l]) for l in range(len(sizes))], device=DEV)

    def trilinear(self, x, level, volume):
        """x: level-0 voxel coordinates [P,3]; level [P]; volume [P] or 0."""
        m = self.n >> level
        u = x / (2.0 ** level.double())[:, None] - 0.5
        b = u.floor()
        f, b = u - b, b.long()
        first = self.start[level] + volume * m ** 3
        out = 0.0
        for c in range(8):
            at, w, ok = 0, 1.0, True
            for a in (2, 1, 0):
                i = b[:, a] + (c >> a & 1)
                ok = ok & (i >= 0) & (i < m)
                at = at * m + i
                w = w * (f[:, a] if c >> a & 1 else 1 - f[:, a])
            got = self.flat.index_select(0, torch.where(ok, first + at, torch.zeros_like(at)))
            out = out + got * torch.where(ok, w, torch.zeros_like(w))[:, None]
        return out

    def level(self, x, level, w):
        if not self.aniso:
            return self.trilinear(x, level, 0)
        wt = w * w / (w * w).sum(1, keepdim=True)
        return sum(wt[:, a:a + 1] * self.trilinear(x, level, torch.where(level > 0, 2 * a + (w[:, a] < 0).long(), 0 * level))
                   for a in range(3))

    def __call__(self, x, lam, w):
        lam = lam.clamp(0, self.top)
        l0 = lam.floor().long()
        f = (lam - l0)[:, None]
        return (1 - f) * self.level(x, l0, w) + f * self.level(x, (l0 + 1).clamp(max=self.top), w)


def _march(smp, prm, apex, w, half_tan, fade=False, first_hit=False):
    """Front-to-back march of one cone per row; apex in voxels, half_tan = tan(gamma / 2) per row: (rgb, alpha)."""
    n, beta = smp.n, prm["beta"]
    t = torch.full_like(half_tan, prm["t0_voxels"])
    rgb, tr = torch.zeros_like(apex), torch.ones_like(t)
    open_ = torch.ones_like(t, dtype=torch.bool)
    straight = not prm["flags"] & vct.FLAG_PREMULTIPLIED
    while True:
        on = open_ & (t <= prm["t_max"] * n) & (tr.detach() > 1e-18)
        if not bool(on.any()):
            break
        d = 2 * t * half_tan
        at = on.nonzero()[:, 0]  # the rows that still march
        s = smp(apex[at] + t[at, None] * w[at], torch.log2(d[at]), w[at])
        s = torch.zeros((len(t), 4), device=DEV, dtype=torch.float64).index_add(0, at, s)
        a = s[:, 3]
        if fade:
            u = (torch.sqrt(t / n) * prm["shadow_str"] / prm["occ_max_dist"]).clamp(0, 1)
            a = a * u * u * (3 - 2 * u)
        if first_hit:
            hit = on & (a > 0.01)
            rgb = torch.where(hit[:, None], s[:, :3], rgb)
            tr = torch.where(hit, torch.zeros_like(tr), tr)
            open_ = open_ & ~hit
        else:
            rgb = rgb + (tr * (a if straight else on.double()))[:, None] * s[:, :3]
            tr = tr * (1 - a)
        t = t + beta * d
    return torch.cat([rgb, (1 - tr)[:, None]], 1)


def _f64(v):
    return torch.tensor(np.asarray(v, np.float32), device=DEV).double()


def _trace64(smp, prm, v):
    """D, S, Vis (and L) of a view, as vct.trace lays them out."""
    prm = {k: float(np.float32(x)) if isinstance(x, float) else x for k, x in prm.items()}
    rows = torch.arange(v.width * v.height, device=DEV) if v.mask is None else v.mask.nonzero()[:, 0]
    x, nrm = v.position[rows].double(), v.normal[rows].double()
    cam, light = _f64(v.camera), _f64(prm["light_dir"])
    apex = x * smp.n + prm["normal_offset_voxels"] * nrm
    ax = torch.where((nrm[:, :1].abs() < np.float32(0.9)), _f64((1, 0, 0)), _f64((0, 1, 0)))
    T = torch.linalg.cross(ax, nrm)
    T = T / T.norm(dim=1, keepdim=True)
    B = torch.linalg.cross(nrm, T)
    one = torch.ones(len(rows), device=DEV, dtype=torch.float64)
    D = 0.0
    for d, wt in zip(_f64(prm["diffuse_dir"]), _f64(prm["diffuse_weight"])):
        D = D + wt * _march(smp, prm, apex, T * d[0] + B * d[1] + nrm * d[2], one * math.tan(prm["diffuse_aperture"] / 2),
                            first_hit=bool(prm["flags"] & vct.FLAG_DIFFUSE_FIRST_HIT))
    e = x - cam
    e = e / e.norm(dim=1, keepdim=True)
    R = e - 2 * (e * nrm).sum(1, keepdim=True) * nrm
    f = 0 * one
    if v.roughness is not None:
        f = ((v.roughness[rows].double() - prm["roughness_min"]) / (1 - prm["roughness_min"])).clamp(0, 1)
    g = prm["spec_aperture_min"] + f * (prm["spec_aperture_max"] - prm["spec_aperture_min"])
    S = _march(smp, prm, apex, R, torch.tan(g / 2))
    if prm["flags"] & vct.FLAG_SPEC_GRACE:
        ang = torch.acos(((R * light).sum(1) / (R.norm(dim=1) * light.norm())).clamp(-1, 1))
        k = (1 - (ang - 0.008 * math.pi * prm["shininess"]).clamp(min=0) / math.pi) ** prm["shininess_falloff"]
        S = torch.cat([S[:, :3] * k[:, None], S[:, 3:]], 1)
    vis = one
    if prm["occ_enable"]:
        vis = 1 - _march(smp, prm, apex, light.expand_as(x), one * math.tan(prm["occ_aperture"] / 2),
                         fade=bool(prm["flags"] & vct.FLAG_OCC_SMOOTH))[:, 3]
    px = v.width * v.height
    whole = lambda o, fill: torch.full((px,) + o.shape[1:], fill, device=DEV, dtype=torch.float64).index_put((rows,), o)  # noqa: E731
    out = {"diffuse": whole(D, 0.0), "specular": whole(S, 0.0), "visibility": whole(vis, 1.0)}
    if prm["flags"] & vct.FLAG_SHADE:
        kd, ks = prm["diffuse_str"], prm["specular_str"]
        alb = v.albedo[rows].double()
        nl = (nrm * light).sum(1, keepdim=True)
        wr = (-e * (2 * nl * nrm - light)).sum(1, keepdim=True).clamp(min=0)
        direct = _f64(prm["light_color"]) * alb * (kd * nl.clamp(min=0) + ks * wr ** prm["shininess"])
        if prm["flags"] & vct.FLAG_SHADE_IMPL:
            L = vis[:, None] * (D[:, :3] + direct) + S[:, :3]
        else:
            L = alb * (kd * D[:, :3] + ks * S[:, :3]) + vis[:, None] * direct
        out["radiance"] = whole(torch.cat([L, one[:, None]], 1), 0.0)
    return out


def _voxels64(case, mesh, light):
    """The voxel grid of the mesh: centres of dominant-axis pixels inside the triangle (vertices snapped to
    1/256 voxel, top-left rule), the depth's voxel, the highest triangle index wins."""
    n = case["n"]
    v, idx = mesh.vertices, mesh.indices.long()
    X = torch.round(v * float(256 * n)).long()[idx]  # [T, 3 vertices, 3 axes]
    e1, e2 = X[:, 1] - X[:, 0], X[:, 2] - X[:, 0]
    cross = lambda a, b: torch.stack([a[:, 1] * b[:, 2] - a[:, 2] * b[:, 1], a[:, 2] * b[:, 0] - a[:, 0] * b[:, 2],  # noqa: E731
                                      a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]], 1)
    N = cross(e1, e2)
    mag = N.abs()
    dom = torch.where((mag[:, 0] >= mag[:, 1]) & (mag[:, 0] >= mag[:, 2]), 0, torch.where(mag[:, 1] >= mag[:, 2], 1, 2))
    au, av = torch.tensor([2, 0, 0], device=DEV)[dom], torch.tensor([1, 2, 1], device=DEV)[dom]
    of = lambda t, a: t.gather(t.dim() - 1, a.reshape([-1] + [1] * (t.dim() - 1)).expand(t.shape[:-1] + (1,)))[..., 0]  # noqa: E731
    pu, pv = of(X, au), of(X, av)
    area = (pu[:, 1] - pu[:, 0]) * (pv[:, 2] - pv[:, 0]) - (pv[:, 1] - pv[:, 0]) * (pu[:, 2] - pu[:, 0])
    order = torch.where((area < 0)[:, None], torch.tensor([0, 2, 1], device=DEV), torch.tensor([0, 1, 2], device=DEV))
    qu, qv = pu.gather(1, order), pv.gather(1, order)
    lo = lambda t: ((t.min(1).values + 127) // 256).clamp(min=0)  # noqa: E731
    hi = lambda t: ((t.max(1).values - 128) // 256).clamp(max=n - 1)  # noqa: E731
    i0, j0 = lo(pu), lo(pv)
    w, h = (hi(pu) - i0 + 1).clamp(min=0), (hi(pv) - j0 + 1).clamp(min=0)
    cells = w * h * (area != 0)
    t = torch.repeat_interleave(torch.arange(len(cells), device=DEV), cells)
    k = torch.arange(len(t), device=DEV) - torch.repeat_interleave(cells.cumsum(0) - cells, cells)
    i, j = i0[t] + k % w[t], j0[t] + k // w[t]
    cu, cv = 256 * i + 128, 256 * j + 128
    ok = torch.ones_like(t, dtype=torch.bool)
    for a in range(3):
        b = (a + 1) % 3
        eu, ev = (qu[:, b] - qu[:, a])[t], (qv[:, b] - qv[:, a])[t]
        e = eu * (cv - qv[t, a]) - ev * (cu - qu[t, a])
        ok &= (e > 0) | ((e == 0) & ((ev < 0) | ((ev == 0) & (eu < 0))))
    Nu, Nv, Nd = of(N, au)[t], of(N, av)[t], of(N, dom)[t]
    num = -(Nu * (cu - pu[t, 0]) + Nv * (cv - pv[t, 0]))
    deep = (of(X, dom)[t, 0] + torch.div(num, torch.where(Nd == 0, 1, Nd), rounding_mode="floor")) // 256
    ok &= (deep >= 0) & (deep < n)
    d = dom[t]
    at = torch.where(d == 0, (i * n + j) * n + deep, torch.where(d == 1, (j * n + deep) * n + i, (deep * n + j) * n + i))
    owner = torch.zeros(n ** 3, dtype=torch.int64, device=DEV).scatter_reduce(0, at[ok], t[ok] + 1, "amax")
    p = v.double()[idx]
    face = torch.linalg.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0])
    length = face.norm(dim=1, keepdim=True)
    lam = ((face @ _f64(light["light_dir"]))[:, None] / torch.where(length > 0, length, torch.ones_like(length))).clamp(min=0)
    col = mesh.colors.double() * _f64(light["light_color"]) * (float(np.float32(light["ambient"])) + float(np.float32(light["diffuse_str"])) * lam)
    table = torch.cat([torch.zeros((1, 4), device=DEV, dtype=torch.float64),
                       torch.cat([col, torch.ones_like(lam)], 1)])
    return table[owner].reshape(n, n, n, 4)


def _gbuffer64(case, mesh, cam):
    """Nearest triangle along every pixel's ray, in 64 bits: position, normal, albedo [H*W,3]."""
    W, H = case["width"], case["height"]
    f, r, u, eye = (_f64(cam[k]) for k in ("forward", "right", "up", "eye"))
    th = cam["tan_half"]
    p = mesh.vertices.double()[mesh.indices.long()] - eye
    c = torch.stack([p @ r, p @ u, p @ f], -1)  # camera coordinates (orthonormal basis) [T,3,3]
    nrm = torch.linalg.cross(c[:, 1] - c[:, 0], c[:, 2] - c[:, 0])
    det = (c[:, 0] * nrm).sum(1)
    front = c[..., 2].min(1).values > 1e-3
    z = c[..., 2].clamp(min=1e-3)
    sx, sy = (c[..., 0] / z / (th * W / H) + 1) * W / 2 - 0.5, (1 - c[..., 1] / z / th) * H / 2 - 0.5
    x0, x1 = torch.where(front, sx.min(1).values.clamp(0, W).floor().long(), 0), torch.where(front, sx.max(1).values.clamp(-1, W - 1).ceil().long(), W - 1)
    y0, y1 = torch.where(front, sy.min(1).values.clamp(0, H).floor().long(), 0), torch.where(front, sy.max(1).values.clamp(-1, H - 1).ceil().long(), H - 1)
    seen = (c[..., 2].max(1).values > 0) & (det != 0)
    w, h = (x1.clamp(max=W - 1) - x0 + 1).clamp(min=0), (y1.clamp(max=H - 1) - y0 + 1).clamp(min=0)
    edges = torch.stack([torch.linalg.cross(c[:, (k + 1) % 3], c[:, (k + 2) % 3]) for k in range(3)], 1)
    depth = torch.full((H * W,), math.inf, device=DEV, dtype=torch.float64)
    best = torch.full((H * W,), len(c), device=DEV, dtype=torch.int64)
    tris = (seen & (w * h > 0)).nonzero()[:, 0]
    area = (w * h)[tris]
    # a triangle that reaches behind the eye is tried at every pixel: leave those that lie outside one side
    side = lambda a, lim, s: (s * c[tris, :, a] > lim * c[tris, :, 2].abs().clamp(min=1e-9)).all(1) & (c[tris, :, 2] > -1e9).all(1)  # noqa: E731
    out_ = side(0, th * W / H, 1) | side(0, th * W / H, -1) | side(1, th, 1) | side(1, th, -1)
    tris, area = tris[~out_], area[~out_]
    found = []
    part = (area.cumsum(0) // 50_000_000)
    for q in range(int(part.max()) + 1 if len(tris) else 0):
        tq, aq = tris[part == q], area[part == q]
        t = torch.repeat_interleave(tq, aq)
        k = torch.arange(len(t), device=DEV) - torch.repeat_interleave(aq.cumsum(0) - aq, aq)
        i, j = x0[t] + k % w[t], y0[t] + k // w[t]
        d = torch.stack([((2 * i + 1) / W - 1) * th * W / H, (1 - (2 * j + 1) / H) * th, torch.ones_like(i, dtype=torch.float64)], 1)
        s = det[t].sign()
        ok = torch.ones_like(i, dtype=torch.bool)
        for e in range(3):
            ok &= (edges[t, e] * d).sum(1) * s >= 0
        dist = det[t] / (nrm[t] * d).sum(1)
        ok &= dist > 0
        found.append((t[ok], (j * W + i)[ok], dist[ok]))
    if found:
        t, at, dist = (torch.cat(v) for v in zip(*found))
        depth = depth.scatter_reduce(0, at, dist, "amin")
        near = dist <= depth[at] * (1 + 1e-12)
        best = best.scatter_reduce(0, at[near], t[near], "amin")
    hit = best < len(c)
    b = best.clamp(max=len(c) - 1)
    i, j = torch.arange(H * W, device=DEV) % W, torch.arange(H * W, device=DEV) // W
    ray = f + (((2 * i + 1) / W - 1) * th * W / H)[:, None] * r + ((1 - (2 * j + 1) / H) * th)[:, None] * u
    keep = hit[:, None].double()
    pos = eye + torch.where(hit, depth, torch.zeros_like(depth))[:, None] * ray
    face = torch.linalg.cross(p[:, 1] - p[:, 0], p[:, 2] - p[:, 0])
    face = (face / face.norm(dim=1, keepdim=True))[b]
    face = face * torch.where((face * ray).sum(1, keepdim=True) > 0, -1.0, 1.0)
    return pos * keep, torch.nan_to_num(face) * keep, mesh.colors.double()[b] * keep


def exact(case, seed):
    st = prepare(case, seed)
    kind = case["kind"]
    if kind == "geometry":
        pos, nrm, alb = _gbuffer64(case, st["mesh"], st["cam"])
        return {"grid": _voxels64(case, st["mesh"], st["light"]), "position": pos, "normal": nrm, "albedo": alb,
                "mask": None, "triangle": None}
    if kind == "build":
        out = []
        for g in _mips(st["grid"], case["layout"]):
            code = _morton(g.shape[1])
            out.append(torch.stack([torch.empty_like(v.reshape(-1, 4)).index_copy_(0, code, v.reshape(-1, 4)) for v in g]).reshape(-1))
        return out
    if kind == "views":
        smp = [_Sampler(s["grid"], "dense") for s in st["scenes"]]
        return [_trace64(smp[v.pyramid], st["prm"], v) for v in st["views"]]
    if kind == "train":
        grid = st["grid"].detach().double().requires_grad_(True)
        total, outs = torch.zeros_like(grid), []
        for v, target in zip(st["views"], st["targets"]):  # one view at a time keeps what autograd holds small
            out = _trace64(_Sampler(grid, case["layout"]), st["prm"], v)
            loss = sum(0.5 * (o - t.double()).square().sum() for o, t in zip(out.values(), target))
            total += torch.autograd.grad(loss, grid)[0]
            outs.append({k: o.detach() for k, o in out.items()})
        return {"outputs": list(outs[0].values()) if case["how"] == "render" else outs, "grad": total}
    smp = _Sampler(st["grid"], case.get("layout", "dense"))
    out = _trace64(smp, st["prm"], st["view"])
    if kind == "host":
        return [[o.cpu() for o in out.values()] for _ in range(case["frames"])]
    return out
