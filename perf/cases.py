"""What the SDF generator is measured on.

A case is one call sequence that a program using this library repeats: a frame
of the SDF update, the coarse SDF alone, a rebuilt tree with the exact
occlusion test, the shadow march and its adjoint, and a batched frame of many
scenes.  Scenes are procedural (a floor with walls and mixed objects, clouds
of displaced spheres), made on the GPU from the seed alone, with the sizes of
this repository's configurations and tests and odd ones between them.

``listed()`` and ``draw(rng)`` give cases, ``prepare(case, seed)`` what the
program holds before the call, ``run(state)`` one pass, ``work(case)`` the
bytes and operations of a pass, ``tolerance(case)`` what two correct
implementations may differ by, and ``exact(case, seed)`` the pass in 64 bits,
as plain torch gives it.
"""
import math

import numpy as np
import torch

DEV = "cuda"
BETA = 0.5      # Sec. 2.1 bias, coarse voxels
D_VOX = 2.0     # traced band, coarse voxels
FLOOR = 0.02    # floor and wall offset of a room


# ------------------------------------------------------------------- cases

def listed():
    return [
        # the smallest scene one would animate (a box and a ball): launches and latency
        dict(name="frame_tiny", kind="frame", scene="tiny", n=32, objects=2, lon=16, lat=11, rays=16, motion="static",
             builder="sah", sign="vote", alpha=1.0),
        # a static room converging over frames (128^3 -> 256^3, ~100k triangles, 64 rays)
        dict(name="frame_room", kind="frame", scene="room", n=128, objects=200, lon=32, lat=21, rays=64,
             motion="static", builder="sah", sign="vote", alpha=1.0),
        # a small animated scene of odd size: rigid transforms, refitted tree, fading history, nearest-face sign
        dict(name="frame_rigid_refit", kind="frame", scene="room", n=75, objects=61, lon=20, lat=13, rays=32,
             motion="rigid", builder="two_level", sign="nearest", alpha=0.9),
        # the benchmark frame: 256^3 -> 512^3, 1M triangles, every object moved, tree rebuilt, 64 rays
        dict(name="frame_moving_1m", kind="frame", scene="cloud", n=256, objects=500, lon=50, lat=21, rays=64,
             motion="move", builder="sah", sign="vote", alpha=1.0),
        # the coarse SDF alone, as a preview or for ambient occlusion: small and odd, and the largest grid
        dict(name="coarse_small", kind="coarse", scene="cloud", n=61, objects=12, lon=20, lat=13),
        dict(name="coarse_1m", kind="coarse", scene="cloud", n=256, objects=500, lon=50, lat=21),
        # objects moved, tree rebuilt, exact occlusion of an image: an editor's view, and a full frame
        dict(name="occlusion_small", kind="occlusion", scene="room", n=48, objects=20, lon=16, lat=9, width=320,
             height=200),
        dict(name="occlusion_room", kind="occlusion", scene="room", n=128, objects=200, lon=32, lat=21, width=1920,
             height=1080),
        # soft shadows: one full-HD image; a small jittered view resolved over time
        dict(name="shadow_1080p", kind="shadow", n=128, objects=60, width=1920, height=1080, steps=64, k=8.0,
             jitter=0.0),
        dict(name="shadow_taa", kind="shadow", n=45, objects=17, width=427, height=240, steps=48, k=4.0, jitter=2.0),
        # light and SDF optimisation: shadow image, squared error, gradients (512^3 grid, 1024^2 points)
        dict(name="shadow_grad", kind="shadow_grad", n=256, objects=60, width=1024, height=1024, steps=64, k=8.0),
        # many small scenes updated together
        dict(name="batch_24", kind="batch", scenes=24, n_max=128, objects=120, lon=16, lat=11, rays=32),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "coarse", "occlusion", "shadow", "shadow_grad", "batch"])
    if kind == "shadow":
        return dict(kind=kind, n=_log_int(rng, 12, 200), objects=rng.randint(3, 60), width=_log_int(rng, 64, 1920),
                    height=_log_int(rng, 64, 1080), steps=rng.randint(16, 96), k=rng.choice([2.0, 4.0, 8.0, 16.0]),
                    jitter=rng.choice([0.0, 0.0, 1.0, 2.0]))
    if kind == "shadow_grad":
        return dict(kind=kind, n=_log_int(rng, 16, 200), objects=rng.randint(3, 60), width=_log_int(rng, 64, 1024),
                    height=_log_int(rng, 64, 1024), steps=rng.randint(16, 64), k=rng.choice([2.0, 4.0, 8.0]))
    if kind == "batch":
        return dict(kind=kind, scenes=rng.randint(2, 24), n_max=_log_int(rng, 24, 128), objects=_log_int(rng, 4, 120),
                    lon=rng.randint(6, 24), lat=rng.randint(5, 15), rays=rng.choice([8, 16, 32]))
    scene = rng.choice(["room", "cloud"])
    lon, lat = rng.randint(6, 50), rng.randint(5, 21)
    objects = _log_int(rng, 2, 400 if scene == "cloud" else 200)
    c = dict(kind=kind, scene=scene, n=_log_int(rng, 12, 200), objects=objects, lon=lon, lat=lat)
    if kind == "occlusion":
        c.update(width=_log_int(rng, 64, 1920), height=_log_int(rng, 64, 1080))
    elif kind == "frame":
        c.update(rays=rng.choice([1, 4, 16, 32, 64]), motion=rng.choice(["static", "move", "rigid"]),
                 builder=rng.choice(["sah", "sah", "lbvh", "two_level"]), sign=rng.choice(["vote", "vote", "nearest"]),
                 alpha=rng.choice([1.0, 1.0, 0.9]))
    return c


# ------------------------------------------------------------------ scenes

def _sphere(lon, lat):
    """Unit UV sphere: vertices [V, 3] and outward triangles [2 lon (lat - 1), 3]."""
    th = np.pi * np.arange(1, lat)[:, None] / lat
    ph = 2 * np.pi * np.arange(lon)[None, :] / lon
    ring = np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th) + 0 * ph], -1).reshape(-1, 3)
    v = np.concatenate([[[0, 0, 1.0]], ring, [[0, 0, -1.0]]])
    j, south = np.arange(lon), len(v) - 1
    at = lambda i, k: 1 + i * lon + k % lon  # noqa: E731
    f = [np.stack([0 * j, at(0, j), at(0, j + 1)], -1)]
    for i in range(lat - 2):
        f += [np.stack([at(i, j), at(i + 1, j), at(i + 1, j + 1)], -1),
              np.stack([at(i, j), at(i + 1, j + 1), at(i, j + 1)], -1)]
    f.append(np.stack([0 * j + south, at(lat - 2, j + 1), at(lat - 2, j)], -1))
    return v, np.concatenate(f)


def _box():
    """Cube [-1, 1]^3: 8 vertices and 12 outward triangles."""
    v = np.array([[x, y, z] for z in (-1, 1) for y in (-1, 1) for x in (-1, 1)], np.float64)
    q = [(0, 2, 3, 1), (4, 5, 7, 6), (0, 1, 5, 4), (2, 6, 7, 3), (0, 4, 6, 2), (1, 3, 7, 5)]
    return v, np.array([t for a, b, c, d in q for t in ((a, b, c), (a, c, d))])


def _rotations(q):
    q = q / np.linalg.norm(q, axis=1, keepdims=True)
    w, x, y, z = q.T
    return np.stack([np.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)], -1),
                     np.stack([2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)], -1),
                     np.stack([2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], -1)], 1)


def _mesh(scene, objects, lon, lat, seed):
    """(verts float32 [V, 3], tris int32 [T, 3], object of each vertex int32 [V], number of objects), on the GPU."""
    rng = np.random.default_rng([seed, objects, lon, lat])
    if scene == "tiny":
        kinds, centre = np.array([0, 1]), np.array([[0.3, 0.3, 0.3], [0.7, 0.6, 0.65]]) + rng.uniform(-0.03, 0.03, (2, 3))
        size, rot = np.array([0.2, 0.15]), np.stack([np.eye(3)] * 2)
    else:
        kinds = np.ones(objects, int) if scene == "cloud" else (np.arange(objects) % 5 < 2).astype(int)
        centre = rng.uniform(0.1, 0.9, (objects, 3))
        top = 0.05 if scene == "cloud" else 0.1
        size = np.exp(rng.uniform(math.log(0.02), math.log(top), objects))
        rot = _rotations(rng.standard_normal((objects, 4)))
    amp = 0.1 if scene == "cloud" else 0.0
    vs, fs, ob, base = [], [], [], 0
    for kind, (tv, tf) in ((0, _box()), (1, _sphere(lon, lat))):
        ids = np.nonzero(kinds == kind)[0]
        if not len(ids):
            continue
        v = torch.tensor(tv, device=DEV)[None].expand(len(ids), -1, -1)
        if kind and amp:   # smooth radial displacement: a few waves over the sphere
            waves = torch.tensor(rng.standard_normal((len(ids), 4, 3)) * 3.0, device=DEV)
            phase = torch.tensor(rng.uniform(0, 6.283, (len(ids), 1, 4)), device=DEV)
            v = v * (1 + amp * 0.5 * torch.sin(v @ waves.transpose(1, 2) + phase).sum(-1, keepdim=True))
        v = (v * torch.tensor(size[ids], device=DEV)[:, None, None]) @ torch.tensor(rot[ids], device=DEV).transpose(1, 2)
        v = v + torch.tensor(centre[ids], device=DEV)[:, None, :]
        f = torch.tensor(tf, device=DEV)[None] + base + len(tv) * torch.arange(len(ids), device=DEV)[:, None, None]
        vs.append(v.reshape(-1, 3))
        fs.append(f.reshape(-1, 3))
        ob.append(torch.tensor(ids, device=DEV).repeat_interleave(len(tv)))
        base += len(ids) * len(tv)
    n_obj = len(kinds)
    if scene == "room":   # the floor and three walls, two triangles each, as one more object that stays
        lo, hi = FLOOR, 1 - FLOOR
        q = np.array([[(0, lo, 0), (0, lo, 1), (1, lo, 1), (1, lo, 0)], [(lo, 0, 0), (lo, 1, 0), (lo, 1, 1), (lo, 0, 1)],
                      [(hi, 0, 0), (hi, 0, 1), (hi, 1, 1), (hi, 1, 0)], [(0, 0, lo), (1, 0, lo), (1, 1, lo), (0, 1, lo)]])
        vs.append(torch.tensor(q.reshape(-1, 3), device=DEV))
        fs.append(torch.tensor([t for i in range(4) for t in ((4 * i, 4 * i + 1, 4 * i + 2), (4 * i, 4 * i + 2, 4 * i + 3))],
                               device=DEV) + base)
        ob.append(torch.full((16,), n_obj, device=DEV))
        n_obj += 1
    return (torch.cat(vs).float().contiguous(), torch.cat(fs).int().contiguous(), torch.cat(ob).int().contiguous(), n_obj)


def _motion(case, n_obj, seed):
    """Two opposite moves of every object but a room's walls, by at most half a coarse voxel, taken in turn so that
    the scene stays in place over any number of frames."""
    rng = np.random.default_rng([seed, 7])
    step = rng.standard_normal((n_obj, 3))
    step *= (0.5 / case["n"]) * rng.uniform(0, 1, (n_obj, 1)) ** (1 / 3) / np.linalg.norm(step, axis=1, keepdims=True)
    if case["scene"] == "room":
        step[-1] = 0
    if case.get("motion") != "rigid":
        return [torch.tensor(s * step, dtype=torch.float32, device=DEV) for s in (1, -1)]
    ang = rng.uniform(-0.3, 0.3, n_obj) / case["n"]
    if case["scene"] == "room":
        ang[-1] = 0
    out = []
    for s in (1, -1):
        m = np.zeros((n_obj, 3, 4))
        m[:, 0, 0] = m[:, 2, 2] = np.cos(ang)
        m[:, 0, 2], m[:, 2, 0], m[:, 1, 1] = s * np.sin(ang), -s * np.sin(ang), 1
        m[:, :, 3] = s * step
        out.append(torch.tensor(m, dtype=torch.float32, device=DEV))
    return out


def _balls(case, seed):
    rng = np.random.default_rng([seed, case["objects"], 11])
    c = torch.tensor(rng.uniform(0.1, 0.9, (case["objects"], 3)), device=DEV)
    return c, torch.tensor(np.exp(rng.uniform(math.log(0.02), math.log(0.1), case["objects"])), device=DEV)


def _grid_distance(n, balls):
    """Signed distance of the balls over the floor at the n^3 cell centres, float32 [z, y, x]."""
    x = ((torch.arange(n, device=DEV, dtype=torch.float64) + 0.5) / n).float()
    d = (x - FLOOR)[None, :, None].expand(n, n, n).clone()
    for (cx, cy, cz), r in zip(balls[0].tolist(), balls[1].tolist()):
        s = torch.sqrt((x - cx)[None, None, :] ** 2 + (x - cy)[None, :, None] ** 2 + (x - cz)[:, None, None] ** 2)
        d = torch.minimum(d, s - r)
    return d


def _fine_sdf(n, balls):
    """The fine grid (2n)^3 of such a scene as the update leaves it: distances near surfaces, the coarse voxel's
    value (one for its 8 texels, biased) elsewhere."""
    c = _grid_distance(n, balls)
    c8 = c.repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2)
    return torch.where(c8.abs() <= D_VOX / n, _grid_distance(2 * n, balls), c8 - BETA / n).reshape(-1).contiguous()


def _view(width, height, balls):
    """Points and normals of the scene seen from above (floor and ball tops), float32 [height, width, 3]."""
    x = ((torch.arange(width, device=DEV, dtype=torch.float64) + 0.5) / width)[None, :].expand(height, width)
    z = ((torch.arange(height, device=DEV, dtype=torch.float64) + 0.5) / height)[:, None].expand(height, width)
    y = torch.full_like(x, FLOOR)
    nrm = torch.zeros(height, width, 3, device=DEV, dtype=torch.float64)
    nrm[..., 1] = 1
    for c, r in zip(balls[0], balls[1]):
        q = r * r - (x - c[0]) ** 2 - (z - c[2]) ** 2
        top = torch.where(q > 0, c[1] + torch.sqrt(q.clamp(min=0)), -1.0)
        up = top > y
        y = torch.where(up, top, y)
        nrm = torch.where(up[..., None], torch.stack([x - c[0], top - c[1], z - c[2]], -1) / r, nrm)
    return torch.stack([x, y, z], -1).float().contiguous(), nrm.float().contiguous()


def _light(seed):
    rng = np.random.default_rng([seed, 13])
    return [float(np.float32(v)) for v in (rng.uniform(-0.6, 0.6), 1.0, rng.uniform(-0.6, 0.6))]


def _batch_sizes(case):
    """Grid size and object count of every scene: uneven, up to the case's."""
    rng = np.random.default_rng([case["scenes"], case["n_max"], case["objects"]])
    n = np.maximum(8, np.rint(case["n_max"] * rng.uniform(0.25, 1, case["scenes"])).astype(int))
    return n, np.maximum(2, np.rint(case["objects"] * np.exp(rng.uniform(-3, 0, case["scenes"]))).astype(int))


# ------------------------------------------------------------ prepare, run

def _views(rt, names, owner):
    """Views of a context's grids that a program keeps (integer grids as int32).  They are valid while their context
    lives, so each holds its owner."""
    g, out = rt.grids(), {}
    for k in names:
        out[k] = g[k].view(torch.int32) if k in ("seeds", "counts") else g[k]
        out[k].owner = owner
    return out


def _grids(rt, names=("seeds", "coarse", "fine", "accum", "counts")):
    """A frame's coarse part runs first, so that the views are those that every later frame writes."""
    rt.voxelize()
    rt.jfa()
    return _views(rt, names, rt)


def prepare(case, seed):
    from paper_2210_04449_gb300 import RTSDF, RTSDFBatch
    kind = case["kind"]
    s = dict(case=case, pass_=0)
    if kind in ("shadow", "shadow_grad"):
        balls = _balls(case, seed)
        s["rt"] = RTSDF(case["n"], beta_vox=BETA, seed=seed)
        s["sdf"] = _fine_sdf(case["n"], balls)
        s["pos"], s["nrm"] = _view(case["width"], case["height"], balls)
        s["light"] = _light(seed)
        if kind == "shadow_grad":
            s["sdf"].requires_grad_(True)
            s["light"] = torch.tensor(s["light"], requires_grad=True)
            s["target"] = _target(case, seed)
        else:
            s["vis"] = torch.empty(case["height"], case["width"], device=DEV)
            s["hist"] = torch.full((case["height"], case["width"]), 0.5, device=DEV)
        return s
    if kind == "batch":
        n, objects = _batch_sizes(case)
        s["rt"] = RTSDFBatch([dict(coarse_n=int(k), beta_vox=BETA, seed=seed + i) for i, k in enumerate(n)])
        s["rt"].set_tuning(split_trace=1)
        meshes = [_mesh("room" if i % 2 else "cloud", int(m), case["lon"], case["lat"], seed + 100 * i)
                  for i, m in enumerate(objects)]
        torch.cuda.synchronize()     # the batch uploads on a stream of its own
        for sc, (v, t, _, _) in zip(s["rt"].scenes, meshes):
            sc.upload_mesh(v, t)
            sc.build_bvh()
        s["rt"].frame(D_VOX, case["rays"], 0)
        s["rt"].sync()
        s["out"] = [_views(sc, ("fine", "counts"), s["rt"]) for sc in s["rt"].scenes]
        s["pass_"] = 1
        return s
    v, t, obj, n_obj = _mesh(case["scene"], case["objects"], case["lon"], case["lat"], seed)
    rt = s["rt"] = RTSDF(case["n"], beta_vox=BETA, alpha=case.get("alpha", 1.0), seed=seed)
    rt.upload_mesh(v, t)
    if kind == "coarse":
        s["out"] = _grids(rt, ("seeds", "coarse"))
        return s
    rt.set_objects(obj, n_obj)
    s["moves"] = _motion(case, n_obj, seed)
    if kind == "occlusion":
        s["pos"], s["nrm"] = _view(case["width"], case["height"], _balls(case, seed))
        s["light"] = _light(seed)
        s["blocked"] = torch.zeros(case["height"], case["width"], device=DEV, dtype=torch.uint8)
        rt.build_bvh()
        return s
    rt.set_bvh_builder(case["builder"])
    rt.set_sign_mode(case["sign"])
    rt.build_bvh()
    s["out"] = _grids(rt)
    rt.sync()
    return s


def run(s):
    case, rt, k = s["case"], s["rt"], s["pass_"]
    kind = case["kind"]
    s["pass_"] = k + 1
    if kind == "frame":
        if case["motion"] != "static":
            (rt.transform_objects if case["motion"] == "rigid" else rt.move_objects)(s["moves"][k % 2])
            rt.build_bvh(refit=case["builder"] == "two_level")
        rt.update(D_VOX, case["rays"], k)
        return s["out"]
    if kind == "coarse":
        rt.voxelize()
        rt.jfa()
        return s["out"]
    if kind == "occlusion":
        rt.move_objects(s["moves"][k % 2])
        rt.build_bvh()
        rt.shadow_fallback(s["pos"], s["nrm"], s["light"], blocked=s["blocked"])
        return s["blocked"]
    if kind == "shadow":
        rt.shadow(s["pos"], s["nrm"], s["light"], k=case["k"], steps=case["steps"], sdf=s["sdf"], out=s["vis"],
                  jitter_vox=case["jitter"], frame=k)
        if not case["jitter"]:
            return s["vis"]
        rt.taa_resolve(s["vis"], s["hist"], 0.1)
        return s["vis"], s["hist"]
    if kind == "shadow_grad":
        from paper_2210_04449_gb300 import soft_shadow
        vis = soft_shadow(rt, s["sdf"], s["light"], s["pos"], s["nrm"], k=case["k"], steps=case["steps"])
        loss = ((vis - s["target"]) ** 2).mean()
        dsdf, dlight = torch.autograd.grad(loss, (s["sdf"], s["light"]))
        return vis.detach(), dsdf, dlight
    rt.frame(D_VOX, case["rays"], k)
    return s["out"]


# -------------------------------------------------------- work, tolerance

def _tris(case):
    """Triangles of a case's scene (a batch: of one scene of the mean size)."""
    per = 2 * case["lon"] * (case["lat"] - 1)
    if case.get("scene") == "tiny":
        return 12 + per
    if case.get("scene") == "cloud":
        return case["objects"] * per
    return case["objects"] * (0.4 * per + 0.6 * 12) + 8


def _traced(case, n, objects, scene):
    """Texels of the traced band, from the surface area of the scene: a shell of 2 (d + beta) + 1 coarse voxels."""
    r2 = {"tiny": 0.08, "cloud": 0.0011, "room": 0.0033}[scene]
    area = objects * 4 * math.pi * r2 + (4.0 if scene == "room" else 0.0)
    return min(8.0 * n ** 3, 8 * area * n * n * (2 * (D_VOX + BETA) + 1))


def _ray_flops(tris):
    # a direction, then per level of a 4-wide tree four box tests (two slabs of six flops each), one triangle test
    return 60 + 4 * 12 * max(1.0, math.log(max(tris, 4), 4)) + 30


def work(case):
    kind = case["kind"]
    if kind in ("shadow", "shadow_grad"):
        pts, grid = case["width"] * case["height"], 4.0 * (2 * case["n"]) ** 3
        # a march takes about a third of its steps; a step is a trilinear sample (30 flops) and the penumbra (15);
        # it reads a slab of the grid above the view once
        flops = pts * case["steps"] / 3 * 45
        if kind == "shadow":
            return dict(bytes=28.0 * pts + 0.25 * grid + (12.0 * pts if case["jitter"] else 0), flops=flops)
        return dict(bytes=(28.0 + 28.0 + 12.0) * pts + 0.5 * grid + grid, flops=2.5 * flops)
    if kind == "batch":
        n, obj, frac = 0.65 * case["n_max"], case["objects"] * 0.32, case["scenes"]
        tris = obj * 2 * case["lon"] * (case["lat"] - 1) * 0.7
        tex = 0.5 * (_traced(case, n, obj, "room") + _traced(case, n, obj, "cloud"))
        return dict(bytes=frac * (24 * tris + 12 * n ** 3 + 4 * 8 * n ** 3 + 16 * tex),
                    flops=frac * tex * case["rays"] * _ray_flops(tris))
    tris, n3 = _tris(case), float(case["n"]) ** 3
    mesh = 12.0 * tris + 6.0 * tris
    if kind == "coarse":
        # mesh in, seeds and distances out; a distance to a candidate is 5 operations, 27 candidates a pass
        return dict(bytes=mesh + 8 * n3, flops=n3 * math.ceil(math.log2(case["n"])) * 27 * 5)
    build = mesh + 64.0 * tris + 43.0 * tris     # triangles in, leaf triangles and nodes out
    if kind == "occlusion":
        pts = case["width"] * case["height"]
        return dict(bytes=mesh + build + 25.0 * pts, flops=pts * _ray_flops(tris))
    tex = _traced(case, case["n"], case["objects"], case["scene"])
    # fine grid out, accumulator and counts of the traced texels in and out
    return dict(bytes=mesh + 8 * n3 + 32 * n3 + 16 * tex + (build if case["motion"] != "static" else 0),
                flops=tex * case["rays"] * _ray_flops(tris))


def tolerance(case):
    kind = case["kind"]
    if kind == "occlusion":
        return "exact"       # occlusion flags
    if kind == "coarse":
        return dict(rel=1e-6, max=1e-5, differ=0.0)     # seeds exact, one fp32 rounding chain per distance
    if kind in ("frame", "batch"):
        # distances to fp32 rounding; a ray that grazes an edge may hit on one side and miss on the other, which
        # changes a texel's count, and its distance where that hit was the nearest
        return dict(rel=1e-4, max=0.5, differ=1e-4)
    # a march that comes within rounding of a decision (h < eps) can end on either side; a texel's gradient is a sum
    # over few marches, each of which amplifies the rounding of its distances
    return dict(rel=2e-3 if kind == "shadow" else 2e-2, max=0.99)


# ------------------------------------------------------------------- exact

def _voxelize64(v, t, n):
    """Occupied voxels of the closed triangles on vertices quantised to 1/256 voxel: separating axes in int64."""
    q = torch.round((v.float() - 0.0) * float(n * 256)).long()[t.long()]            # [T, 3, 3]
    lo = torch.clamp(-((256 - q.amin(1)) // 256), min=0)
    hi = torch.clamp(q.amax(1) // 256, max=n - 1)
    cnt = (hi - lo + 1).clamp(min=0)
    total = cnt.prod(1)
    occ = torch.zeros(n ** 3, dtype=torch.bool, device=DEV)
    eye = torch.eye(3, dtype=torch.int64, device=DEV)
    order = torch.nonzero(total > 0).flatten()
    left = torch.cumsum(total[order], 0)
    cut = 0
    while cut < len(order):   # groups of triangles with at most 8M candidate voxels (or one triangle)
        done = int(left[cut - 1]) if cut else 0
        end = max(cut + 1, int(torch.searchsorted(left, torch.tensor(done + 8_000_000, device=DEV), right=True)))
        ids = order[cut:end].repeat_interleave(total[order[cut:end]])
        local = torch.arange(len(ids), device=DEV) - (left[cut:end] - total[order[cut:end]] - done).repeat_interleave(
            total[order[cut:end]])
        c = cnt[ids]
        vox = lo[ids] + torch.stack([local % c[:, 0], local // c[:, 0] % c[:, 1], local // (c[:, 0] * c[:, 1])], 1)
        p = q[ids] - (256 * vox + 128)[:, None, :]
        e = [p[:, 1] - p[:, 0], p[:, 2] - p[:, 1], p[:, 0] - p[:, 2]]
        ok = torch.ones(len(ids), dtype=torch.bool, device=DEV)
        for ax in [torch.linalg.cross(e[0], e[1])] + [torch.linalg.cross(a, u.expand_as(a)) for a in e for u in eye]:
            d, r = (p * ax[:, None, :]).sum(2), 128 * ax.abs().sum(1)
            ok &= (d.amin(1) <= r) & (d.amax(1) >= -r)
        occ[(vox[:, 0] + n * (vox[:, 1] + n * vox[:, 2]))[ok]] = True
        cut = end
    return occ


def _flood64(occ, n):
    """Jump flooding in int64: (squared distance, packed seed) of every voxel, -1 where there is none."""
    far = 1 << 40
    i = torch.arange(n, device=DEV)
    z, y, x = torch.meshgrid(i, i, i, indexing="ij")
    here = x | y << 8 | z << 16
    seed = torch.where(occ.view(n, n, n), here, far)
    k = 1 << max(0, math.ceil(math.log2(n)) - 1)
    d2 = torch.where(seed < far, 0, far)
    while k >= 1 and n > 1:
        best, out = torch.full_like(seed, far), torch.full_like(seed, far)
        for oz in (-k, 0, k):
            for oy in (-k, 0, k):
                for ox in (-k, 0, k):
                    if max(abs(ox), abs(oy), abs(oz)) >= n:
                        continue
                    to = tuple(slice(max(0, -o), n - max(0, o)) for o in (oz, oy, ox))
                    fr = tuple(slice(max(0, o), n - max(0, -o)) for o in (oz, oy, ox))
                    s = seed[fr]
                    d = ((s & 255) - x[to]) ** 2 + ((s >> 8 & 255) - y[to]) ** 2 + ((s >> 16 & 255) - z[to]) ** 2
                    d = torch.where(s < far, d, far)
                    b, o = best[to], out[to]
                    take = (d < b) | ((d == b) & (s < o))
                    best[to], out[to] = torch.where(take, d, b), torch.where(take, s, o)
        seed, d2 = out, best
        k >>= 1
    return d2, torch.where(seed < far, seed, -1)


def _coarse64(v, t, n):
    d2, seed = _flood64(_voxelize64(v, t, n), n)
    c = torch.where(seed >= 0, (torch.sqrt(d2.double()) - BETA) / n, math.inf)
    return seed.reshape(-1).int(), c.reshape(-1), d2.reshape(-1)


def _philox64(ctr, key):
    """Philox-4x32-10 over int64 tensors of 32-bit words."""
    m32 = 0xFFFFFFFF

    def mul(a, b):   # (high, low) 32-bit words of a 32 x 32 product
        lo = (a & 0xFFFF) * b
        hi = (a >> 16) * b + (lo >> 16)
        return hi >> 16 & m32, ((hi & 0xFFFF) << 16 | lo & 0xFFFF) & m32

    c, (k0, k1) = list(ctr), key
    for _ in range(10):
        h0, l0 = mul(c[0], 0xD2511F53)
        h1, l1 = mul(c[2], 0xCD9E8D57)
        c = [h1 ^ c[1] ^ k0, l1, h0 ^ c[3] ^ k1, l0]
        k0, k1 = (k0 + 0x9E3779B9) & m32, (k1 + 0xBB67AE85) & m32
    return c


def _directions64(texel, frame, rays, seed):
    """Marsaglia's sphere points from the counters (draw, ray, frame, texel): float64 [texels, rays, 3]."""
    tx = texel[:, None].expand(-1, rays)
    ray = torch.arange(rays, device=DEV)[None].expand_as(tx)
    out = torch.zeros(*tx.shape, 3, dtype=torch.float64, device=DEV)
    out[..., 2] = 1
    have = torch.zeros_like(tx, dtype=torch.bool)
    for draw_ in range(8):
        w = _philox64([torch.full_like(tx, draw_), ray, torch.full_like(tx, frame), tx],
                      (seed & 0xFFFFFFFF, seed >> 32))
        for a, b in ((w[0], w[1]), (w[2], w[3])):
            a, b = (2 * (u >> 9) + 1 - (1 << 23) for u in (a, b))
            ss = a * a + b * b
            take = (ss < 1 << 46) & ~have
            p, r, u = a.double() / 2 ** 23, b.double() / 2 ** 23, ss.double() / 2 ** 46
            root = 2 * torch.sqrt((1 - u).clamp(min=0))
            out = torch.where(take[..., None], torch.stack([p * root, r * root, 1 - 2 * u], -1), out)
            have |= take
    return out


def _trace64(v, t, n, masked, frame, rays, seed):
    """Nearest hit distance of every texel's rays over all triangles, and its front and back hit counts."""
    nf = 2 * n
    ch = torch.arange(8, device=DEV)
    px, py, pz = masked % n, masked // n % n, masked // (n * n)
    tx = ((2 * px[:, None] + (ch & 1)) + nf * ((2 * py[:, None] + (ch >> 1 & 1)) + nf * (2 * pz[:, None] + (ch >> 2))))
    tx = tx.reshape(-1)
    near = torch.full((len(tx),), math.inf, dtype=torch.float64, device=DEV)
    front, back = torch.zeros_like(tx), torch.zeros_like(tx)
    p = v.double()[t.long()]
    e1, e2 = p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]
    group = max(1, 30_000_000 // (rays * len(t)))
    for a in range(0, len(tx), group):
        g = tx[a:a + group]
        o = (torch.stack([g % nf, g // nf % nf, g // (nf * nf)], 1).double() + 0.5) / nf
        d = _directions64(g, frame, rays, seed)[:, :, None, :]
        pv = torch.linalg.cross(d, e2.expand(*d.shape[:2], -1, -1))
        det = (pv * e1).sum(-1)
        tv = (o[:, None, :] - p[:, 0])[:, None]
        u = (pv * tv).sum(-1) / det
        qv = torch.linalg.cross(tv, e1.expand_as(tv))
        w = (qv * d).sum(-1) / det
        s = (qv * e2).sum(-1) / det
        s = torch.where((u >= 0) & (w >= 0) & (u + w <= 1) & (s >= 0) & (det != 0), s, math.inf)
        best, at = s.min(-1)
        hit = torch.isfinite(best)
        f = torch.gather(det, -1, at[..., None])[..., 0] > 0
        near[a:a + group], front[a:a + group] = best.min(-1).values, (hit & f).sum(-1)
        back[a:a + group] = (hit & ~f).sum(-1)
    return tx, near, front, back


def _march64(case, sdf, pos, nrm, light, jitter=None):
    """The shadow march in 64 bits, differentiable in sdf and light; every point takes all steps under a mask."""
    nf = 2 * case["n"]
    h1, ln = 1.0 / nf, light / torch.linalg.vector_norm(light)
    o = pos.double().reshape(-1, 3) + 2 * h1 * nrm.double().reshape(-1, 3)
    if jitter is not None:
        o = o + jitter[:, None] * ln
    t = torch.zeros(len(o), dtype=torch.float64, device=DEV)
    res, ph = torch.ones_like(t), torch.full_like(t, 1e20)
    live, dark = torch.ones_like(t, dtype=torch.bool), torch.zeros_like(t, dtype=torch.bool)
    for _ in range(case["steps"]):
        q = o + t[:, None] * ln
        live = live & ((q >= 0) & (q <= 1)).all(1)
        if not bool(live.any()):
            break
        g = (q * nf - 0.5).clamp(0, nf - 1)
        b = g.detach().floor().clamp(0, nf - 2).long()
        f = g - b
        x0, x1 = b, b + 1
        at, w = [], []
        for c in range(8):
            i = [(x1 if c >> a & 1 else x0)[:, a] for a in range(3)]
            at.append(i[0] + nf * (i[1] + nf * i[2]))
            u = [(f[:, a] if c >> a & 1 else 1 - f[:, a]) for a in range(3)]
            w.append(u[0] * u[1] * u[2])
        h = (sdf[torch.stack(at)].double() * torch.stack(w)).sum(0)
        stop = live & (h < h1)
        dark, live = dark | stop, live & ~stop
        y = h * h / (2 * ph)
        a2 = h * h - y * y
        good = live & (t - y > 0)
        dd = torch.where(a2 > 0, torch.where(a2 > 0, a2, 1.0).sqrt(), 0.0)
        cand = torch.where(good, case["k"] * dd / torch.where(good, t - y, 1.0), math.inf)
        res = torch.where(cand < res, cand, res)
        ph = torch.where(live, h, ph)
        t = torch.where(live, t + h.clamp(max=4 * h1), t)
    res = torch.where(dark, 0.0, res.clamp(0, 1))
    return res.reshape(pos.shape[:-1])


def _target(case, seed):
    """The shadow image under the light turned by 5 degrees, that the optimisation aims at."""
    balls = _balls(case, seed)
    pos, nrm = _view(case["width"], case["height"], balls)
    x, y, z = _light(seed)
    c, s = math.cos(math.radians(5)), math.sin(math.radians(5))
    light = torch.tensor([c * x - s * y, s * x + c * y, z], dtype=torch.float64, device=DEV)
    return _march64(case, _fine_sdf(case["n"], balls), pos, nrm, light).float()


def exact(case, seed):
    kind = case["kind"]
    if kind in ("shadow", "shadow_grad"):
        balls = _balls(case, seed)
        sdf, (pos, nrm) = _fine_sdf(case["n"], balls), _view(case["width"], case["height"], balls)
        light = torch.tensor(_light(seed), dtype=torch.float64, device=DEV)
        if kind == "shadow_grad":
            sdf = sdf.double().requires_grad_(True)
            light.requires_grad_(True)
            vis = _march64(case, sdf, pos, nrm, light)
            loss = ((vis - _target(case, seed).double()) ** 2).mean()
            dsdf, dlight = torch.autograd.grad(loss, (sdf, light))
            return vis.detach(), dsdf, dlight
        if not case["jitter"]:
            return _march64(case, sdf, pos, nrm, light)
        i = torch.arange(case["width"] * case["height"], device=DEV)
        xi = _philox64([i, 0 * i, 0 * i, 0 * i + 0x53484457], (seed & 0xFFFFFFFF, seed >> 32))[0] >> 8
        vis = _march64(case, sdf, pos, nrm, light, xi.double() / 2 ** 24 * case["jitter"] / (2 * case["n"]))
        p = torch.nn.functional.pad(vis[None, None], (1, 1, 1, 1), mode="replicate")[0, 0].unfold(0, 3, 1).unfold(1, 3, 1)
        hc = torch.full_like(vis, 0.5).clamp(p.amin((2, 3)), p.amax((2, 3)))
        return vis, hc + 0.1 * (vis - hc)
    if kind in ("occlusion", "batch"):
        return None          # whole values; a batch is many frames
    v, t, obj, n_obj = _mesh(case["scene"], case["objects"], case["lon"], case["lat"], seed)
    n = case["n"]
    if case.get("motion", "static") != "static":     # the first pass's move, in fp32 as the entry point states it
        m = _motion(case, n_obj, seed)[0][obj.long()]
        v = v + m if m.dim() == 2 else \
            m[:, :, 0] * v[:, :1] + m[:, :, 1] * v[:, 1:2] + m[:, :, 2] * v[:, 2:] + m[:, :, 3]
    seeds, coarse, d2 = _coarse64(v, t, n)
    if kind == "coarse":
        return dict(seeds=seeds, coarse=coarse)
    # a frame: the coarse part always, the traced part where every ray can be tested against every triangle
    masked = torch.nonzero(d2 <= int((D_VOX + BETA) ** 2)).flatten()
    if 8.0 * len(masked) * case["rays"] * len(t) > 3e9 or case["sign"] != "vote" or case["alpha"] != 1.0:
        return dict(seeds=seeds, coarse=coarse, fine=None, accum=None, counts=None)
    tx, near, front, back = _trace64(v, t, n, masked, 0, case["rays"], seed)
    fine = coarse.view(n, n, n).repeat_interleave(2, 0).repeat_interleave(2, 1).repeat_interleave(2, 2).reshape(-1).clone()
    u = torch.where(torch.isfinite(near), near, fine[tx])
    accum, counts = torch.full_like(fine, math.inf), torch.zeros(len(fine), dtype=torch.int64, device=DEV)
    accum[tx], counts[tx] = near, front | back << 16
    fine[tx] = torch.where(back > front, -u, u)
    return dict(seeds=seeds, coarse=coarse, fine=fine, accum=accum, counts=counts.int())
