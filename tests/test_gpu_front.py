"""GPU parity of the tracer's fronts (the BVH cut that the rays of neighbouring
texels share): units of every size -- one texel to many, whole and partial --
trees smaller and deeper than a front, and rays that stop at a texel's
accumulated distance.  Both sides take every hit decision in fp32 with the
same operation order, so distances and counts are equal."""
import numpy as np
import pytest

import oracle
from synth import scenes as S

pytestmark = pytest.mark.gpu

BMIN = np.zeros(3, np.float32)


def _triangles(n):
    """n large triangles, stacked closely so that most boxes overlap."""
    z = 0.3 + 0.4 * np.arange(n, dtype=np.float32) / max(n, 2)
    v = np.stack([np.stack([np.array([a, b, 0], np.float32) + np.array([0, 0, k], np.float32)
                            for a, b in ((0.1, 0.1), (0.9, 0.2), (0.3, 0.9))]) for k in z])
    return v.reshape(-1, 3), np.arange(3 * n, dtype=np.int32).reshape(-1, 3)


def _unit(rt, R, chunk, blocks):
    """Rays of a unit: doubled from one texel's (32 at least) up to the chunk,
    512 rays and 32 texels, while every warp of the grid gets two units."""
    import torch
    total = rt.masked_count() * 8 * R
    warps = torch.cuda.get_device_properties(0).multi_processor_count * blocks * 4
    u, most = max(R, 32), min(chunk, 512, 32 * R)
    while 2 * u <= most and 2 * u * 2 * warps <= total:
        u *= 2
    return u


SCENES = {
    "one": lambda: _triangles(1),
    "two": lambda: _triangles(2),
    "stacked": lambda: _triangles(200),
    "soup": lambda: (lambda m: (m.verts, m.tris))(S.random_soup(3, 2500, size=0.3)),
    "room": lambda: (lambda m: (m.verts, m.tris))(S.room_scene(2, n_objects=20, n_spheres=8, subdiv=2)),
}


def _match(rt, scene, nc, R):
    verts, tris = SCENES[scene]()
    rt.upload_mesh(verts, tris)
    rt.build_bvh()
    pipe = oracle.FinePipeline(BMIN, 1.0, nc, 0.5, 2.0, 1.0, 7, accel="bvh")
    for t in range(2):
        rt.update(2.0, R, t)
        pipe.frame(verts, tris, t, R)
    rt.sync()
    g = rt.grids()
    cnt = g["counts"].cpu().numpy().astype(np.int64)
    assert np.array_equal(g["accum"].cpu().numpy().astype(np.float64), pipe.u)
    assert np.array_equal(cnt & 0xFFFF, pipe.nF) and np.array_equal(cnt >> 16, pipe.nB)


# (a full grid has more warps than these frames have units: the smallest ones,
# of 32 rays or one texel, up to 128 in the last but one)
@pytest.mark.parametrize("scene, nc, R, chunk", [
    ("one", 7, 4, 1024), ("two", 7, 1, 32), ("stacked", 9, 2, 64), ("stacked", 9, 64, 4096),
    ("soup", 11, 1, 1024), ("soup", 11, 16, 32), ("room", 13, 8, 256), ("room", 21, 32, 1024), ("room", 5, 1024, 64),
])
def test_units_and_fronts_match_the_oracle(scene, nc, R, chunk):
    from paper_2210_04449_gb300 import RTSDF
    rt = RTSDF(nc, seed=7)
    rt.set_tuning(ray_chunk=chunk)
    _match(rt, scene, nc, R)


@pytest.mark.parametrize("scene, nc, R, chunk, unit", [
    ("soup", 11, 16, 1024, 128), ("room", 28, 4, 1024, 128), ("room", 21, 32, 256, 256), ("room", 24, 16, 1024, 512),
    ("room", 21, 32, 1024, 512), ("stacked", 20, 64, 4096, 512),
])
def test_units_of_many_texels_match_the_oracle(scene, nc, R, chunk, unit):
    """One block per SM, so that units grow: 8 to 32 texels each, with fronts
    of 40 (below 256 rays) and 64 entries."""
    from paper_2210_04449_gb300 import RTSDF
    rt = RTSDF(nc, seed=7)
    rt.set_tuning(ray_chunk=chunk, trace_blocks_per_sm=1)
    _match(rt, scene, nc, R)
    assert _unit(rt, R, chunk, 1) == unit


def test_vote_does_not_depend_on_the_unit():
    """A full grid: units of one texel against units of 512 rays."""
    from paper_2210_04449_gb300 import RTSDF
    m = S.room_scene(3, n_objects=30, n_spheres=12, subdiv=2)
    out = []
    for chunk in (32, 1024):
        rt = RTSDF(56, seed=3)
        rt.set_tuning(ray_chunk=chunk)
        rt.upload_mesh(m.verts, m.tris)
        rt.build_bvh()
        for t in range(2):
            rt.update(2.0, 64, t)
        rt.sync()
        assert _unit(rt, 64, chunk, 8) == (64 if chunk == 32 else 512)
        out.append({k: rt.grids()[k].cpu().numpy().copy() for k in ("accum", "counts", "fine")})
    for k in out[0]:
        assert np.array_equal(out[0][k], out[1][k]), k


def test_nearest_face_does_not_depend_on_the_unit():
    """A unit's front is cut at its texels' largest accumulated distance; with
    a fading history (alpha < 1) that distance can be negative for some."""
    from paper_2210_04449_gb300 import RTSDF
    m = S.room_scene(3, n_objects=30, n_spheres=12, subdiv=2)
    out = []
    for chunk in (32, 1024):   # one texel a unit, and a whole coarse voxel and more
        rt = RTSDF(40, alpha=0.8, seed=3)
        rt.set_sign_mode("nearest")
        rt.set_tuning(ray_chunk=chunk)
        rt.upload_mesh(m.verts, m.tris)
        rt.build_bvh()
        for t in range(5):
            rt.update(2.0, 32, t)
        rt.sync()
        out.append({k: rt.grids()[k].cpu().numpy().copy() for k in ("accum", "counts", "fine")})
    u, c = out[0]["accum"], rt.grids()["coarse"].cpu().numpy().reshape(40, 40, 40)
    c = c.repeat(2, 0).repeat(2, 1).repeat(2, 2).reshape(-1)
    assert (0.8 * u + 0.2 * c < 0)[np.isfinite(u)].any()   # what the next frame's rays would start from
    for k in out[0]:
        assert np.array_equal(out[0][k], out[1][k]), k
