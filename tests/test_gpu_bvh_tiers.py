"""The SAH build at the edges of its tiers (warp, block, levels) and on meshes
whose splits are far off the middle, so that a build takes more than one batch
of levels, top-down and in the 4-wide collapse: every tree is valid over all
triangles, and the distances traced through it equal the oracle's."""
import numpy as np
import pytest

import oracle
from tests.test_gpu_bvh import _check_tree

pytestmark = pytest.mark.gpu


def _soup(n, seed=5):
    rng = np.random.default_rng(seed)
    c = rng.uniform(0.1, 0.9, (n, 1, 3))
    return c + rng.uniform(-0.03, 0.03, (n, 3, 3))


def _geometric(n):
    """Triangles that shrink and close in on a corner by a constant factor."""
    f = 0.993 ** np.arange(n)[:, None, None]
    shape = np.array([[0.0, 0, 0], [0.02, 0, 0.01], [0, 0.02, 0.005]])[None]
    return 0.1 + f * (0.8 * np.array([1.0, 0.6, 0.3])[None, None] + shape)


@pytest.mark.parametrize("name, n", [("soup", n) for n in (2, 3, 31, 32, 33, 64, 255, 256, 257, 513, 1024, 1025, 4099)] +
                         [("geometric", 700), ("geometric", 3000)])
def test_tiers(name, n):
    from paper_2210_04449_gb300 import RTSDF
    v = (_soup(n) if name == "soup" else _geometric(n)).reshape(-1, 3).astype(np.float32)
    t = np.arange(3 * n, dtype=np.int32).reshape(-1, 3)
    nc, R = 8, 8
    rt = RTSDF(nc, seed=2)
    rt.upload_mesh(v, t)
    rt.build_bvh()
    ch, lt, root = rt.bvh_topology()
    _check_tree(ch, lt, root, n)
    rt.update(2.0, R, 0)
    rt.sync()
    pipe = oracle.FinePipeline(np.zeros(3, np.float32), 1.0, nc, 0.5, 2.0, 1.0, 2, accel="bvh")
    pipe.frame(v, t, 0, R)
    assert np.array_equal(rt.grids()["accum"].cpu().numpy().astype(np.float64), pipe.u)


@pytest.mark.parametrize("n", [200000, 200001, 500000, 500001])
def test_large_meshes(n):
    # either side of the mesh sizes at which the build's block tier and its
    # chunks change: the SAH and the two-level tree (an object of most of the
    # triangles, one of 300, one of 2) trace the same grids as the Morton tree
    from paper_2210_04449_gb300 import RTSDF
    rng = np.random.default_rng(n)
    c = rng.uniform(0.1, 0.9, (n, 1, 3))
    v = (c + rng.uniform(-0.004, 0.004, (n, 3, 3))).reshape(-1, 3).astype(np.float32)
    t = np.arange(3 * n, dtype=np.int32).reshape(-1, 3)
    obj = np.zeros(3 * n, np.int32)
    obj[:900], obj[-6:] = 1, 2
    got = {}
    for builder in ("lbvh", "sah", "two_level"):
        rt = RTSDF(10, seed=2)
        rt.upload_mesh(v, t)
        rt.set_objects(obj, 3)
        rt.set_bvh_builder(builder)
        rt.build_bvh()
        rt.update(2.0, 4, 0)
        rt.sync()
        got[builder] = {k: rt.grids()[k].cpu().numpy() for k in ("accum", "counts", "fine")}
        rt.close()
    assert got["lbvh"]["counts"].any()
    for builder in ("sah", "two_level"):
        for k, ref in got["lbvh"].items():
            assert np.array_equal(got[builder][k], ref), (builder, k)


@pytest.mark.parametrize("builder", ["sah", "two_level"])
@pytest.mark.parametrize("n", [700, 5000])
def test_moves_out_of_all_range(builder, n):
    # a move to NaN, to infinity or so far that areas overflow is an error at
    # the next sync, and a build before it still makes a valid tree: the splits
    # of ranges that hold such triangles, alone or among others, are the same
    # for every lane
    from paper_2210_04449_gb300 import RTSDF, RtsdfError
    v = _soup(n).reshape(-1, 3).astype(np.float32)
    t = np.arange(3 * n, dtype=np.int32).reshape(-1, 3)
    obj = (np.arange(3 * n, dtype=np.int32) // 3) % 50
    rt = RTSDF(8, seed=2)
    rt.set_bvh_builder(builder)
    rt.upload_mesh(v, t)
    rt.set_objects(obj, 50)
    by = np.zeros((50, 3), np.float32)
    by[::7, 0] = np.nan
    by[3] = np.inf
    by[11, 1], by[12, 2], by[13] = 3e38, -3e38, 1e25
    rt.move_objects(by)
    rt.build_bvh()
    ch, lt, root = rt.bvh_topology()
    _check_tree(ch, lt, root, n, in_order=builder == "sah")
    with pytest.raises(RtsdfError) as ei:
        rt.sync()
    assert ei.value.name == "RTSDF_E_MESH"
    rt.upload_mesh(v, t)
    rt.build_bvh()
    rt.update(2.0, 8, 0)
    rt.sync()
    pipe = oracle.FinePipeline(np.zeros(3, np.float32), 1.0, 8, 0.5, 2.0, 1.0, 2, accel="bvh")
    pipe.frame(v, t, 0, 8)
    assert np.array_equal(rt.grids()["accum"].cpu().numpy().astype(np.float64), pipe.u)
