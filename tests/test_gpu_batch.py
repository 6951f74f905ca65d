"""Batched form: one persistent launch per frame for many uneven scenes must
give every scene exactly the grids of a plain per-scene frame (the same
arithmetic on the same rays), with and without CUDA-graph replay; a bounded
grid-barrier wait that runs out is reported as RTSDF_E_TIMEOUT and the next
frame is correct again."""
import numpy as np
import pytest

from synth import scenes as S
from tests._util import seeds_to_linear

pytestmark = pytest.mark.gpu


def _workload():
    """Seven scenes of uneven grid size and triangle count (one empty, one 1^3)."""
    items = [
        (dict(coarse_n=16, beta_vox=0.5, seed=1), S.tiny_scene()),
        (dict(coarse_n=37, beta_vox=0.25, seed=2), S.random_soup(5, 400, size=0.05)),
        (dict(coarse_n=48, beta_vox=0.5, seed=3, alpha=0.5), S.room_scene(7, n_objects=12, n_spheres=5, subdiv=2)),
        (dict(coarse_n=24, beta_vox=1.0, seed=4), S.merge([S.box_mesh((0.5, 0.5, 0.5), 0.3)])),
        (dict(coarse_n=1, beta_vox=0.5, seed=5), S.tiny_scene()),
        (dict(coarse_n=8, beta_vox=0.5, seed=6), S.Mesh(np.zeros((0, 3), np.float32), np.zeros((0, 3), np.int32))),
        (dict(coarse_n=64, beta_vox=0.5, seed=7), S.animated_scene(9, n_objects=20, n_lon=16, n_lat=9)),
    ]
    return items


def _grids(rt):
    g = rt.grids()
    n = rt.coarse_n
    m = rt.masked_count()
    return {"seeds": seeds_to_linear(g["seeds"].cpu().numpy(), n), "coarse": g["coarse"].cpu().numpy(),
            "accum": g["accum"].cpu().numpy(), "counts": g["counts"].cpu().numpy(),
            "fine": g["fine"].cpu().numpy(), "masked": np.sort(g["masked"].cpu().numpy()[:m])}


def _run_plain(items, frames, d, R):
    from paper_2210_04449_gb300 import RTSDF
    out = []
    for cfg, mesh in items:
        rt = RTSDF(**cfg)
        rt.upload_mesh(mesh.verts, mesh.tris)
        rt.build_bvh()
        for f in frames:
            rt.update(d, R, f)
        rt.sync()
        out.append(_grids(rt))
        rt.close()
    return out


def _make_batch(items):
    from paper_2210_04449_gb300 import RTSDFBatch
    b = RTSDFBatch([cfg for cfg, _ in items])
    for sc, (_, mesh) in zip(b.scenes, items):
        sc.upload_mesh(mesh.verts, mesh.tris)
        sc.build_bvh()
    return b


@pytest.mark.parametrize("use_graph,split", [(1, 0), (0, 0), (1, 1), (0, 1)])
def test_batch_equals_sequential(use_graph, split):
    # split = 1: the trace (with Eq. 1) runs as a launch of its own after the
    # pipeline launch; the grids must not change
    items = _workload()
    d, R, frames = 2.0, 8, [0, 1, 2]
    b = _make_batch(items)
    b.set_tuning(use_graph=use_graph, split_trace=split)
    assert b.get_tuning()["split_trace"] == split
    for f in frames:
        b.frame(d, R, f)
    b.sync()
    info = b.stats()
    if use_graph:
        print("batch graph replay:", info)
    ref = _run_plain(items, frames, d, R)
    for i, sc in enumerate(b.scenes):
        got = _grids(sc)
        for k in ("seeds", "coarse", "accum", "counts", "fine", "masked"):
            assert np.array_equal(got[k], ref[i][k]), (i, k)
    assert info["frames"] == len(frames)
    b.close()


@pytest.mark.parametrize("split", [0, 1])
def test_batch_barrier_timeout_reported_then_recovers(split):
    # with split = 1 the flood's and the trace's launches see the abort flag
    # and skip their work
    from paper_2210_04449_gb300 import RtsdfError
    items = _workload()
    d, R = 2.0, 4
    b = _make_batch(items)
    b.set_tuning(barrier_spins=1, use_graph=0, split_trace=split)
    b.frame(d, R, 0)
    with pytest.raises(RtsdfError) as ei:
        b.sync()
    assert ei.value.name == "RTSDF_E_TIMEOUT"
    b.set_tuning(barrier_spins=0)
    for f in (0, 1):
        b.frame(d, R, f)
    b.sync()
    ref = _run_plain(items, [0, 1], d, R)
    for i, sc in enumerate(b.scenes):
        got = _grids(sc)
        for k in ("seeds", "accum", "counts", "fine"):
            assert np.array_equal(got[k], ref[i][k]), (i, k)
    b.close()


@pytest.mark.parametrize("split", [0, 1])
def test_batch_nearest_face_variant_equals_sequential(split):
    # scenes in the nearest-face mode (and one left in the vote mode) give the
    # grids of plain per-scene frames in the same modes
    items = _workload()
    d, R, frames = 2.0, 8, [0, 1, 2]
    b = _make_batch(items)
    b.set_tuning(split_trace=split)
    for i, sc in enumerate(b.scenes):
        if i != 2:
            sc.set_sign_mode("nearest")
    for f in frames:
        b.frame(d, R, f)
    b.sync()
    from paper_2210_04449_gb300 import RTSDF
    for i, ((cfg, mesh), sc) in enumerate(zip(items, b.scenes)):
        rt = RTSDF(**cfg)
        if i != 2:
            rt.set_sign_mode("nearest")
        rt.upload_mesh(mesh.verts, mesh.tris)
        rt.build_bvh()
        for f in frames:
            rt.update(d, R, f)
        rt.sync()
        want, got = _grids(rt), _grids(sc)
        for k in ("accum", "counts", "fine", "masked"):
            assert np.array_equal(got[k], want[k]), (i, k)
        rt.close()
    b.close()


@pytest.mark.parametrize("split", [0, 1])
def test_batch_with_any_builder_and_a_one_triangle_scene(split):
    # scenes built by every builder (the animated one two-level, over its
    # objects) plus a scene of a single triangle: the grids of plain frames
    from paper_2210_04449_gb300 import RTSDFBatch
    one = S.Mesh(np.array([[0.3, 0.4, 0.3], [0.7, 0.45, 0.35], [0.4, 0.5, 0.7]], np.float32),
                 np.array([[0, 1, 2]], np.int32))
    items = _workload() + [(dict(coarse_n=16, beta_vox=0.5, seed=8), one)]
    d, R, frames = 2.0, 8, [0, 1]
    b = RTSDFBatch([cfg for cfg, _ in items])
    b.set_tuning(split_trace=split)
    builders = ["sah", "lbvh", "two_level", "lbvh", "sah", "two_level", "two_level", "sah"]
    for i, (sc, (_, mesh)) in enumerate(zip(b.scenes, items)):
        sc.set_bvh_builder(builders[i])
        sc.upload_mesh(mesh.verts, mesh.tris)
        if mesh.vert_object is not None and mesh.n_objects > 0:
            sc.set_objects(mesh.vert_object, mesh.n_objects)
        sc.build_bvh()
    for f in frames:
        b.frame(d, R, f)
    b.sync()
    ref = _run_plain(items, frames, d, R)
    for i, sc in enumerate(b.scenes):
        got = _grids(sc)
        for k in ("seeds", "accum", "counts", "fine", "masked"):
            assert np.array_equal(got[k], ref[i][k]), (i, k)
    assert (ref[-1]["counts"] != 0).any()                  # the one-triangle scene was hit
    b.close()


def test_batch_matches_oracle():
    # the batched frames against the oracle itself (Sec. 2.1-2.2, Eq. 1),
    # not only against plain GPU frames: four of the uneven scenes --
    # including the non-power-of-two 37^3 grid and the alpha = 0.5 decay --
    # on 400 texels each sampled from the oracle's own frame-0 mask, three
    # frames of 8 rays; the bar of the per-scene trace tests (distances
    # within 2e-5 x diagonal, counts equal, grazing mismatches < 1e-4)
    import oracle
    items = _workload()
    pick = [0, 1, 2, 6]
    d, R, frames = 2.0, 8, [0, 1, 2]
    b = _make_batch(items)
    b.set_tuning(split_trace=1)
    for f in frames:
        b.frame(d, R, f)
    b.sync()
    bmin = np.zeros(3, np.float32)
    tol = 2e-5 * np.sqrt(3.0)
    for i in pick:
        cfg, mesh = items[i]
        nc, beta, alpha, seed = cfg["coarse_n"], cfg["beta_vox"], cfg.get("alpha", 1.0), cfg["seed"]
        occ = oracle.voxelize(mesh.verts, mesh.tris, bmin, 1.0, nc)
        seeds, _ = oracle.jfa(occ, nc)
        c = oracle.coarse_sdf(seeds, nc, 1.0, beta)
        mask, _ = oracle.mask_fill(seeds, nc, d, beta, c)
        tex = np.nonzero(mask)[0]
        track = np.sort(np.random.default_rng(100 + i).choice(tex, min(400, tex.size), replace=False))
        assert track.size >= 256
        pipe = oracle.FinePipeline(bmin, 1.0, nc, beta, d, alpha, seed, track=track, accel="bvh")
        for f in frames:
            pipe.frame(mesh.verts, mesh.tris, f, R)
        g = b.scenes[i].grids()
        u = g["accum"].cpu().numpy().astype(np.float64)[track]
        cnt = g["counts"].cpu().numpy().astype(np.int64)[track]
        fg = g["fine"].cpu().numpy().astype(np.float64)[track]
        both_inf = np.isinf(u) & np.isinf(pipe.u)
        with np.errstate(invalid="ignore"):
            du = np.where(both_inf, 0.0, np.abs(u - pipe.u))
        bad = (du > tol) | ((cnt & 0xFFFF) != pipe.nF) | ((cnt >> 16) != pipe.nB) | (np.abs(fg - pipe.f) > tol)
        print(f"batched scene {i} (nc={nc}, alpha={alpha}): texels={track.size} mismatched={int(bad.sum())} "
              f"hit={np.isfinite(pipe.u).mean():.2f}")
        assert bad.mean() <= 1e-4, (i, int(bad.sum()))
        assert np.isfinite(pipe.u).mean() > 0.5
    b.close()


def _shifted(mesh, by):
    return S.Mesh((mesh.verts + np.asarray(by, np.float32)).astype(np.float32), mesh.tris)


@pytest.mark.parametrize("use_graph,split", [(1, 0), (0, 0), (1, 1)])
@pytest.mark.parametrize("single", [True, False])
def test_batch_follows_rebuilt_and_refitted_trees(use_graph, split, single):
    # a rebuild after an upload of the same size, and a refit, keep every
    # pointer and count of a scene: the batch's copy of the tree must follow
    # them all the same (a batch of one scene has no later scene's offset that
    # could tell either)
    from paper_2210_04449_gb300 import RTSDF
    items = _workload()[1:2] if single else _workload()[1:4]
    d, R = 2.0, 8
    b = _make_batch(items)
    b.set_tuning(use_graph=use_graph, split_trace=split)
    plain = []
    for cfg, mesh in items:
        rt = RTSDF(**cfg)
        rt.upload_mesh(mesh.verts, mesh.tris)
        rt.build_bvh()
        plain.append(rt)

    def frame_and_compare(f, step):
        b.frame(d, R, f)
        b.sync()
        for i, (sc, rt) in enumerate(zip(b.scenes, plain)):
            rt.update(d, R, f)
            rt.sync()
            got, want = _grids(sc), _grids(rt)
            for k in ("seeds", "coarse", "accum", "counts", "fine", "masked"):
                assert np.array_equal(got[k], want[k]), (step, i, k)

    frame_and_compare(0, "first")
    last = len(items) - 1
    cfg, mesh = items[last]
    moved = _shifted(mesh, (0.03, -0.02, 0.04))
    for rt in (b.scenes[last], plain[last]):
        rt.upload_mesh(moved.verts, moved.tris)
        rt.build_bvh()
    frame_and_compare(1, "same-size upload")
    for scene in (0, last):
        for rt in (b.scenes[scene], plain[scene]):
            rt.set_reset(False)
            rt.set_objects(np.zeros(items[scene][1].verts.shape[0], np.int32), 1)
            rt.move_objects(np.array([[-0.05, 0.03, 0.01]], np.float32))
            rt.build_bvh(refit=True)
    frame_and_compare(2, "refit")
    for rt in plain:
        rt.close()
    b.close()


@pytest.mark.parametrize("split", [0, 1])
def test_batch_follows_two_level_refits(split):
    # a two-level refit collapses the tree anew: the number of its 4-wide nodes
    # may change, also in the last scene, where no later offset shows it
    from paper_2210_04449_gb300 import RTSDF, RTSDFBatch
    d, R = 2.0, 8
    meshes = [S.animated_scene(k, n_objects=15, n_lon=12, n_lat=7) for k in (4, 5)]
    b = RTSDFBatch([dict(coarse_n=24, seed=k) for k in range(2)])
    b.set_tuning(split_trace=split)
    plain = [RTSDF(24, seed=k) for k in range(2)]
    for rts in (b.scenes, plain):
        for rt, m in zip(rts, meshes):
            rt.set_bvh_builder("two_level")
            rt.upload_mesh(m.verts, m.tris)
            rt.set_objects(m.vert_object, m.n_objects)
            rt.set_reset(False)
            rt.build_bvh()
    rng = np.random.default_rng(2)
    for f in range(4):
        b.frame(d, R, f)
        b.sync()
        for sc, rt in zip(b.scenes, plain):
            rt.update(d, R, f)
            rt.sync()
            got, want = _grids(sc), _grids(rt)
            for k in ("accum", "counts", "fine", "masked"):
                assert np.array_equal(got[k], want[k]), (f, k)
        for i, m in enumerate(meshes):
            by = rng.uniform(-0.02, 0.02, (m.n_objects, 3)).astype(np.float32)
            for rt in (b.scenes[i], plain[i]):
                rt.move_objects(by)
                rt.build_bvh(refit=True)
    for rt in plain:
        rt.close()
    b.close()


@pytest.mark.parametrize("split", [0, 1])
def test_batch_pipeline_blocks_per_sm(split):
    # the pipeline launch is bounded to registers for eight blocks per SM; its
    # shared memory (the tracer's state in the single-launch form) must let
    # eight in too
    import torch
    b = _make_batch(_workload()[:2])
    b.set_tuning(split_trace=split, blocks_per_sm=0)
    b.frame(2.0, 4, 0)
    b.sync()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert b.stats()["grid"] >= 8 * sms
    b.close()
