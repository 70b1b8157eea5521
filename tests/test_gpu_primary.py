"""The ray-cast G-buffer on both sides of the line between one ray per lane and packets, in pixels and
in triangles: the bits of the object-order producer, over either tree."""

import pytest

from synth import make_workload
from synth.scenes import scene_grass_field

pytestmark = pytest.mark.gpu


def _same(dof, ctx, sc, w, W, H):
    import torch
    cam = w.camera(0)
    want = dof.gbuffer(ctx, sc, cam, w.params, W, H, raster=True)
    for width in (4, 2):
        ctx.set_bvh_width(width)
        got = dof.gbuffer(ctx, sc, cam, w.params, W, H)
        torch.cuda.synchronize()
        assert int((want["prim"] >= 0).sum()) > 0
        for k in want:
            assert torch.equal(want[k], got[k]), (k, W, H, width)


@pytest.mark.parametrize("builder", ["ploc", "lbvh"])
def test_both_sides_of_the_line(builder):
    from paper_2210_06158_gb300 import dof
    ctx = dof.Context(0)
    ctx.set_bvh_builder(builder)
    # 2.8k triangles, four pixels each: the line lies near 140 x 80
    w = make_workload("c1", W=64, H=36)
    sc = dof.Scene(ctx, w.scene)
    for W, H in ((2, 2), (18, 10), (106, 102), (130, 90), (258, 146)):
        _same(dof, ctx, sc, make_workload("c1", W=W, H=H), W, H)
    # above 45k triangles it is 180,000 pixels: 600 x 300 (packets), 598 x 300 (one ray per lane)
    w = make_workload("c2", W=64, H=36, n_frames=1)
    sc = dof.Scene(ctx, scene_grass_field(w.params["albedo_seed"], 0.12, f_m=w.intr["f_m"], near=(1.2, 4.7)))
    assert sc.info().n_tris > 46_000
    for W, H in ((34, 18), (598, 300), (600, 300)):
        _same(dof, ctx, sc, make_workload("c2", W=W, H=H, n_frames=1), W, H)


@pytest.mark.parametrize("n", [0, 1, 2, 70])
def test_tiny_scenes_with_few_pixels(n):
    """No tree, a tree of one leaf, triangles kept out of the tree: one ray per lane and packets."""
    from paper_2210_06158_gb300 import dof
    import torch
    from synth import tiny_scene
    ctx = dof.Context(0)
    sc = dof.Scene(ctx, tiny_scene(500 + n, n, ties=n >= 8))
    w = make_workload("c1", W=64, H=36)
    for W, H in ((2, 2), (4, 2), (16, 16), (66, 34)):
        cam = make_workload("c1", W=W, H=H).camera(0)
        want = dof.gbuffer(ctx, sc, cam, w.params, W, H, raster=True)
        got = dof.gbuffer(ctx, sc, cam, w.params, W, H)
        torch.cuda.synchronize()
        for k in want:
            assert torch.equal(want[k], got[k]), (k, W, H)


def test_a_fine_mesh_over_part_of_the_image():
    """A ball of 60k triangles of a few pixels over a tenth of the image takes one ray per lane where the
    image alone would not: the same bits."""
    import numpy as np
    import torch
    from paper_2210_06158_gb300 import dof
    from synth import Camera, Scene, camera_pose
    rng = np.random.default_rng(4)
    d = rng.normal(size=(60_000, 3))
    at = np.array([0.4, 0.2, 10.0]) + d / np.linalg.norm(d, axis=1, keepdims=True)
    v = (at[:, None, :] + 0.01 * rng.uniform(-1, 1, (60_000, 3, 3))).astype(np.float32).reshape(-1, 3)
    ctx = dof.Context(0)
    sc = dof.Scene(ctx, Scene(v, np.arange(len(v), dtype=np.uint32).reshape(-1, 3), np.zeros(len(v) // 3, np.uint32), 1))
    cam = Camera.from_poses(dict(f_m=0.035, f_number=2.0, focus_m=10.0, sensor_w_m=0.036), camera_pose((0.0, 0.0, 0.0), 0.0))
    prm = make_workload("c2", W=64, H=36, n_frames=1).params
    for W, H in ((1280, 720), (1922, 1082)):
        want = dof.gbuffer(ctx, sc, cam, prm, W, H, raster=True)
        got = dof.gbuffer(ctx, sc, cam, prm, W, H)
        torch.cuda.synchronize()
        assert int((want["prim"] >= 0).sum()) > 10_000
        for k in want:
            assert torch.equal(want[k], got[k]), (k, W, H)
