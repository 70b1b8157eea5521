"""Which tracer runs on a context that leaves it open: the tree width does not pin it, nor does
tuning a scene's tree.  With its counters off the packet tracer reports no node visits, one ray per
lane always does."""

import pytest

from synth import make_workload

pytestmark = pytest.mark.gpu

W, H = 256, 144


def test_width_and_scene_tuning_leave_the_tracer_open():
    import torch
    from paper_2210_06158_gb300 import dof, tune
    ctx = dof.Context(0)
    ctx.set_trace(stats=False)
    w = make_workload("c1", W=W, H=H)
    sc = dof.Scene(ctx, w.scene)
    gb = dof.gbuffer(ctx, sc, w.camera(0), w.params, W, H)
    h = dof.History(ctx, W, H, max_rays=1)
    torch.cuda.synchronize()

    def packets():
        dof.frame(ctx, sc, gb, w.camera(0), w.params, h)
        st = h.stats()
        assert st.rays > 0
        return st.node_visits == 0

    assert packets()
    for width in (2, 4):
        ctx.set_bvh_width(width)
        assert packets(), width
    tuned, _, _ = tune.tune_scene(ctx, w.scene, lambda s, k: dof.frame(ctx, s, gb, w.camera(0), w.params, h), radii=[8, 48],
                                  frames=1)
    assert packets()
    ctx.set_trace(packets=False)
    assert not packets()
    ctx.set_trace(packets=True)
    assert packets()
    tuned.close()


@pytest.mark.parametrize("share,lanes", [(0.4, True), (0.2, False)])
def test_few_rays_through_a_wide_lens_stay_one_per_lane_in_a_dense_scene(share, lanes):
    """518k rays at cocK 8: one ray per lane with 200k triangles (whose packets are 10 to 15% slower),
    packets with 100k; the image is the same."""
    import torch
    from paper_2210_06158_gb300 import dof
    from synth.scenes import scene_grass_field
    w = make_workload("c3", W=960, H=540, n_frames=1)
    scene = scene_grass_field(w.params["albedo_seed"], share, f_m=w.intr["f_m"], near=(1.3, 4.8))
    prm = dict(w.params, spp=4)
    images = []
    for setting in (None, dict(packets=0), dict(packets=1)):
        ctx = dof.Context(0)
        ctx.set_trace(stats=False)
        if setting:
            ctx.set_trace(**setting)
        sc = dof.Scene(ctx, scene)
        gb = dof.gbuffer(ctx, sc, w.camera(0), prm, 960, 540)
        h = dof.History(ctx, 960, 540, max_rays=4)
        images.append(dof.frame(ctx, sc, gb, w.camera(0), prm, h))
        torch.cuda.synchronize()
        if setting is None:
            assert h.stats().rays > 100_000
            assert (h.stats().node_visits > 0) == lanes
    assert torch.equal(images[0], images[1]) and torch.equal(images[0], images[2])


@pytest.mark.parametrize("centre,lanes", [((0.0, 0.0, 1.0), True), ((0.0, 0.0, 12.0), False)])
def test_a_fine_mesh_in_the_blurred_foreground_is_traced_one_ray_per_lane(centre, lanes):
    """A ball of 20k small triangles in front of (or behind, where it takes no ray) a wall of 800
    large ones near the camera: its triangles are a fraction of what a packet covers.  518k rays, so
    that no other rule speaks; the image is the same either way."""
    import numpy as np
    import torch
    from paper_2210_06158_gb300 import dof
    from synth import Camera, Scene, camera_pose
    rng = np.random.default_rng(3)
    d = rng.normal(size=(20_000, 3))
    at = np.asarray(centre) + 0.3 * d / np.linalg.norm(d, axis=1, keepdims=True)
    ball = at[:, None, :] + 0.004 * rng.uniform(-1, 1, (20_000, 3, 3))
    wall = rng.uniform((-1.5, -1, 2.0), (1.5, 1, 2.5), (800, 3))[:, None, :] + 0.3 * rng.uniform(-1, 1, (800, 3, 3))
    v = np.concatenate([ball, wall] if lanes else [np.repeat(wall, 20, 0), ball[:4000]]).astype(np.float32).reshape(-1, 3)
    scene = Scene(v, np.arange(len(v), dtype=np.uint32).reshape(-1, 3), np.zeros(len(v) // 3, np.uint32), 1)
    cam = Camera.from_poses(dict(f_m=0.035, f_number=2.0, focus_m=10.0, sensor_w_m=0.036), camera_pose((0.0, 0.0, 0.0), 0.0))
    prm = dict(make_workload("c2", W=64, H=36, n_frames=1).params, spp=1)
    images = []
    for setting in (None, dict(packets=0), dict(packets=1)):
        ctx = dof.Context(0)
        ctx.set_trace(stats=False)
        if setting:
            ctx.set_trace(**setting)
        sc = dof.Scene(ctx, scene)
        gb = dof.gbuffer(ctx, sc, cam, prm, 1920, 1080)
        h = dof.History(ctx, 1920, 1080, max_rays=1)
        images.append(dof.frame(ctx, sc, gb, cam, prm, h))
        torch.cuda.synchronize()
        if setting is None:
            assert h.stats().rays > 10_000
            assert (h.stats().node_visits > 0) == lanes
    assert torch.equal(images[0], images[1]) and torch.equal(images[0], images[2])
