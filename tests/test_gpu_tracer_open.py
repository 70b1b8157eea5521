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
