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
