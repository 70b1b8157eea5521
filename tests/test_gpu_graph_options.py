"""A captured step keeps the tracer's options of its capture: what the context is set to later
refuses a replay only where the captured launches could not run it."""

import numpy as np
import pytest

from synth import Scene, make_workload

pytestmark = pytest.mark.gpu

W, H = 130, 74


def _deep_scene():
    """Centres at halving distances along each axis: their Morton codes have one leading bit each, so
    the radix tree takes one triangle off per level."""
    c = np.zeros((61, 1, 3))
    for k in range(60):
        c[k, 0, k % 3] = 0.5 ** (k // 3)
    c += (0.0, 0.0, 4.0)
    v = (c + 1e-9 * np.array([[-1, -1, 0], [1, -1, 0], [0, 1, 0]])).astype(np.float32).reshape(-1, 3)
    return Scene(v, np.arange(len(v), dtype=np.uint32).reshape(-1, 3), np.zeros(len(v) // 3, np.uint32), 1)


def _item(ctx, scene=None):
    from paper_2210_06158_gb300 import dof
    w = make_workload("c1", W=W, H=H)
    sc = dof.Scene(ctx, scene if scene is not None else w.scene)
    gb = dof.gbuffer(ctx, sc, w.camera(0), w.params, W, H)
    return dict(scene=sc, gbuf=gb, cam=w.camera(0), params=dict(w.params), hist=dof.History(ctx, W, H, max_rays=1))


def _replays(ctx, g, item, n=2):
    """n replays give the images of the same frames enqueued directly on another history."""
    import torch
    from paper_2210_06158_gb300 import dof
    ref = dict(item, hist=dof.History(ctx, W, H, max_rays=1))
    item["hist"].reset()
    for _ in range(n):
        want = dof.batch_frame(ctx, [ref])[0].clone()
        got = g.launch([item])[0]
        torch.cuda.synchronize()
        assert torch.equal(want, got)


@pytest.mark.parametrize("packets", [0, 1])
def test_stack_request_of_the_capture_holds(packets):
    from paper_2210_06158_gb300 import dof
    ctx = dof.Context(0)
    item = _item(ctx)
    ctx.set_trace(packets=packets, stack=32)
    g = dof.Graph(ctx, [item])
    for later in (96, 64, 32):
        ctx.set_trace(stack=later)
        _replays(ctx, g, item)
    g.close()


def test_a_deeper_tree_than_the_captured_stack_is_refused():
    from paper_2210_06158_gb300 import dof
    ctx = dof.Context(0)
    item = _item(ctx)
    ctx.set_bvh_builder("lbvh")
    deep = dof.Scene(ctx, _deep_scene())
    assert item["scene"].info().depth <= 32 < deep.info().depth
    ctx.set_trace(packets=1, stack=32)
    g = dof.Graph(ctx, [item])
    with pytest.raises(dof.DofError) as e:
        g.launch([dict(item, scene=deep)])
    assert e.value.code == -7
    _replays(ctx, g, item)
    g.close()


def test_the_tree_width_does_not_matter_to_captured_packets():
    """Packets read the binary tree, whatever DOF_OPT_BVH_WIDTH says and whether there is a 4-wide
    one; one ray per lane is captured for one kind of tree."""
    from paper_2210_06158_gb300 import dof
    ctx = dof.Context(0)
    item = _item(ctx)
    one = _item(ctx, Scene(np.array([[-1, -1, 4], [1, -1, 4], [0, 1, 4]], np.float32), np.array([[0, 1, 2]], np.uint32),
                           np.zeros(1, np.uint32), 1))
    assert item["scene"].info().n_nodes4 > 0 == one["scene"].info().n_nodes4
    ctx.set_trace(packets=1)
    g = dof.Graph(ctx, [item])
    for width in (2, 4):
        ctx.set_bvh_width(width)
        _replays(ctx, g, item)
    _replays(ctx, g, dict(item, scene=one["scene"]))
    g.close()
    ctx.set_trace(packets=0, bvh_width=4)
    g = dof.Graph(ctx, [item])
    ctx.set_bvh_width(2)
    with pytest.raises(dof.DofError) as e:
        g.launch([item])
    assert e.value.code == -7
    g.close()
