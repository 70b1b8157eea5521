"""A context that leaves the tracer open gives the images of either tracer, on both sides of
the library's rule (narrow and wide apertures, few and many rays, a mixed batch), and a graph
captured under it keeps replaying when the cameras would now choose the other one."""

import numpy as np
import pytest

from synth import make_workload

pytestmark = pytest.mark.gpu


def _session(dof, ctx, name, W, H, spp, frames=3):
    import torch
    w = make_workload(name, W=W, H=H, n_frames=frames)
    prm = dict(w.params, spp=spp)
    sc = dof.Scene(ctx, w.scene)
    gbs = [dof.gbuffer(ctx, sc, w.camera(k), prm, W, H) for k in range(frames)]
    h = dof.History(ctx, W, H, max_rays=spp, record_rays=True)
    torch.cuda.synchronize()
    return w, prm, sc, gbs, h


@pytest.mark.parametrize("name,W,H,spp", [("c2", 322, 182, 1), ("c2", 322, 182, 4), ("c3", 322, 182, 1), ("c3", 642, 362, 16),
                                          ("bokeh", 256, 144, 4)])
def test_open_tracer_equals_either(name, W, H, spp):
    from paper_2210_06158_gb300 import dof
    results = []
    for setting in (None, dict(packets=0, bvh_width=4, ray_grid=4), dict(packets=1, ray_grid=8), dict(bvh_width=2)):
        ctx = dof.Context(0)
        if setting:
            ctx.set_trace(**setting)
        w, prm, sc, gbs, h = _session(dof, ctx, name, W, H, spp)
        outs = [dof.frame(ctx, sc, gbs[k], w.camera(k), prm, h).cpu().numpy() for k in range(3)]
        st = h.stats()
        assert st.device_status == 0 and st.rays > 0 and st.node_visits > 0
        results.append((outs, h.read("RAY_PRIM", np.int32)))
    for r in results[1:]:
        assert np.array_equal(results[0][1], r[1])
        for a, b in zip(results[0][0], r[0]):
            assert np.array_equal(a, b)


def test_open_tracer_in_a_mixed_batch_and_graph():
    """c3's lens at 362 lines alone would take one ray per lane, c2's packets; the graph's
    launches also focus nearer, which widens the blur past the rule's line."""
    import torch
    from paper_2210_06158_gb300 import dof
    kinds = [("c3", 642, 362, 1), ("c2", 322, 182, 2), ("c1", 130, 74, 1)]

    def camera(w, k):
        cam = w.camera(min(k, w.n_frames - 1))
        cam.focus_m = cam.focus_m / (1 + 2 * k)
        return cam

    ctx = dof.Context(0)
    ss = [_session(dof, ctx, *q, frames=1 if q[0] == "c1" else 3) for q in kinds]
    alone = [[dof.frame(ctx, s[2], s[3][min(k, len(s[3]) - 1)], camera(s[0], k), s[1], s[4]).cpu().numpy() for k in range(3)]
             for s in ss]
    for graph in (False, True):
        for s in ss:
            s[4].reset()
        step = lambda k: [dict(scene=s[2], gbuf=s[3][min(k, len(s[3]) - 1)], cam=camera(s[0], k), params=s[1], hist=s[4])  # noqa: E731
                          for s in ss]
        g = dof.Graph(ctx, step(0)) if graph else None
        for k in range(3):
            outs = g.launch(step(k)) if graph else dof.batch_frame(ctx, step(k))
            torch.cuda.synchronize()
            for i, o in enumerate(outs):
                assert np.array_equal(o.cpu().numpy(), alone[i][k]), (graph, k, i)
