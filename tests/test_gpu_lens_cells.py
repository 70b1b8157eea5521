"""Rays grouped by lens cells take their lens samples from the mask kernel, rays in pixel order
draw them in the tracer: the images are the same bits either way."""

import numpy as np
import pytest

from synth import make_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blades", [0, 5])
@pytest.mark.parametrize("mode", [dict(spp=1), dict(spp=3), dict(ray_mode=1, m=5)])
def test_lens_cells_keep_every_bit(mode, blades):
    import torch
    from paper_2210_06158_gb300 import dof
    ctx = dof.Context(0)
    ss = []
    for k, (W, H) in enumerate([(2, 2), (66, 34), (202, 118)]):
        w = make_workload("c3", W=W, H=H, n_frames=2, session=k)
        prm = dict(w.params, blades=blades, **mode)
        sc = dof.Scene(ctx, make_workload("c1", session=k).scene)
        gb = [dof.gbuffer(ctx, sc, w.camera(f), prm, W, H) for f in range(2)]
        ss.append((w, prm, sc, gb, dof.History(ctx, W, H, max_rays=5)))
    want = None
    for grid, packets in ((1, False), (4, False), (1, True), (8, True), (16, True)):
        ctx.set_trace(bvh_width=2, ray_grid=grid, packets=packets)
        for s in ss:
            s[4].reset()
        got = []
        for f in range(2):
            outs = dof.batch_frame(ctx, [dict(scene=sc, gbuf=gb[f], cam=w.camera(f), params=prm, hist=h)
                                         for w, prm, sc, gb, h in ss])
            got += [o.cpu().numpy() for o in outs]
        torch.cuda.synchronize()
        for s in ss:
            assert s[4].stats().device_status == 0
        if want is None:
            want = got
        for a, b in zip(want, got):
            assert np.array_equal(a, b), (grid, packets)
