"""Sessions on both sides of the size from which the reconstruction takes one thread per pixel: a
session's frames have the same bits alone, in a batch with larger ones and for any block
shape."""

import numpy as np
import pytest

from synth import make_workload

pytestmark = pytest.mark.gpu

SIZES = [(2, 2), (34, 18), (250, 142), (398, 400), (400, 400), (402, 398)]     # 40,000 half-resolution pixels at 400 x 400


@pytest.mark.parametrize("storage", [0, 1])
def test_split_and_unsplit_sessions_alone_and_together(storage):
    import torch
    from paper_2210_06158_gb300 import dof
    ctx = dof.Context(0)
    ss = []
    for k, (W, H) in enumerate(SIZES):
        w = make_workload("c2" if k % 2 else "c3", W=W, H=H, n_frames=3, session=k)
        prm = dict(w.params, spp=1, image_storage=storage)
        sc = dof.Scene(ctx, make_workload("c1", session=k).scene)
        gb = [dof.gbuffer(ctx, sc, w.camera(f), prm, W, H) for f in range(3)]
        ss.append((w, prm, sc, gb, dof.History(ctx, W, H, max_rays=1)))
    want = None
    for block, batch in (((32, 8), False), ((32, 8), True), ((16, 16), False), ((16, 8), True), ((64, 4), False), ((8, 8), True)):
        ctx.set_gather(recon_block=block)
        got = []
        for s in ss:
            s[4].reset()
        for f in range(3):
            items = [dict(scene=sc, gbuf=gb[f], cam=w.camera(f), params=prm, hist=h) for w, prm, sc, gb, h in ss]
            outs = dof.batch_frame(ctx, items) if batch else [dof.batch_frame(ctx, [i])[0] for i in items]
            got.append([o.cpu().numpy() for o in outs])
        got.append([s[4].read("RECON").copy() for s in ss])
        torch.cuda.synchronize()
        if want is None:
            want = got
        for a, b in zip(want, got):
            for k, (x, y) in enumerate(zip(a, b)):
                assert np.array_equal(x, y), (block, batch, k)
