"""The main filter's form: the one the caller names runs, and every form gives the same bits."""

import numpy as np
import pytest

from synth import make_workload

pytestmark = pytest.mark.gpu

W, H = 1002, 730            # 182,865 half-resolution pixels: the open choice takes the columns


def _session(ctx):
    import torch
    from paper_2210_06158_gb300 import dof
    w = make_workload("c1", W=W, H=H)
    sc = dof.Scene(ctx, w.scene)
    gb = dof.gbuffer(ctx, sc, w.camera(0), w.params, W, H)
    torch.cuda.synchronize()
    return dict(scene=sc, gbuf=gb, cam=w.camera(0), params=dict(w.params), hist=dof.History(ctx, W, H, max_rays=1))


def test_a_named_form_is_the_form_that_runs():
    """A graph captured under one form refuses to replay under another, so the forms are told
    apart: 1 (one pixel per thread) is not 3 (columns)."""
    from paper_2210_06158_gb300 import dof
    ctx = dof.Context(0)
    item = _session(ctx)
    for captured, other in ((1, 3), (3, 1), (1, 0)):
        ctx.set_gather(block=(32, 4), main_form=captured)
        g = dof.Graph(ctx, [item])
        g.launch([item])
        ctx.set_gather(main_form=other)
        with pytest.raises(dof.DofError) as e:
            g.launch([item])
        assert e.value.code == -7
        g.close()


@pytest.mark.parametrize("storage", [0, 1])
def test_open_choice_and_every_form_give_the_same_bits(storage):
    import torch
    from paper_2210_06158_gb300 import dof
    want = None
    for setting in (None, dict(main_form=0), dict(main_form=1), dict(main_form=2), dict(main_form=3),
                    dict(main_form=3, block=(32, 2)), dict(main_form=1, block=(32, 4)), dict(block=(16, 16))):
        ctx = dof.Context(0)
        if setting:
            ctx.set_gather(**setting)
        item = _session(ctx)
        out = dof.frame(ctx, item["scene"], item["gbuf"], item["cam"], dict(item["params"], image_storage=storage),
                        item["hist"])
        torch.cuda.synchronize()
        got = (out.cpu().numpy(), item["hist"].read("MAIN"))
        if want is None:
            want = got
        for a, b in zip(want, got):
            assert np.array_equal(a, b), setting
