"""Polygonal apertures with the lens samples that the mask kernel hands to the tracer."""

import pytest

from synth import make_workload


BLADES = [0, 3, 6]


@pytest.mark.gpu
@pytest.mark.parametrize("blades", BLADES)
@pytest.mark.parametrize("mode", [dict(spp=3), dict(ray_mode=1, m=5)])
def test_lens_samples_handed_to_the_tracer_keep_the_aperture(mode, blades):
    """Rays grouped by lens cells take the samples that the mask kernel drew, rays in pixel order
    draw them in the tracer: the same bits with a polygonal aperture, and not those of the
    circle."""
    import torch
    from paper_2210_06158_gb300 import dof
    W, H = 202, 118
    w = make_workload("c3", W=W, H=H, n_frames=2)
    ctx = dof.Context(0)
    sc = dof.Scene(ctx, make_workload("c1").scene)
    images = {}
    for b in {blades, 0}:
        prm = dict(w.params, aperture_blades=b, **mode)
        gb = [dof.gbuffer(ctx, sc, w.camera(f), prm, W, H) for f in range(2)]
        for grid, packets in ((1, False), (4, False), (1, True), (8, True)):
            ctx.set_trace(ray_grid=grid, packets=packets)
            h = dof.History(ctx, W, H, max_rays=5)
            out = [dof.frame(ctx, sc, gb[f], w.camera(f), prm, h).clone() for f in range(2)]
            torch.cuda.synchronize()
            assert h.stats().device_status == 0 and h.stats().rays > 0
            want = images.setdefault(b, out)
            assert all(torch.equal(x, y) for x, y in zip(want, out)), (b, grid, packets)
    if blades:
        assert not torch.equal(images[0][1], images[blades][1])
