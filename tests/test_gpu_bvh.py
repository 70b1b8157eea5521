"""The SAH builder's seams: cluster counts on both sides of the warp-sized segments and of
the chunks, planes that separate nothing, and coordinates that need deep trees.  The
ray-cast G-buffer (which traverses the tree) has to give the bits of the object-order
producer (which does not)."""

import numpy as np
import pytest

from synth import Camera, Scene, camera_pose
from synth.scenes import default_params

pytestmark = pytest.mark.gpu


def _scene(kind, n):
    rng = np.random.default_rng(100 + n)
    if kind == "random":
        c = rng.uniform((-1.5, -1, 2), (1.5, 1, 6), (n, 3))
        size = 0.3
    elif kind == "same_centre":         # nested around one point: no plane separates the centroids
        c = np.tile(np.array([[0.0, 0.0, 4.0]]), (n, 1))
        size = np.linspace(0.05, 0.6, n)[:, None, None]
    elif kind == "geometric":           # each centroid gap half the one before: one triangle split off per level
        c = np.zeros((n, 3))
        c[:, 0] = 1.5 * 0.5 ** np.arange(n)
        c[:, 2] = 4.0 + 1e-3 * np.arange(n)
        size = 0.05
    else:                               # a flat sheet: one axis without extent
        c = np.stack([rng.uniform(-2, 2, n), rng.uniform(-1, 1, n), np.full(n, 4.0)], -1)
        size = 0.2
    d = rng.uniform(-1, 1, (n, 3, 3))
    if kind == "same_centre":
        # symmetric about the point, so that the box's centre is the point itself
        d = np.array([[-1.0, -1.0, 0.0], [1.0, -1.0, 0.0], [0.0, 1.0, 0.0]])[None] * np.ones((n, 1, 1))
    if kind == "sheet":
        d[..., 2] = 0
    v = (c[:, None, :] + size * d).astype(np.float32).reshape(-1, 3)
    return Scene(v, np.arange(3 * n, dtype=np.uint32).reshape(n, 3), np.zeros(n, np.uint32), 1)


@pytest.mark.parametrize("kind,n", [("random", n) for n in (2, 3, 5, 255, 256, 257, 258, 511, 513, 1025, 2049, 5000, 40001)]
                         + [("same_centre", n) for n in (2, 3, 300, 700, 3000)]
                         + [("geometric", n) for n in (40, 300, 1200)] + [("sheet", n) for n in (64, 1500)])
def test_tree_sees_what_the_rasteriser_sees(kind, n):
    import torch
    from paper_2210_06158_gb300 import dof
    ctx = dof.Context(0)
    cam = Camera.from_poses(dict(f_m=0.035, f_number=2.0, focus_m=4.0, sensor_w_m=0.036), camera_pose((0.0, 0.0, 0.0), 0.0))
    prm = default_params()
    host = _scene(kind, n)
    want = None
    for radius, rotations, width in ((48, 0, 4), (1, 0, 2), (256, 2, 2)):
        ctx.set_ploc_radius(radius)
        ctx.set_bvh_rotations(rotations)
        ctx.set_bvh_width(width)
        sc = dof.Scene(ctx, host)
        i = sc.info()
        assert i.depth <= i.stack_limit and i.n_nodes == max(0, n - i.n_large - 1)
        if want is None:
            want = dof.gbuffer(ctx, sc, cam, prm, 320, 180, raster=True)
            assert int((want["prim"] >= 0).sum()) > 0
        got = dof.gbuffer(ctx, sc, cam, prm, 320, 180)
        torch.cuda.synchronize()
        for k in want:
            assert torch.equal(want[k], got[k]), (k, radius, rotations, width)


def test_bounds_without_a_finite_area_are_refused():
    """Boxes whose areas overflow cannot be clustered by area: an error, as before (more such
    triangles than may stay out of the tree)."""
    from paper_2210_06158_gb300 import dof
    ctx = dof.Context(0)
    host = _scene("random", 100)
    host.verts[:] = np.sign(host.verts - host.verts.mean(0)) * np.float32(3e38)
    with pytest.raises(dof.DofError) as e:
        dof.Scene(ctx, host)
    assert e.value.code == -6
