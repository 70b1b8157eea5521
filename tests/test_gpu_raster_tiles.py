"""The object-order producer's tiles, lists and batches at the sizes where they can go wrong:
images that are no multiple of the 8- and 64-pixel tiles, triangles that are cut into chunks
(planes over the whole image) among ones of a few pixels, and scenes on both sides of the
sorted batches.  Bits as the ray-cast producer gives them."""

import numpy as np
import pytest

from synth import Camera, Scene, camera_pose
from synth.scenes import default_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [3, 900, 65535, 65537, 90001])
@pytest.mark.parametrize("W,H", [(2, 2), (6, 10), (66, 62), (130, 64), (514, 258), (1366, 768)])
def test_tiles_chunks_and_batches(n, W, H):
    import torch
    from paper_2210_06158_gb300 import dof
    rng = np.random.default_rng(n + W)
    depth = rng.uniform(1.5, 12, n)
    c = np.stack([rng.uniform(-0.6, 0.6, n) * depth, rng.uniform(-0.4, 0.4, n) * depth, depth], -1)
    # mostly thin blades, some specks, and a few that span the image at several depths
    size = np.where(rng.random(n) < 0.6, 0.25, 0.004)[:, None, None] * np.array([0.1, 1.0, 0.3])
    v = c[:, None, :] + size * rng.uniform(-1, 1, (n, 3, 3))
    for k, z in enumerate((3.0, 6.0, 14.0)[:min(3, n)]):
        x = 0.2 * k - 0.3
        v[k] = [[-40, -40, z], [x, 40, z + 1], [x, -40, z + 2]]
    ctx = dof.Context(0)
    sc = dof.Scene(ctx, Scene(v.astype(np.float32).reshape(-1, 3), np.arange(3 * n, dtype=np.uint32).reshape(n, 3),
                              np.zeros(n, np.uint32), 1))
    prm = default_params()
    for pitch in (0.0, 20.0):
        cam = Camera.from_poses(dict(f_m=0.035, f_number=2.0, focus_m=4.0, sensor_w_m=0.036), camera_pose((0.0, 0.0, 0.0), pitch))
        want = dof.gbuffer(ctx, sc, cam, prm, W, H)
        got = dof.gbuffer(ctx, sc, cam, prm, W, H, raster=True)
        torch.cuda.synchronize()
        for k in want:
            assert torch.equal(want[k], got[k]), (k, pitch)
