"""The allocation-free tile map at ragged sizes and dilation radii: strips of four tiles, blocks of
32 x 8 tiles and their halo against a plain maximum in torch."""

import pytest

from synth import Camera, camera_pose
from synth.scenes import default_params

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("coc", [1.0, 16.0, 17.0, 256.0])
@pytest.mark.parametrize("W,H", [(2, 2), (14, 16), (16, 18), (66, 130), (514, 130), (530, 274), (3842, 2162)])
def test_tile_map_equals_plain_maxima(W, H, coc):
    import torch
    from paper_2210_06158_gb300 import dof
    cam = Camera.from_poses(dict(f_m=0.085, f_number=1.2, focus_m=20.0, sensor_w_m=0.036), camera_pose((0.0, 0.0, 0.0)))
    prm = default_params(max_coc_px=coc)
    g = torch.Generator(device="cuda").manual_seed(W * 7 + H)
    depth = torch.rand((H, W), device="cuda", generator=g) * 60 + 0.5
    depth[torch.rand((H, W), device="cuda", generator=g) < 0.1] = float("inf")
    got = dof.coc_tiles_noalloc(depth, cam, prm)
    z = depth.double().clamp(max=prm["z_far_m"]).view(H // 2, 2, W // 2, 2).amin((1, 3))
    c = 0.085 / 1.2 * 0.085 * W / (0.036 * (20.0 - 0.085)) * (z - 20.0) / z
    rho = (c / 4).clamp(-coc / 2, coc / 2)
    v = torch.nn.functional.pad(torch.stack(((-rho).clamp(min=0), rho.abs()))[None], (0, -(W // 2) % 8, 0, -(H // 2) % 8))
    k = -(-int(coc) // 16)
    want = torch.nn.functional.max_pool2d(torch.nn.functional.max_pool2d(v, 8), 2 * k + 1, stride=1, padding=k)[0].permute(1, 2, 0)
    # rho in FP32: cocK, a subtraction, a product and a division round once each (relative 2^-24
    # of terms no larger than cocK |z - d| / z, where |z - d| >= 2^-24 z is exact)
    assert got.shape == want.shape
    assert torch.all((got.double() - want).abs() <= 4 * 2.0 ** -23 * want.abs() + 1e-6)
