"""A frame of few tiles is rendered a quarter tile per warp, a larger one, and
every batch, a half: the images are the same bit for bit, on both sides of the
line (8 tiles per SM) and for ragged sizes."""
import numpy as np
import pytest

from paper_2605_04844_gb300 import synth

from gpu_util import to_device

pytestmark = pytest.mark.gpu


def sizes():
    # 1216 = 8 * 152 tiles is the last quarter frame of a 152-SM chip
    return [(1, 1), (16, 4), (17, 33), (203, 117), (608, 512), (609, 512)]


@pytest.mark.parametrize("W,H", sizes())
@pytest.mark.parametrize("mode", ["quadbox", "aabb3s"])
def test_quarter_and_half_tiles_agree(W, H, mode):
    import torch
    from paper_2605_04844_gb300 import rasterizer as R
    cam = synth.pinhole(W, H, viewmat=synth.look_at((0.0, 0.5, -6.0), (0.0, 0.0, 0.0)))
    scene = synth.scene_ball(6000, 5, radius=3.0, deg=1)
    scene["opacities"][::3] += 4.0   # some beyond the 0.99 cap's test
    scene["scales"][::5, 0] += 2.5   # some elongated
    sd = to_device(scene)
    img, _ = R.forward(sd, cam, mode, bg=(0.1, 0.2, 0.3))
    b = R.calibrated_batch(sd, [cam], mode=mode, group=1)
    b.render(R.scene_struct(sd), R.camera_array([cam]), mode, bg=(0.1, 0.2, 0.3))
    torch.cuda.synchronize()
    b.check()
    np.testing.assert_array_equal(b.image(0).cpu().numpy(), img.cpu().numpy())
